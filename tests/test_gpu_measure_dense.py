"""y = A x on matrices large enough for the nonzero marks, for x on both sides
of the sample that decides whether x is marked at all: bit for bit against the
oracle, whichever way the sample points and however wrong it is about the rest
of x."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SAMPLE = 256  # columns looked at, of which more than 5 nonzero make x dense


@pytest.fixture(scope="module")
def ccs():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1508_01256_gb300 import build, ccs
    build.build()
    return ccs


@pytest.fixture(scope="module")
def orc():
    import oracle
    oracle.build()
    return oracle


def _sampled(n):
    """Eight stretches of 32 columns."""
    q = np.arange(SAMPLE, dtype=np.uint64)
    start = ((q >> np.uint64(5)) * 0x9e3779b9 % 2 ** 32) * np.uint64(n) >> np.uint64(32)
    return (start + q % np.uint64(32)).astype(np.int64)


# marks of one column, of two, of 256; rows of a few columns and of many; the
# bits and the word behind them fill y but for less than a word
SHAPES = [(600011, 20011, 7), (2400007, 600011, 7), (2097151, 3001, 2), (4194305, 1025, 1),
          (4194304, 263, 1)]


@pytest.mark.parametrize("x_is", ["dense", "dense_but_the_sample", "sample_only", "five", "six",
                                  "three_percent", "special"])
@pytest.mark.parametrize("n,m,d", SHAPES)
def test_measure_whatever_the_sample_says(ccs, orc, n, m, d, x_is):
    import torch
    rng = np.random.default_rng(n + m)
    csc, ptr, cols = ccs.make_expander(n, m, d, 31 + n)
    A = csc.cpu().numpy()
    values = rng.standard_normal(n)
    at = _sampled(n)
    at = at[at < n]
    x = np.zeros(n)
    if x_is in ("dense", "dense_but_the_sample", "special"):
        x = values.copy()
        if x_is == "dense_but_the_sample":
            x[at] = 0.0
        if x_is == "special":
            x[:4] = [np.inf, np.nan, -np.inf, -0.0]
    elif x_is == "three_percent":
        x = np.where(rng.random(n) < 0.03, values, 0.0)
    else:
        chosen = at[:{"sample_only": SAMPLE, "five": 5, "six": 6}[x_is]]
        x[chosen] = values[chosen]
    s = rng.uniform(0.5, 2.0, n)
    xd, sd = torch.from_numpy(x).cuda(), torch.from_numpy(s).cuda()
    with np.errstate(invalid="ignore"):
        y = ccs.measure(ptr, cols, xd, m, d).cpu().numpy()
        assert np.array_equal(y, orc.measure(A, m, x), equal_nan=True)
        ys = ccs.measure_scaled(ptr, cols, sd, xd, m, d).cpu().numpy()
        assert np.array_equal(ys, orc.measure_scaled(A, m, s, x), equal_nan=True)
