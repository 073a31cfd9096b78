"""y = A x and y = A diag(s) x on matrices large enough for the nonzero marks,
bit for bit against the oracle: every mark width, rows of a few and of many
columns, sparse and dense x, infinities and NaN."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


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


# n, m, d: marks of one column (rows of a few columns and of many), of 2, 16,
# 32, 64 and 256; fewer rows than CTAs; rows without columns; the last word
# of marks short; and shapes below the marks
SHAPES = [(600011, 20011, 7), (2400007, 600011, 7), (2097151, 3001, 2), (1398107, 21001, 3),
          (1048577, 1025, 4), (4194305, 2053, 1), (4194305, 1025, 1), (4194307, 263, 1),
          (1398107, 150, 3), (1048577, 2000003, 16), (20001, 2001, 7), (400001, 100, 3)]


@pytest.mark.parametrize("k", ["one", "sparse", "dense", "special"])
@pytest.mark.parametrize("n,m,d", SHAPES)
def test_measure_bitwise(ccs, orc, n, m, d, k):
    import torch
    rng = np.random.default_rng(n + m)
    csc, ptr, cols = ccs.make_expander(n, m, d, 31 + n)
    A = csc.cpu().numpy()
    x = np.zeros(n)
    count = {"one": 1, "sparse": max(1, m // 20), "dense": n, "special": max(8, m // 20)}[k]
    at = np.sort(rng.choice(n, count, replace=False))
    x[at] = rng.standard_normal(count)
    x[at[:1]] = 5e-324
    s = rng.uniform(0.5, 2.0, n)
    if k == "special":
        x[at[1]], x[at[2]], x[at[3]], x[at[4]] = np.inf, -np.inf, np.nan, -0.0
        s[at[5] - 1] = np.inf  # times zero, mostly: the product is NaN
        s[at[6]] = 5e-324      # a product that rounds to zero
    xd, sd = torch.from_numpy(x).cuda(), torch.from_numpy(s).cuda()
    with np.errstate(invalid="ignore"):
        y = ccs.measure(ptr, cols, xd, m, d).cpu().numpy()
        assert np.array_equal(y, orc.measure(A, m, x), equal_nan=True)
        ys = ccs.measure_scaled(ptr, cols, sd, xd, m, d).cpu().numpy()
        assert np.array_equal(ys, orc.measure_scaled(A, m, s, x), equal_nan=True)


def test_unscale_special_values(ccs):
    """Zeros of either sign over ordinary, zero, infinite and NaN scales give
    what binary64 division gives."""
    import torch
    z = np.array([0.0, -0.0, 1.5, -2.5, np.inf, np.nan, 5e-324])
    s = np.array([1.25, -1.25, 0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, 1e308])
    zz, ss = (a.ravel() for a in np.meshgrid(z, s))
    x = ccs.unscale(torch.from_numpy(ss.copy()).cuda(), torch.from_numpy(zz.copy()).cuda())
    with np.errstate(all="ignore"):
        want = zz / ss
    got = x.cpu().numpy()
    assert np.array_equal(np.isnan(got), np.isnan(want))
    ok = ~np.isnan(want)
    assert np.array_equal(got[ok].view(np.int64), want[ok].view(np.int64))
