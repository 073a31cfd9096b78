"""Values at the end of the binary64 range, infinities and NaN.

Near the largest double a sum can overflow in one order and not in another,
so a residual kept by subtracting accepted values in any order is only exact
while no partial sum can leave the range; beyond that the ordered sums of
Alg. 2 decide, in every engine."""
import numpy as np
import pytest

from gpu_util import assert_same_decode, upload_matrix
from paper_1508_01256_gb300 import inputs

pytestmark = pytest.mark.gpu

HUGE = 1.5 * 2.0 ** 1023  # two of them overflow


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


def _cancelling(blocks, padding, minus):
    """`blocks` groups of three columns that share one row and have two rows
    of their own each; their values are HUGE but for column `minus` of each
    group, which is -HUGE, so the shared row's ordered sum stays finite.
    The groups' columns lie far apart, `padding` columns between them."""
    n, m = 3 * blocks + 2 * padding, 7 * blocks + 3
    A = np.empty((n, 3), dtype=np.int32)
    A[:] = [7 * blocks, 7 * blocks + 1, 7 * blocks + 2]  # rows of zeros: never accepted
    x = np.zeros(n)
    for t in range(3):
        j0 = t * (blocks + padding)
        for b in range(blocks):
            A[j0 + b] = [b, blocks + 6 * b + 2 * t, blocks + 6 * b + 2 * t + 1]
            x[j0 + b] = -HUGE if t == minus else HUGE
    return A, m, x


# 3 columns of 3 rows in one CTA on chip, and 6300 of them over several
SIZES = {"one_cta": (5, 0), "several_ctas": (100, 3000)}


@pytest.mark.parametrize("engine", [0, 3], ids=["auto", "persistent"])
@pytest.mark.parametrize("minus", [0, 1])
@pytest.mark.parametrize("size", list(SIZES))
def test_sums_that_overflow_in_another_order(ccs, orc, size, minus, engine):
    import torch
    A, m, x = _cancelling(*SIZES[size], minus)
    y = orc.measure(A, m, x)
    assert np.isfinite(y).all()
    ref = orc.parallel_l0(A, m, y)
    assert (ref["status"], ref["iterations"]) == (ccs.CONVERGED, 1) and np.array_equal(ref["x_hat"], x)
    csc, ptr, cols = upload_matrix(orc, A, m)
    g = ccs.decode_parallel_l0(csc, ptr, cols, torch.from_numpy(y).cuda(), engine=engine)
    assert_same_decode(g, ref)
    assert g.residual_form == ccs.RESIDUAL_ORDERED


@pytest.mark.parametrize("engine", [0, 3], ids=["auto", "persistent"])
def test_largest_values_still_certified(ccs, orc, engine):
    """Multiples of 2^980 whose sums stay far inside the range: exact."""
    import torch
    p = inputs.make_problem(1201, 200, 5, 12, 3, "pm1")
    A = orc.make_expander(p.n, p.m, p.d, p.a_seed)
    y = orc.measure(A, p.m, p.x * 2.0 ** 980)
    ref = orc.parallel_l0(A, p.m, y, max_iter=20)
    csc, ptr, cols = upload_matrix(orc, A, p.m)
    g = ccs.decode_parallel_l0(csc, ptr, cols, torch.from_numpy(y).cuda(), engine=engine, max_iter=20)
    assert_same_decode(g, ref)
    assert g.residual_form == ccs.RESIDUAL_EXACT


@pytest.mark.parametrize("values", ["inf", "inf_only", "nan", "mixed"])
@pytest.mark.parametrize("shape", [(401, 60, 7, 6), (9001, 900, 7, 60)], ids=["one_cta", "several_ctas"])
def test_infinite_and_nan_measurements(ccs, orc, shape, values):
    """Infinities and NaN in y: the engine on chip and the persistent one
    reach the same bits, and the first iteration (before any inf - inf) is
    the oracle's when y holds no NaN."""
    import torch
    p = inputs.make_problem(*shape, 17)
    A = orc.make_expander(p.n, p.m, p.d, p.a_seed)
    x = p.x.copy()
    at = np.nonzero(x)[0]
    if values == "inf_only":
        x[:] = 0.0
        x[at[:3]] = [np.inf, -np.inf, np.inf]
    else:
        x[at[:3]] = {"inf": [np.inf, -np.inf, 1.0], "nan": [np.nan, 1.0, np.nan],
                     "mixed": [np.inf, np.nan, -np.inf]}[values]
    with np.errstate(invalid="ignore"):
        y = orc.measure(A, p.m, x)
    csc, ptr, cols = upload_matrix(orc, A, p.m)
    yd = torch.from_numpy(y).cuda()
    for iters in (1, 2, 12):
        small, engine = (ccs.decode_parallel_l0(csc, ptr, cols, yd, engine=e, max_iter=iters)
                         for e in (ccs.ENGINE_AUTO, ccs.ENGINE_PERSISTENT))
        for key in ("status", "iterations", "r0_final", "r0_hist", "residual_form"):
            assert small[key] == engine[key], key
        assert small.residual_form == ccs.RESIDUAL_ORDERED
        for key in ("x_hat", "r"):
            assert torch.equal(small[key].view(torch.int64), engine[key].view(torch.int64)), key
        if iters == 1 and not np.isnan(y).any():
            with np.errstate(invalid="ignore"):
                ref = orc.parallel_l0(A, p.m, y, max_iter=1)
            assert small.iterations == ref["iterations"]
            assert np.array_equal(small.x_hat.cpu().numpy(), ref["x_hat"])
            assert np.array_equal(small.r.cpu().numpy(), ref["r"], equal_nan=True)
