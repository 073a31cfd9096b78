"""The small engine: problems decoded by one thread-block cluster on chip.

Every decode is compared bit for bit with the oracle: clusters of 1 to 8
CTAs, sizes at the edges of a CTA's part, more accepted columns than the
CTAs' lists hold, rows with more contributors than their records hold, both
residual forms and the switch between them, every d, the shifted variant;
and the same problems in one batch, where the persistent engine takes the
large ones.
"""
import numpy as np
import pytest

from gpu_util import assert_same_decode, device_problem, oracle_problem
from paper_1508_01256_gb300 import inputs

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


# (n, m, d, k, values, decode options)
CASES = {
    "one_column": (1, 5, 5, 1, "gauss-grid", {}),
    "one_cta": (800, 90, 5, 9, "gauss-raw", {}),
    "two_ctas": (1171, 130, 7, 30, "gauss-grid", {}),
    "four_ctas": (1601, 170, 9, 20, "gauss-raw", {}),
    "ragged_parts": (4097, 411, 7, 41, "gauss-grid", {}),
    "empty_part": (33, 40, 3, 2, "pm1", {}),
    "many_accepted": (9001, 3001, 5, 900, "gauss-grid", {}),
    "few_rows": (7001, 72, 11, 4, "gauss-grid", {}),
    "oscillates": (8746, 87, 5, 40, "gauss-raw", {}),
    "dense": (12001, 1201, 7, 420, "gauss-grid", {}),
    "count": (9000, 900, 7, 130, "gauss-raw", dict(score_mode=1, alpha=4)),
    "alpha3": (9000, 900, 7, 220, "gauss-raw", dict(alpha=3)),
    "shifted": (6007, 700, 5, 70, "gauss-grid", dict(shifted=True)),
    "d8": (5003, 500, 8, 60, "gauss-raw", {}),
    "d16": (4011, 401, 16, 30, "gauss-raw", {}),
}


def _problem(case):
    n, m, d, k, values, kw = CASES[case]
    return inputs.make_problem(n, m, d, k, 300 + n % 89, values), kw


@pytest.mark.parametrize("case", list(CASES))
@pytest.mark.parametrize("form", [0, 2, 4], ids=["certified", "ordered", "switch"])
def test_small_engine_matches_oracle(ccs, orc, case, form):
    p, kw = _problem(case)
    csc, ptr, cols, y = device_problem(ccs, p)
    A, y_ref = oracle_problem(orc, p)
    ref = orc.parallel_l0(A, p.m, y_ref, max_iter=30, **kw)
    small = ccs.decode_parallel_l0(csc, ptr, cols, y, max_iter=30, debug_flags=form, **kw)
    engine = ccs.decode_parallel_l0(csc, ptr, cols, y, max_iter=30, debug_flags=form | 32, **kw)
    for g in (small, engine):
        assert_same_decode(g, ref)
    assert small.residual_form == engine.residual_form


def test_batch_of_small_and_large_problems(ccs, orc):
    """One batch over both engines, decoded twice from one workspace."""
    import torch
    names = [c for c in CASES if not CASES[c][5]]
    probs = [_problem(c)[0] for c in names]
    probs += [inputs.make_problem(120001, 12001, 7, 1500, 5), inputs.make_problem(70001, 40001, 9, 900, 6),
              inputs.make_problem(60001, 600, 9, 70, 7)]
    items = [device_problem(ccs, p) for p in probs]
    refs = []
    for p in probs:
        A, y_ref = oracle_problem(orc, p)
        refs.append(orc.parallel_l0(A, p.m, y_ref))
    outs = ccs.decode_batch(items, history=True)
    for g, ref in zip(outs, refs):
        assert_same_decode(g, ref)
    bufs, pbs = [], []
    for (csc, ptr, cols, y), p in zip(items, probs):
        x_hat = torch.full((p.n,), float("nan"), dtype=torch.float64, device="cuda")
        r = torch.empty(p.m, dtype=torch.float64, device="cuda")
        bufs.append((x_hat, r))
        pbs.append(ccs.problem(csc, ptr, cols, y, x_hat, r))
    graph = ccs.BatchGraph(pbs)
    for _ in range(2):
        graph.launch()
    torch.cuda.synchronize()
    for (x_hat, r), ref, res in zip(bufs, refs, graph.read_results()):
        assert (res.status, res.iterations, res.r0_final, res.error) == \
            (ref["status"], ref["iterations"], ref["r0_final"], 0)
        assert np.array_equal(x_hat.cpu().numpy(), ref["x_hat"])
        assert np.array_equal(r.cpu().numpy(), ref["r"])
    graph.close()


@pytest.mark.parametrize("small, large", [(1, 3), (1, 2), (2, 2)])
def test_batch_on_both_sides_of_the_rule(ccs, orc, small, large):
    """The small engine takes a batch's small problems when they are a third of it."""
    probs = [_problem(c)[0] for c in ("ragged_parts", "oscillates")[:small]]
    probs += [inputs.make_problem(120001, 12001, 7, 1500, 5), inputs.make_problem(130001, 1300, 9, 90, 6),
              inputs.make_problem(140001, 1400, 7, 140, 7)][:large]
    for g, p in zip(ccs.decode_batch([device_problem(ccs, p) for p in probs], history=True), probs):
        A, y_ref = oracle_problem(orc, p)
        assert_same_decode(g, orc.parallel_l0(A, p.m, y_ref))
