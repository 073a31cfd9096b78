"""The persistent engine on problems that the library's own choice decodes on
chip: server rounds, and batches with few small problems, still run them
there.  Every d and score, tiny shapes, overflowing rows, the shifted variant
and tuned launch shapes, bit for bit against the oracle."""
import numpy as np
import pytest

from gpu_util import assert_same_decode, device_problem, oracle_problem, upload_matrix
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


def _same(ccs, orc, p, max_iter=40, debug_flags=0, **kw):
    csc, ptr, cols, y = device_problem(ccs, p)
    A, y_ref = oracle_problem(orc, p)
    g = ccs.decode_parallel_l0(csc, ptr, cols, y, engine=ccs.ENGINE_PERSISTENT, max_iter=max_iter,
                               debug_flags=debug_flags, **kw)
    assert_same_decode(g, orc.parallel_l0(A, p.m, y_ref, max_iter=max_iter, **kw))


@pytest.mark.parametrize("d", [2, 3, 5, 8, 11, 13, 16])
@pytest.mark.parametrize("mode", [0, 1])
def test_all_d_and_modes(ccs, orc, d, mode):
    p = inputs.make_problem(6007, max(d, 700), d, 70, 900 + d, "gauss-grid")
    for alpha in sorted({2, (d + 1) // 2 + (d % 2 == 0), d}):
        if alpha >= 2:
            _same(ccs, orc, p, alpha=alpha, score_mode=mode)


@pytest.mark.parametrize("flags", [0, 2, 4])
def test_overflow_rows(ccs, orc, flags):
    """Rows of ~47 nonzero contributors, in every residual form."""
    _same(ccs, orc, inputs.make_problem(4000, 60, 7, 400, 77), max_iter=20, debug_flags=flags)


@pytest.mark.parametrize("shape", [(1, 2, 2, 1), (2, 2, 2, 1), (7, 3, 3, 2), (33, 5, 4, 3),
                                   (257, 16, 16, 5), (3000, 300, 7, 0)])
def test_tiny_shapes(ccs, orc, shape):
    for flags in (0, 2):
        _same(ccs, orc, inputs.make_problem(*shape, shape[0] * 31 + shape[1]), debug_flags=flags)


def test_stalled_and_oscillating(ccs, orc):
    import torch
    for rows, y, mode in (([[0, 1, 2], [2, 3, 4]], [1.0, 2.0, 3.0, 4.0, 5.0], 0),
                          ([[0, 1, 2], [0, 1, 3], [2, 3, 4]], [0.5, 0.5, 0.5, 0.0, 0.0], 1)):
        A, y = np.array(rows, dtype=np.int32), np.array(y)
        csc, ptr, cols = upload_matrix(orc, A, 5)
        g = ccs.decode_parallel_l0(csc, ptr, cols, torch.from_numpy(y).cuda(), score_mode=mode,
                                   max_iter=9, engine=ccs.ENGINE_PERSISTENT)
        assert_same_decode(g, orc.parallel_l0(A, 5, y, score_mode=mode, max_iter=9))


@pytest.mark.parametrize("shape", [(4096, 410, 7, 41, 0), (6007, 700, 5, 70, 1), (20000, 2000, 9, 300, 0)])
def test_shifted(ccs, orc, shape):
    n, m, d, k, mode = shape
    p = inputs.make_problem(n, m, d, k, 500 + d)
    for alpha in sorted({2, d // 2 + 1, d}):
        _same(ccs, orc, p, max_iter=60, alpha=alpha, score_mode=mode, shifted=True)


def test_tuned_shapes_keep_results(ccs, orc):
    """A batch under the shapes ccs_autotune recorded, all of it in the
    persistent engine."""
    import torch
    probs = inputs.batch_problems(12, seed=57, log2n_hi=15.0)
    items = [device_problem(ccs, p) for p in probs]
    pbs = []
    for it, p in zip(items, probs):
        pbs.append(ccs.problem(*it, torch.empty(p.n, dtype=torch.float64, device="cuda"),
                               torch.empty(p.m, dtype=torch.float64, device="cuda")))
    try:
        assert any(ccs.ccs_autotune(pbs, ccs.params(), ccs.workspace(ccs.ccs_batch_workspace_size(pbs))))
        outs = ccs.decode_batch(items, history=True, engine=ccs.ENGINE_PERSISTENT)
        for p, g in zip(probs, outs):
            A, y_ref = oracle_problem(orc, p)
            assert_same_decode(g, orc.parallel_l0(A, p.m, y_ref))
    finally:
        ccs.ccs_autotune_reset()
