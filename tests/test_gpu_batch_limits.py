"""Batches at and beyond the launch limits: more problems than one launch of
the persistent engine takes, and a batch whose bounded waits run out."""
import ctypes

import numpy as np
import pytest

from gpu_util import device_problem, oracle_problem
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


def _many(ccs, count):
    """`count` problems over two tiny matrices (d = 3 and d = 9), outputs of their own."""
    import torch
    probs = [inputs.make_problem(20, 12, 3, 1, 5), inputs.make_problem(20, 12, 9, 1, 6)]
    items = [device_problem(ccs, p) for p in probs]
    x = torch.full((count, 20), float("nan"), dtype=torch.float64, device="cuda")
    r = torch.full((count, 12), float("nan"), dtype=torch.float64, device="cuda")
    pbs = [ccs.problem(*items[q % 2], x[q], r[q]) for q in range(count)]
    return probs, items, pbs, x


def test_more_problems_than_a_launch(ccs, orc):
    """4097 problems: the host-driven engine decodes them, ccs_autotune takes
    them (no launch group of it holds more than 4096), a single launch of the
    persistent engine cannot and the call says so."""
    probs, items, pbs, x = _many(ccs, 4097)
    ws = ccs.workspace(ccs.ccs_batch_workspace_size(pbs))
    with pytest.raises(ccs.CcsError) as ei:
        ccs.ccs_decode_batch(pbs, ccs.params(), ws)
    assert ei.value.code == ccs.CCS_EINVAL
    refs = []
    for p in probs:
        A, y = oracle_problem(orc, p)
        refs.append(orc.parallel_l0(A, p.m, y))
    res = ccs.ccs_decode_batch(pbs, ccs.params(engine=ccs.ENGINE_HOST_LOOP), ws)
    got = x.cpu().numpy()
    for q in range(4097):
        ref = refs[q % 2]
        assert (res[q].status, res[q].iterations) == (ref["status"], ref["iterations"])
        assert np.array_equal(got[q], ref["x_hat"])
    try:
        assert sum(t != 0 for t in ccs.ccs_autotune(pbs, ccs.params(), ws)) == 2
    finally:
        ccs.ccs_autotune_reset()


def test_batch_that_times_out_reports_where_it_stood(ccs):
    """CTA 0 never arrives at the first score barrier (test hook), so every
    bounded wait runs out; each problem reports the time-out and the state
    it was in: no iteration done, ||r||_0 of y."""
    import torch
    probs = [inputs.make_problem(5003, 500, 7, 20, 8), inputs.make_problem(6007, 600, 5, 30, 9)]
    items = [device_problem(ccs, p) for p in probs]
    pbs = [ccs.problem(*it, torch.empty(p.n, dtype=torch.float64, device="cuda"),
                       torch.empty(p.m, dtype=torch.float64, device="cuda"))
           for it, p in zip(items, probs)]
    ws = ccs.workspace(ccs.ccs_batch_workspace_size(pbs))
    ws.fill_(0x55)
    torch.cuda.synchronize()
    arr = (ccs.Problem * 2)(*pbs)
    out = (ccs.Result * 2)()
    prm = ccs.params(engine=ccs.ENGINE_PERSISTENT, watchdog_ms=200, debug_flags=1)
    rc = ccs.lib().ccs_decode_batch(arr, 2, ctypes.byref(prm), out, ws.data_ptr(), ws.numel(), None)
    assert rc == ccs.CCS_ETIMEOUT
    for (_, _, _, y), res in zip(items, out):
        assert (res.status, res.iterations, res.error) == (-1, 0, ccs.CCS_ETIMEOUT)
        assert res.r0_final == int((y != 0).sum())
