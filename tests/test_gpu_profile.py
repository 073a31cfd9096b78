"""The measurement hooks: every blocking decode, whichever engine runs it,
reports its score and residual phases, and ccs_profile_phases never answers
with an older launch's."""
import pytest

from gpu_util import device_problem
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


def _check_phases(ccs, times, iterations, stalled):
    assert times["persistent"][0] == 1
    for kind in ("score", "residual"):
        assert times[kind][0] == iterations and times[kind][1] > 0.0
    total = 0.0
    for it in range(iterations):
        us = ccs.ccs_profile_phases(it)
        assert us is not None and us[0] > 0.0 and us[1] > 0.0
        total += us[0] + us[1]
    # (the iteration in which a decode stalls is not counted, but has phases)
    assert ccs.ccs_profile_phases(iterations + stalled) is None
    # the phases lie within the launch (event time; 5 us of slack for its resolution)
    assert total <= times["persistent"][1] * 1e3 + 5.0


@pytest.mark.parametrize("form", [0, 2])
@pytest.mark.parametrize("shape", [(501, 60, 7, 6), (60001, 6000, 7, 600)], ids=["on_chip", "engine"])
def test_single_decode_reports_its_phases(ccs, shape, form):
    csc, ptr, cols, y = device_problem(ccs, inputs.make_problem(*shape, 31))
    ccs.ccs_profile_begin()
    g = ccs.decode_parallel_l0(csc, ptr, cols, y, debug_flags=form)
    times = ccs.ccs_profile_end()
    assert g.iterations > 0
    _check_phases(ccs, times, g.iterations, g.status == ccs.STALLED)


@pytest.mark.parametrize("sizes", [[(30011, 3001, 7, 200), (26001, 2600, 5, 150)],
                                   [(300, 40, 5, 3), (290, 41, 5, 4)]], ids=["engine", "on_chip"])
def test_batch_of_one_class_reports_its_phases(ccs, sizes):
    """One launch: the engine's phases cover the longest decode; on chip, where
    each problem goes at its own pace, they are the largest problem's."""
    probs = [inputs.make_problem(*s, 40 + q) for q, s in enumerate(sizes)]
    items = [device_problem(ccs, p) for p in probs]
    on_chip = probs[0].n * probs[0].d < 4096
    ccs.ccs_profile_begin()
    outs = ccs.decode_batch(items, engine=ccs.ENGINE_AUTO if on_chip else ccs.ENGINE_PERSISTENT)
    times = ccs.ccs_profile_end()
    last = outs[0] if on_chip else max(outs, key=lambda g: (g.iterations, g.status == ccs.STALLED))
    _check_phases(ccs, times, last.iterations, last.status == ccs.STALLED)


def test_phases_of_an_older_launch_are_not_returned(ccs):
    import torch
    p = inputs.make_problem(60001, 6000, 7, 600, 5)
    csc, ptr, cols, y = device_problem(ccs, p)
    x = torch.empty(p.n, dtype=torch.float64, device="cuda")
    r = torch.empty(p.m, dtype=torch.float64, device="cuda")
    ws = ccs.workspace(ccs.ccs_workspace_size(ccs.OP_DECODE, p.n, p.m, p.d))
    buf = ccs.result_buffer(1)
    ccs.ccs_profile_begin()
    ccs.decode_parallel_l0(csc, ptr, cols, y)
    assert ccs.ccs_profile_phases(0) is not None
    ccs.ccs_decode_parallel_l0_async(p.n, p.m, p.d, csc, ptr, cols, y, x, r, None, None, buf, ws)
    assert ccs.ccs_profile_phases(0) is None
    torch.cuda.synchronize()
    ccs.ccs_profile_end()
