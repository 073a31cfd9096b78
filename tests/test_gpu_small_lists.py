"""Problems on one thread-block cluster whose CTAs accept more columns in an
iteration than their lists hold (64), so that they read one another's sums:
every cluster size, every residual form, alone and in a batch.

Each CTA's part of the columns holds 110 with two rows of their own, which
the first iteration accepts; in `c8` the rows that all columns share collect
more contributors than their records hold."""
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


# n, shared rows, d: clusters of 1, 2, 4 and 8 CTAs (4096 entries a CTA); m <=
# 2560 and n d <= 300,000, so that a lone problem stays on chip too
CASES = {"c1": (1301, 300, 3), "c2": (2501, 400, 3), "c4": (5003, 500, 3), "c8": (6007, 40, 3),
         "c8_wide": (40009, 700, 7)}
EACH = 110  # columns of each part with two rows of their own


def _parts(n, d):
    """CTAs of the cluster and columns of each one's part."""
    C = 1
    while C < 8 and n * d > 4096 * C:
        C *= 2
    return C, (-(-n // C) + 31) // 32 * 32


def _problem(case, raw):
    n, shared, d = CASES[case]
    rng = np.random.default_rng(n)
    C, pitch = _parts(n, d)
    m = shared + 2 * C * EACH
    A = np.array([rng.choice(shared, d, replace=False) for _ in range(n)], dtype=np.int32)
    x = np.zeros(n)
    x[rng.choice(n, 20, replace=False)] = rng.standard_normal(20)
    for c in range(C):
        own = c * pitch + rng.choice(min(n, (c + 1) * pitch) - c * pitch, EACH, replace=False)
        A[own, 0] = shared + 2 * (c * EACH + np.arange(EACH))
        A[own, 1] = A[own, 0] + 1
        x[own] = rng.standard_normal(EACH)
    if not raw:
        x = np.round(x * 2.0 ** 32) / 2.0 ** 32
    return np.sort(A, axis=1), m, x


def _fewest_accepted(orc, A, y):
    """Fewest columns that a part accepts in the first iteration."""
    n, d = A.shape
    C, pitch = _parts(n, d)
    acc, _, _ = orc.score_all(A, y)
    return min(int(np.count_nonzero(acc[c * pitch:(c + 1) * pitch])) for c in range(C))


@pytest.mark.parametrize("raw", [False, True], ids=["grid", "raw"])
@pytest.mark.parametrize("case", list(CASES))
def test_more_accepted_columns_than_the_lists_hold(ccs, orc, case, raw):
    import torch
    A, m, x = _problem(case, raw)
    y = orc.measure(A, m, x)
    assert _parts(*A.shape)[0] == int(case[1]) and m <= 2560 and A.size <= 300000
    assert _fewest_accepted(orc, A, y) > 64
    ref = orc.parallel_l0(A, m, y, max_iter=25)
    csc, ptr, cols = upload_matrix(orc, A, m)
    yd = torch.from_numpy(y).cuda()
    for flags in (0, 2, 4):
        g = ccs.decode_parallel_l0(csc, ptr, cols, yd, max_iter=25, debug_flags=flags)
        assert_same_decode(g, ref)
        again = ccs.decode_parallel_l0(csc, ptr, cols, yd, max_iter=25, debug_flags=flags)
        assert_same_decode(again, ref)


@pytest.mark.parametrize("flags", [0, 2, 4])
def test_batch_with_long_lists(ccs, orc, flags):
    import torch
    items, refs = [], []
    for case in CASES:
        for raw in (False, True):
            A, m, x = _problem(case, raw)
            y = orc.measure(A, m, x)
            refs.append(orc.parallel_l0(A, m, y, max_iter=25))
            items.append((*upload_matrix(orc, A, m), torch.from_numpy(y).cuda()))
    for g, ref in zip(ccs.decode_batch(items, max_iter=25, history=True, debug_flags=flags), refs):
        assert_same_decode(g, ref)


def test_clusters_that_start_at_different_times(ccs, orc):
    """Batches of small problems on two streams beside decodes that fill the
    GPU: a cluster's CTAs start as SMs become free, each problem once and
    with its own results."""
    import torch
    probs = [inputs.make_problem(60001, 6000, 7, 600, 5)]
    probs += [inputs.make_problem(3001 + 997 * q, 400 + 60 * q, 7, 30 + 6 * q, 60 + q) for q in range(6)]
    items = [device_problem(ccs, p) for p in probs]
    refs = []
    for p in probs:
        A, y = oracle_problem(orc, p)
        refs.append(orc.parallel_l0(A, p.m, y))

    def outputs(chosen):
        return [(torch.full((probs[q].n,), float("nan"), dtype=torch.float64, device="cuda"),
                 torch.empty(probs[q].m, dtype=torch.float64, device="cuda")) for q in chosen]

    lanes = []
    for chosen in ([0], range(1, 7), range(1, 7)):
        bufs = outputs(chosen)
        pbs = [ccs.problem(*items[q], *b) for q, b in zip(chosen, bufs)]
        lanes.append((list(chosen), bufs, pbs, ccs.BatchGraph(pbs), torch.cuda.Stream()))
    torch.cuda.synchronize()
    for _ in range(20):
        for _, _, _, graph, stream in lanes:
            graph.launch(stream)
    torch.cuda.synchronize()
    for chosen, bufs, _, graph, _ in lanes:
        for q, (x, _), res in zip(chosen, bufs, graph.read_results()):
            assert (res.status, res.iterations, res.error) == \
                (refs[q]["status"], refs[q]["iterations"], 0)
            assert np.array_equal(x.cpu().numpy(), refs[q]["x_hat"])
        graph.close()


# n d just below and above a cluster size's entries; the last CTA's part short,
# and empty (160 columns a part: 6 full ones, 70 columns, none)
@pytest.mark.parametrize("shape, ctas", [((585, 70, 7, 7), 1), ((586, 70, 7, 7), 2), ((1170, 130, 7, 30), 2),
                                         ((1171, 130, 7, 30), 4), ((2341, 300, 7, 30), 8),
                                         ((1030, 160, 16, 12), 8)])
def test_cluster_sizes(ccs, orc, shape, ctas):
    n, m, d, k = shape
    C, pitch = _parts(n, d)
    assert C == ctas and (shape[0] != 1030 or 7 * pitch >= n)
    for values in ("gauss-grid", "gauss-raw"):
        p = inputs.make_problem(n, m, d, k, 300 + n, values)
        items = device_problem(ccs, p)
        A, y = oracle_problem(orc, p)
        ref = orc.parallel_l0(A, m, y, max_iter=30)
        for flags in (0, 2, 4):
            g = ccs.decode_parallel_l0(*items, max_iter=30, debug_flags=flags)
            assert_same_decode(g, ref)
            h = ccs.decode_batch([items, items], max_iter=30, history=True, debug_flags=flags)
            for b in h:
                assert_same_decode(b, ref)


@pytest.mark.parametrize("small, large", [(2, 4), (2, 3), (3, 4)])
def test_batch_around_two_fifths(ccs, orc, small, large):
    """From two fifths of small problems on they are decoded on chip; the
    results are the same on both sides."""
    probs = [inputs.make_problem(3001 + 1000 * q, 400 + 90 * q, 7, 40, 20 + q) for q in range(small)]
    probs += [inputs.make_problem(120001 + 10000 * q, 12001, 7 + 2 * (q % 2), 900, 30 + q)
              for q in range(large)]
    for g, p in zip(ccs.decode_batch([device_problem(ccs, p) for p in probs], history=True), probs):
        A, y_ref = oracle_problem(orc, p)
        assert_same_decode(g, orc.parallel_l0(A, p.m, y_ref))
