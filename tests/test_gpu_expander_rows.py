"""Expanders of very many rows: the row offsets on both sides of the sizes at
which the block totals get a scan of their own (1024 blocks of 1024 rows), rows
that are sorted only if one of them holds two columns, and a construction time
that grows with the number of rows, not its square."""
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


# n > 2^25: six bits left for a row beside a column, so that these m take the
# row-by-row construction
@pytest.mark.parametrize("m", [2 ** 20 - 1, 2 ** 20, 2 ** 20 + 1, 2 ** 21 + 1025, 3 * 2 ** 20])
def test_offsets_around_the_scan_of_totals(ccs, orc, m):
    n, d = 2 ** 25 + 1, 1
    csc, ptr, cols = ccs.make_expander(n, m, d, 9 + m)
    A = orc.make_expander(n, m, d, 9 + m)
    ptr_ref, cols_ref = orc.transpose(A, m)
    assert np.array_equal(csc.cpu().numpy(), A)
    assert np.array_equal(ptr.cpu().numpy(), ptr_ref)
    assert np.array_equal(cols.cpu().numpy(), cols_ref)


@pytest.mark.parametrize("m", [2 ** 22, 2 ** 22 + 1])
def test_both_ways_to_place_the_entries(ccs, orc, m):
    """Counted again, and by the ranks that the count handed out."""
    n, d = 2 ** 24 + 3, 3
    csc, ptr, cols = ccs.make_expander(n, m, d, 5)
    A = orc.make_expander(n, m, d, 5)
    ptr_ref, cols_ref = orc.transpose(A, m)
    assert np.array_equal(csc.cpu().numpy(), A)
    assert np.array_equal(ptr.cpu().numpy(), ptr_ref)
    assert np.array_equal(cols.cpu().numpy(), cols_ref)


def test_time_grows_with_the_rows(ccs):
    """Four times the rows: about four times the passes over them (a sum over
    all totals before it in every block makes it 13 times)."""
    import torch

    def best(m):
        n, d = 1003, 3
        csc = torch.empty(n, d, dtype=torch.int32, device="cuda")
        ptr = torch.empty(m + 1, dtype=torch.int64, device="cuda")
        cols = torch.empty(n * d, dtype=torch.int32, device="cuda")
        ws = ccs.workspace(ccs.ccs_workspace_size(ccs.OP_MAKE_EXPANDER, n, m, d))
        times = []
        for _ in range(4):
            e0, e1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            e0.record()
            ccs.ccs_make_expander(n, m, d, 77, csc, ptr, cols, ws)
            e1.record()
            torch.cuda.synchronize()
            times.append(e0.elapsed_time(e1))
        return min(times)

    assert best(2 ** 29) < 8 * best(2 ** 27)


# about one expected pair of entries in a row (entries^2 / 2m), and hardly any
@pytest.mark.parametrize("n,m,d", [(2895, 2 ** 26, 4), (2897, 2 ** 26, 4), (1003, 2 ** 26, 3)])
def test_rows_that_most_likely_need_no_sort(ccs, orc, n, m, d):
    """Eight seeds each: some draw two columns into a row (which must come out
    ascending), others do not."""
    import torch
    longest = set()
    for seed in range(8):
        csc, ptr, cols = ccs.make_expander(n, m, d, seed)
        A = orc.make_expander(n, m, d, seed)
        assert np.array_equal(csc.cpu().numpy(), A)
        rows = torch.from_numpy(A.reshape(-1).astype(np.int64)).cuda()
        order = torch.sort(rows, stable=True)
        assert torch.equal(cols.long(), order.indices // d)
        assert torch.equal(ptr[1:], torch.searchsorted(order.values, torch.arange(m, device="cuda"),
                                                       right=True))
        longest.add(int((ptr[1:] - ptr[:-1]).max()))
    assert longest == {1, 2} or (n == 1003 and 1 in longest)


def test_rows_without_pairs_cost_no_sort(ccs):
    """2^27 rows with one column at most are drawn without the pass that sorts
    rows, which takes most of the time where some hold two."""
    import torch
    times = []
    for n, d in ((1003, 3), (40009, 3)):  # 0.03 and 54 expected pairs
        m = 2 ** 27
        csc = torch.empty(n, d, dtype=torch.int32, device="cuda")
        ptr = torch.empty(m + 1, dtype=torch.int64, device="cuda")
        cols = torch.empty(n * d, dtype=torch.int32, device="cuda")
        ws = ccs.workspace(ccs.ccs_workspace_size(ccs.OP_MAKE_EXPANDER, n, m, d))
        best = float("inf")
        for _ in range(4):
            e0, e1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            e0.record()
            ccs.ccs_make_expander(n, m, d, 77, csc, ptr, cols, ws)
            e1.record()
            torch.cuda.synchronize()
            best = min(best, e0.elapsed_time(e1))
        times.append(best)
    assert times[0] < 0.5 * times[1]  # the second is sorted
