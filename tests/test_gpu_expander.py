"""The expander's construction paths, bit for bit against the oracle: grouped
(rows sorted a group at a time on chip), ranks packed beside the row indices
(too many groups, or no room for a row beside a column), and neither (row
indices that leave no bits for a rank)."""
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


# n around a block of columns, n d not a multiple of 4, d = m, one row, rows
# without columns, groups of one row and of many, the last group short; then
# shapes beyond the groups: more than 8192 of them with rows up to the warp
# sort's sizes
SHAPES = [(1, 1, 1), (3, 2, 1), (255, 5, 5), (257, 9, 3), (511, 16, 16), (4001, 700, 5),
          (513, 100003, 3), (30011, 400, 7), (60001, 1025, 9), (65537, 900, 7),
          (100003, 70001, 3), (60001, 300, 5), (30001, 1, 1), (40001, 17, 3),
          (200001, 1000, 7), (300007, 33, 1), (131073, 800, 8), (250003, 2999, 16),
          (1000003, 1500, 2), (2 ** 21 + 5, 30011, 15), (2 ** 20 + 3, 2 ** 17 + 1, 7),
          (5000003, 2500001, 5), (2 ** 24 + 1, 1100003, 3)]


@pytest.mark.parametrize("n,m,d", SHAPES)
def test_expander_paths_bitwise(ccs, orc, n, m, d):
    csc, ptr, cols = ccs.make_expander(n, m, d, 4242 + n)
    A = orc.make_expander(n, m, d, 4242 + n)
    ptr_ref, cols_ref = orc.transpose(A, m)
    assert np.array_equal(csc.cpu().numpy(), A)
    assert np.array_equal(ptr.cpu().numpy(), ptr_ref)
    assert np.array_equal(cols.cpu().numpy(), cols_ref)


def test_expander_without_room_for_ranks(ccs, orc):
    import torch
    n, m, d = 1003, 2 ** 29, 3
    csc, ptr, cols = ccs.make_expander(n, m, d, 77)
    A = orc.make_expander(n, m, d, 77)
    assert np.array_equal(csc.cpu().numpy(), A)
    rows = torch.from_numpy(A.reshape(-1).astype(np.int64)).cuda()
    order = torch.sort(rows, stable=True)
    assert torch.equal(cols.long(), order.indices // d)
    at = torch.unique(rows)  # ptr steps only after these rows
    assert int(ptr[0]) == 0 and int(ptr[m]) == n * d
    assert torch.equal(ptr[at + 1], torch.searchsorted(order.values, at, right=True))
    assert int((ptr[1:] != ptr[:-1]).sum()) == at.numel()
