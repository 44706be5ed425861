"""Tree nodes of the panel factorizations at the edges of their kernels: rows
and columns around a thread's, a warp's, a CTA's and a cluster's share, nodes
one row or one column wide, ties and all-zero columns -- against the oracle."""
import numpy as np
import pytest

import oracle
from paper_1303_5837_gb300 import inputs
from tests.parity import check, lu_err

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-12  # of each element's first-order rounding scale


@pytest.fixture(scope="module")
def ca():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1303_5837_gb300 as ca
    ca.load()
    return ca


def to_dev(A):
    return torch.from_numpy(np.ascontiguousarray(np.asarray(A).T)).cuda().t()


def to_host(T):
    return np.asfortranarray(T.cpu().numpy())


def lu_case(ca, A, L, lv):
    n = A.shape[1]
    LU_o, ipiv_o, info_o, nt = oracle.calu(A, n, oracle.make_tree(L, lv))
    Ad = to_dev(A)
    ipiv, info = ca.tslu(Ad, ca.make_tree(L, lv))
    torch.cuda.synchronize()
    assert info.cpu().tolist() == [info_o, 0]
    assert np.array_equal(ipiv.cpu().numpy(), ipiv_o)
    return to_host(Ad), LU_o, nt


# (rows, columns, leaf rows, levels)
LU_NODES = [
    (1, 1, 1, [(0, 0)]), (5, 1, 5, [(0, 0)]), (3, 3, 3, [(0, 0)]), (31, 15, 31, [(0, 0)]), (33, 16, 33, [(0, 0)]),
    (257, 16, 257, [(0, 0)]), (97, 17, 97, [(0, 0)]), (128, 32, 128, [(0, 0)]), (129, 33, 129, [(0, 0)]),
    (64, 64, 64, [(0, 0)]), (65, 64, 65, [(0, 0)]), (256, 61, 256, [(0, 0)]), (513, 64, 513, [(0, 0)]),
    (2048, 64, 2048, [(0, 0)]), (2049, 64, 2049, [(0, 0)]),       # a register cluster's most rows, one more
    (65, 65, 65, [(0, 0)]), (128, 127, 128, [(0, 0)]), (129, 128, 129, [(0, 0)]), (1024, 128, 1024, [(0, 0)]),
    (1025, 96, 1025, [(0, 0)]),
    (20000, 24, 64, [(3, 1), (0, 0)]),                            # more nodes than SMs, three-way merges
    (1000, 40, 192, [(0, 1)]),                                    # a last leaf of 40 rows, one flat merge
    (700, 60, 128, [(0, 0)]),                                     # a promoted node
]


@pytest.mark.parametrize("m,n,L,lv", LU_NODES)
def test_lu_node_shapes(ca, m, n, L, lv):
    got, want, nt = lu_case(ca, inputs.gaussian(m, n, 11 * m + n), L, lv)
    assert nt == 0
    check(lu_err(got, want), TOL, (m, n, L))


@pytest.mark.parametrize("m,L", [(300, 300), (1000, 100), (640, 64)])
def test_lu_node_ties_take_the_first_row(ca, m, L):
    """+-1 entries: every comparison of a column ties, all arithmetic is exact."""
    A = np.asfortranarray(np.where(inputs.gaussian(m, 3, m) > 0, 1.0, -1.0))
    got, want, _ = lu_case(ca, A, L, [(2, 0), (0, 1)])
    assert np.array_equal(got, want)


@pytest.mark.parametrize("m,n,L", [(512, 48, 512), (100, 20, 100), (4000, 70, 250)])
def test_lu_node_zero_column_keeps_the_order(ca, m, n, L):
    A = inputs.gaussian(m, n, m * n)
    A[:, n // 2] = 0.0
    _, ipiv_o, info_o, _ = oracle.calu(A, n, oracle.make_tree(L))
    ipiv, info = ca.tslu(to_dev(A), ca.make_tree(L))
    torch.cuda.synchronize()
    assert info.cpu().tolist()[0] == info_o == n // 2 + 1
    assert np.array_equal(ipiv.cpu().numpy(), ipiv_o)
