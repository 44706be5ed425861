"""Tree nodes of the panel factorizations at the edges of their kernels: rows
and columns around a thread's, a warp's, a CTA's and a cluster's share, nodes
one row or one column wide, ties and all-zero columns -- against the oracle."""
import numpy as np
import pytest

import oracle
from paper_1303_5837_gb300 import inputs
from tests.parity import check, lu_err, qr_err, qtree_err

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


# (rows, columns, leaf rows, levels)
QR_NODES = [
    (1, 1, 1, [(0, 0)]), (16, 16, 16, [(0, 0)]), (33, 17, 33, [(0, 0)]), (256, 64, 256, [(0, 0)]),
    (70, 65, 70, [(0, 0)]), (128, 128, 128, [(0, 0)]), (256, 127, 256, [(0, 0)]), (257, 100, 257, [(0, 0)]),
    (513, 128, 513, [(0, 0)]), (1024, 128, 1024, [(0, 0)]), (1025, 96, 1025, [(0, 0)]),
    (1024, 128, 128, [(0, 0)]),                # binary merges of equal heights
    (1400, 110, 150, [(3, 1), (0, 1)]),        # flat merges, a last leaf shorter than the panel is wide
    (900, 70, 280, [(0, 1)]),                  # the last child's R is shorter: rows in their own order
    (700, 60, 128, [(0, 0)]), (1000, 40, 192, [(0, 1)]), (6000, 24, 64, [(3, 1), (0, 0)]),
]


def qr_case(ca, A, L, lv):
    n = A.shape[1]
    t_o = oracle.make_tree(L, lv)
    QR_o, T_o = oracle.caqr(A, n, t_o)
    Ad = to_dev(A)
    qtree, info = ca.tsqr(Ad, ca.make_tree(L, lv))
    torch.cuda.synchronize()
    assert info.cpu().tolist() == [0, 0]
    check(qr_err(to_host(Ad), QR_o), TOL, (A.shape, L))
    check(qtree_err(qtree.cpu().numpy(), T_o, QR_o, n, t_o, oracle.tree_counts), TOL, (A.shape, L))


@pytest.mark.parametrize("m,n,L,lv", QR_NODES)
def test_qr_node_shapes(ca, m, n, L, lv):
    qr_case(ca, inputs.gaussian(m, n, 13 * m + n), L, lv)


@pytest.mark.parametrize("m,n,L,lv", [c for c in QR_NODES if c[1] > 1] + [(512, 70, 512, [(0, 0)])])
def test_qr_node_shapes_of_the_digit_form(ca, m, n, L, lv):
    """One panel of the digit factorization, which keeps its own order of sums."""
    A = inputs.gaussian(m, n, 13 * m + n)
    t_o = oracle.make_tree(L, lv)
    QR_o, T_o = oracle.caqr(A, n, t_o)
    Ad = to_dev(A)
    qtree, info = ca.caqr_factor_mixed(Ad, n, ca.make_tree(L, lv))
    torch.cuda.synchronize()
    assert info.cpu().tolist() == [0, 0]
    check(qr_err(to_host(Ad), QR_o), TOL, (m, n, L))
    check(qtree_err(qtree.cpu().numpy(), T_o, QR_o, n, t_o, oracle.tree_counts), TOL, (m, n, L))


@pytest.mark.parametrize("scale", [1e-200, 1e150, 1e-305])
@pytest.mark.parametrize("m,n,L", [(200, 24, 100), (600, 100, 300)])
def test_qr_node_reflectors_at_the_ends_of_the_range(ca, m, n, L, scale):
    """Norms whose squares leave the normal range, or come near its ends,
    take the library's square root and divisions: as the oracle where its sums
    of squares are finite, the same non-finite elements otherwise."""
    A = inputs.gaussian(m, n, m + n) * scale
    QR_o, _ = oracle.caqr(A, n, oracle.make_tree(L))
    Ad = to_dev(A)
    ca.tsqr(Ad, ca.make_tree(L))
    got = to_host(Ad)
    assert np.array_equal(np.isfinite(got), np.isfinite(QR_o))
    if scale == 1e150:
        check(qr_err(got / scale, QR_o / scale), 1e-9)


def test_qr_node_zero_column(ca):
    """A column that is zero below its diagonal: tau = 0, nothing changes."""
    A = inputs.gaussian(500, 90, 4)
    A[:, 0] = 0.0
    A[0, 0] = 2.0
    QR_o, _ = oracle.caqr(A, 90, oracle.make_tree(500))
    Ad = to_dev(A)
    ca.tsqr(Ad, ca.make_tree(500))
    check(qr_err(to_host(Ad), QR_o), TOL)


# batched QR items around the sizes where a node leaves the registers:
# (op, m, n, b, leaf rows, levels)
QR_ITEMS = [("qr", m, n, n, L, lv) for m, n, L, lv in [
    (512, 32, 512, [(0, 0)]), (513, 32, 513, [(0, 0)]), (512, 33, 512, [(0, 0)]), (256, 64, 256, [(0, 0)]),
    (257, 64, 257, [(0, 0)]), (17, 16, 17, [(0, 0)]), (1024, 31, 64, [(0, 1)]), (1100, 64, 64, [(4, 1), (0, 1)]),
    (1000, 30, 160, [(0, 1)]), (70, 20, 25, [(0, 1)])]] + [("qr", 700, 200, 32, 512, [(0, 1)]),
                                                           ("qr", 600, 150, 64, 256, [(0, 0)])]


@pytest.mark.parametrize("name", ["float64", "float32"])
def test_batched_qr_node_shapes(ca, name):
    dt, tdt, tol = (np.float64, torch.float64, TOL) if name == "float64" else (np.float32, torch.float32, 1e-4)
    mats = [inputs.gaussian(c[1], c[2], 40 + i).astype(dt) for i, c in enumerate(QR_ITEMS)]
    devs = [torch.from_numpy(np.ascontiguousarray(A.T)).to("cuda", tdt).t() for A in mats]
    bf = ca.BatchedFactor(devs, ["qr"] * len(mats), [c[3] for c in QR_ITEMS],
                          [ca.make_tree(c[4], c[5]) for c in QR_ITEMS])
    bf.run()
    torch.cuda.synchronize()
    for i, (c, A) in enumerate(zip(QR_ITEMS, mats)):
        t = oracle.make_tree(c[4], c[5])
        QR_o, T_o = oracle.caqr(A, c[3], t, dtype=dt)
        check(qr_err(devs[i].cpu().numpy(), QR_o, c[3]), tol, c)
        check(qtree_err(bf.qtree(i).cpu().numpy(), T_o, QR_o, c[3], t, oracle.tree_counts), tol, c)
        assert bf.info(i).cpu().tolist() == [0, 0], c


@pytest.mark.parametrize("n", [2, 31, 32, 33, 64, 65, 96, 127, 128, 129, 300])
@pytest.mark.parametrize("nrhs", [1, 5, 16, 17])
def test_solve_sizes(ca, n, nrhs):
    """Sub-blocks of the triangular solves: a diagonally dominant matrix, so
    the solution is good to a few n units of rounding."""
    A = inputs.gaussian(n, n, n) + 4.0 * np.sqrt(n) * np.eye(n)
    X = inputs.gaussian(n, nrhs, 7)
    F, Y = to_dev(A), to_dev(A @ X)
    ipiv, _ = ca.calu_factor(F, 64, ca.make_tree(128))
    ca.calu_getrs(F, ipiv, Y)
    torch.cuda.synchronize()
    assert np.abs(to_host(Y) - X).max() <= 1e-11
    Q, Y = to_dev(A), to_dev(A @ X)
    qtree, _ = ca.caqr_factor(Q, 64, ca.make_tree(128))
    ca.caqr_geqrs(Q, 64, ca.make_tree(128), qtree, Y)
    torch.cuda.synchronize()
    assert np.abs(to_host(Y) - X).max() <= 1e-11


@pytest.mark.parametrize("n,nrhs", [(130, 16), (200, 3), (333, 16), (100, 9)])
def test_solve_does_not_read_what_an_earlier_one_left(ca, n, nrhs):
    """Rows past a short last block: a solve of NaN right-hand sides first, so
    that whatever the same kernel left behind is not finite."""
    A = inputs.gaussian(n, n, n) + 4.0 * np.sqrt(n) * np.eye(n)
    X = inputs.gaussian(n, nrhs, 7)
    F, Y, bad = to_dev(A), to_dev(A @ X), to_dev(np.full((n, nrhs), np.nan))
    ipiv, _ = ca.calu_factor(F, 64, ca.make_tree(128))
    for _ in range(40):
        ca.calu_getrs(F, ipiv, bad.clone())
    ca.calu_getrs(F, ipiv, Y)
    torch.cuda.synchronize()
    assert np.abs(to_host(Y) - X).max() <= 1e-11


@pytest.mark.parametrize("m,n,b,L,lv", [(600, 100, 200, 256, [(0, 0)]), (700, 128, 129, 700, [(0, 0)]),
                                        (900, 64, 300, 300, [(0, 1)]), (100, 20, 150, 150, [(0, 0)])])
def test_t_blocks_wider_than_the_matrix(ca, m, n, b, L, lv):
    """A panel width beyond the matrix and beyond 128: every b x b block of the
    store is written, zero outside the corner of the panel's T."""
    A = inputs.gaussian(m, n, m + b)
    t_o = oracle.make_tree(L, lv)
    QR_o, T_o = oracle.caqr(A, b, t_o)
    Ad = to_dev(A)
    qtree = torch.full((ca.ca_caqr_workspace(m, n, b, ca.make_tree(L, lv))[0] // 8,), float("nan"), dtype=torch.float64,
                       device="cuda")
    ca.caqr_factor(Ad, b, ca.make_tree(L, lv), qtree=qtree)
    torch.cuda.synchronize()
    check(qr_err(to_host(Ad), QR_o, b), TOL, (m, n, b))
    check(qtree_err(qtree.cpu().numpy(), T_o, QR_o, b, t_o, oracle.tree_counts), TOL, (m, n, b))
    blocks = qtree.view(-1, b, b)
    assert not torch.any(blocks[:, n:, :]) and not torch.any(blocks[:, :, n:])
