"""The FP64 trailing updates on the tensor cores (7 exact digits) against the
oracle and against the same factorization on the FP64 pipe: ragged tiles,
narrow panels, badly scaled rows and columns, values that are not finite."""
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


def lu_on_fp64_pipe(ca, A, b, tree):
    """The workspace of a single panel has no room for digits."""
    m, n = A.shape
    F = to_dev(A)
    work = torch.empty(ca.ca_calu_workspace(m, b, b, tree) // 8, dtype=torch.float64, device="cuda")
    assert work.numel() * 8 < ca.ca_calu_workspace(m, n, b, tree)
    before = ca.ca_launch_count(9)
    ipiv, info = ca.calu_factor(F, b, tree, work=work)
    torch.cuda.synchronize()
    assert ca.ca_launch_count(9) == before
    return to_host(F), ipiv.cpu().numpy(), info.cpu().tolist()


def lu_on_tensor_cores(ca, A, b, tree):
    F = to_dev(A)
    before = ca.ca_launch_count(9)
    ipiv, info = ca.calu_factor(F, b, tree)
    torch.cuda.synchronize()
    assert ca.ca_launch_count(9) > before
    return to_host(F), ipiv.cpu().numpy(), info.cpu().tolist()


@pytest.mark.parametrize("m,n,b,L", [(256, 256, 64, 64), (333, 421, 48, 128), (421, 333, 16, 64), (400, 400, 100, 128),
                                     (600, 300, 17, 96), (500, 650, 128, 256)])
def test_lu_update_matches_the_oracle(ca, m, n, b, L):
    A = inputs.gaussian(m, n, 3 * m + n + b)
    LU_o, ipiv_o, info_o, nt = oracle.calu(A, b, oracle.make_tree(L))
    assert nt == 0
    for got, ipiv, info in (lu_on_tensor_cores(ca, A, b, ca.make_tree(L)), lu_on_fp64_pipe(ca, A, b, ca.make_tree(L))):
        assert info == [info_o, 0]
        assert np.array_equal(ipiv, ipiv_o)
        check(lu_err(got, LU_o), TOL, (m, n, b))


@pytest.mark.parametrize("rows,cols", [(60, 0), (0, 60), (60, 60)])
def test_lu_update_keeps_badly_scaled_rows_and_columns(ca, rows, cols):
    """Rows and columns scaled by random powers of two up to 2^+-rows / cols:
    every element keeps its relative accuracy, as on the FP64 pipe."""
    n, b, L = 400, 64, 64
    g = np.random.default_rng(rows + 7 * cols)
    A = inputs.gaussian(n, n, 77)
    A = np.asfortranarray(np.ldexp(np.ldexp(A, g.integers(-rows, rows + 1, (n, 1))), g.integers(-cols, cols + 1, (1, n))))
    LU_o, ipiv_o, info_o, nt = oracle.calu(A, b, oracle.make_tree(L))
    assert nt == 0
    got, ipiv, info = lu_on_tensor_cores(ca, A, b, ca.make_tree(L))
    assert info == [info_o, 0]
    assert np.array_equal(ipiv, ipiv_o)
    check(lu_err(got, LU_o), TOL, (rows, cols))


@pytest.mark.parametrize("value", [np.inf, np.nan, 1e305, 1e-310])
def test_lu_update_of_odd_values_is_the_fp64_pipes(ca, value):
    """Values that are not finite or near the ends of the range: the same
    elements are finite, infinite and NaN as on the FP64 pipe."""
    A = inputs.gaussian(320, 320, 9)
    A[7, 250] = value      # outside the first panel: met in U12 first
    t = ca.make_tree(64)
    got, ipiv, info = lu_on_tensor_cores(ca, A, 64, t)
    want, ipiv_w, info_w = lu_on_fp64_pipe(ca, A, 64, t)
    assert info == info_w
    first = np.arange(250)  # the columns the value has not reached
    assert np.array_equal(ipiv[:192], ipiv_w[:192])
    assert np.array_equal(np.isnan(got[:, first]), np.isnan(want[:, first]))
    assert np.array_equal(np.isnan(got[:192]), np.isnan(want[:192]))
    assert np.array_equal(np.isinf(got[:192]), np.isinf(want[:192]))
    fin = np.isfinite(want[:192])
    assert np.allclose(got[:192][fin], want[:192][fin], rtol=1e-9, atol=1e-9)


def qr_run(ca, A, b, tree, single_panel_workspace):
    m, n = A.shape
    F = to_dev(A)
    work = None
    if single_panel_workspace:
        work = torch.empty(ca.ca_caqr_workspace(m, b, b, tree)[1] // 8, dtype=torch.float64, device="cuda")
        assert work.numel() * 8 < ca.ca_caqr_workspace(m, n, b, tree)[1]
    before = ca.ca_launch_count(9)
    qtree, info = ca.caqr_factor(F, b, tree, work=work)
    torch.cuda.synchronize()
    assert (ca.ca_launch_count(9) > before) != single_panel_workspace
    return to_host(F), qtree.cpu().numpy(), info.cpu().tolist()


@pytest.mark.parametrize("m,n,b,L,lv", [(2000, 1500, 64, 128, [(0, 0)]), (2501, 1111, 100, 300, [(4, 1), (0, 1)]),
                                        (3000, 1000, 128, 1024, [(0, 1)])])
def test_qr_update_matches_the_oracle(ca, m, n, b, L, lv):
    A = inputs.gaussian(m, n, m + n + b)
    t_o = oracle.make_tree(L, lv)
    QR_o, T_o = oracle.caqr(A, b, t_o)
    for alone in (False, True):
        got, qtree, info = qr_run(ca, A, b, ca.make_tree(L, lv), alone)
        assert info == [0, 0]
        check(qr_err(got, QR_o, b), TOL, (m, n, b, alone))
        check(qtree_err(qtree, T_o, QR_o, b, t_o, oracle.tree_counts), TOL, (m, n, b, alone))


@pytest.mark.parametrize("value", [np.inf, np.nan, 1e-310])
def test_qr_update_of_odd_values_is_the_fp64_pipes(ca, value):
    A = inputs.gaussian(2000, 1400, 5)
    A[70, 1300] = value
    t = ca.make_tree(128)
    got, _, _ = qr_run(ca, A, 64, t, False)
    want, _, _ = qr_run(ca, A, 64, t, True)
    clean = np.arange(1280)  # whole panels before the value's column
    assert np.all(np.isfinite(got[:, clean]) == np.isfinite(want[:, clean]))
    assert np.array_equal(np.isfinite(got[:1280, 1300]), np.isfinite(want[:1280, 1300]))
    assert np.allclose(got[:1280][:, clean], want[:1280][:, clean], rtol=1e-9, atol=1e-9)
