"""Clusters of the register-resident panel nodes: the size a device can place,
waits that run out."""
import numpy as np
import pytest

import oracle
from paper_1303_5837_gb300 import inputs
from tests.parity import check, lu_err, qr_err

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


def tslu(ca, A, L):
    Ad = to_dev(A)
    ipiv, info = ca.tslu(Ad, ca.make_tree(L))
    torch.cuda.synchronize()
    return Ad.cpu().numpy(), ipiv.cpu().numpy(), info.cpu().tolist()


@pytest.mark.parametrize("m,n,L", [(400, 16, 400), (500, 30, 500), (1000, 64, 1000), (2048, 64, 2048), (500, 96, 500),
                                   (1024, 128, 1024), (3000, 100, 1000)])
def test_tournament_nodes_without_clusters_of_16(ca, m, n, L):
    """A device that places no cluster beyond the portable 8 CTAs: the same
    result, bit for bit."""
    A = inputs.gaussian(m, n, m + 3 * n)
    want = tslu(ca, A, L)
    ca.ca_test_cluster_hook(8)
    try:
        got = tslu(ca, A, L)
    finally:
        ca.ca_test_cluster_hook(0)
    assert got[2] == want[2] == [0, 0]
    assert np.array_equal(got[1], want[1]) and np.array_equal(got[0], want[0])


SHORT_WAIT = 2_000_000   # SM clock cycles, about 1 ms


@pytest.fixture
def withheld(ca):
    """The last CTA of every cluster sends nothing."""
    ca.ca_test_panel_hook(SHORT_WAIT, True)
    yield
    ca.ca_test_panel_hook()


# (rows, columns, leaf rows): every instantiation, 2 to 16 CTAs, a merge round
NODES = [(400, 16, 400), (60, 20, 60), (500, 32, 500), (300, 64, 300), (2048, 64, 2048), (500, 96, 500),
         (1024, 128, 1024), (900, 80, 300)]


@pytest.mark.parametrize("m,n,L", NODES)
def test_tournament_wait_that_runs_out(ca, withheld, m, n, L):
    """The kernel returns, the status tells, the interchanges stay inside the
    matrix; the next call is correct again."""
    A = inputs.gaussian(m, n, m + n)
    _, ipiv, info = tslu(ca, A, L)
    assert info[1] & ca.CA_STATUS_PANEL_TIMEOUT
    assert ipiv.min() >= 1 and ipiv.max() <= m and np.all(ipiv >= np.arange(1, n + 1))
    ca.ca_test_panel_hook()
    LU_o, ipiv_o, info_o, _ = oracle.calu(A, n, oracle.make_tree(L))
    LU, ipiv, info = tslu(ca, A, L)
    assert info == [info_o, 0] and np.array_equal(ipiv, ipiv_o)
    check(lu_err(LU, LU_o), TOL, (m, n, L))


# (TSQR nodes of more than 1024 rows wait for nobody)
@pytest.mark.parametrize("m,n,L", [(1000, 64, 1000) if c[0] == 2048 else c for c in NODES])
def test_tsqr_wait_that_runs_out(ca, withheld, m, n, L):
    A = inputs.gaussian(m, n, m + n)

    def tsqr():
        Ad = to_dev(A)
        _, info = ca.tsqr(Ad, ca.make_tree(L))
        torch.cuda.synchronize()
        return Ad.cpu().numpy(), info.cpu().tolist()

    assert tsqr()[1][1] & ca.CA_STATUS_PANEL_TIMEOUT
    ca.ca_test_panel_hook()
    QR_o, _ = oracle.caqr(A, n, oracle.make_tree(L))
    QR, info = tsqr()
    assert info == [0, 0]
    check(qr_err(QR, QR_o, n), TOL, (m, n, L))


def test_factorization_with_a_wait_that_runs_out(ca, withheld):
    """Several panels with look-ahead: every panel gives up, the call returns."""
    A = to_dev(inputs.gaussian(700, 700, 3))
    ipiv, info = ca.calu_factor(A, 64, ca.make_tree(128))
    torch.cuda.synchronize()
    assert info.cpu().tolist()[1] & ca.CA_STATUS_PANEL_TIMEOUT
    p = ipiv.cpu().numpy()
    assert np.all(p >= np.arange(1, 701)) and p.max() <= 700
