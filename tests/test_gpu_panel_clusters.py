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
