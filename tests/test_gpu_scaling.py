"""Matrices whose rows or columns differ in scale by many orders of magnitude:
what a factorization keeps of the small ones."""
import numpy as np
import pytest

from paper_1303_5837_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ca():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1303_5837_gb300 as ca
    ca.load()
    return ca


@pytest.mark.parametrize("name,first,rest", [("float32", 1e-17, 1e-26), ("float64", 1e-150, 1e-170)])
@pytest.mark.parametrize("m,n,L", [(40, 8, 40), (200, 30, 200), (250, 60, 250)])
def test_batched_qr_of_small_columns(ca, name, first, rest, m, n, L):
    """The first reflector meets columns so much smaller that a product of two
    elements is not a normal number, while v^T A is: row 0 of R is good to
    m + 10 units of rounding of its column's norm (a sum of m products)."""
    dt, tdt = (np.float32, torch.float32) if name == "float32" else (np.float64, torch.float64)
    A = inputs.gaussian(m, n, m + n)
    A[:, 0] *= first
    A[:, 1:] *= rest
    A = A.astype(dt)
    dev = torch.from_numpy(np.ascontiguousarray(A.T)).to("cuda", tdt).t()
    bf = ca.BatchedFactor([dev], ["qr"], [n], [ca.make_tree(L)])
    bf.run()
    torch.cuda.synchronize()
    a = A[:, 0].astype(np.float64) / first
    C = A[:, 1:].astype(np.float64) / rest
    beta = -np.copysign(np.linalg.norm(a), a[0])
    v = a.copy()
    v[0] -= beta
    want = C[0] - v[0] * (2.0 / (v @ v)) * (v @ C)
    got = dev[0, 1:].cpu().numpy().astype(np.float64) / rest
    assert np.all(np.abs(got - want) <= (m + 10) * np.finfo(dt).eps * np.linalg.norm(C, axis=0))
