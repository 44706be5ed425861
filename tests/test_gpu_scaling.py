"""Matrices whose rows or columns differ in scale by many orders of magnitude:
what a factorization keeps of the small ones."""
import numpy as np
import pytest

import oracle
from paper_1303_5837_gb300 import inputs
from tests.parity import check, lu_err

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


@pytest.mark.parametrize("m,n,L", [(100, 100, 100), (128, 70, 128), (120, 120, 128)])
def test_tsqr_of_small_columns(ca, m, n, L):
    """The same in a single node of more than 64 columns and up to 128 rows."""
    A = inputs.gaussian(m, n, m + n)
    C = A[:, 1:].copy()
    a = A[:, 0].copy()
    A[:, 0] *= 1e-150
    A[:, 1:] *= 1e-170
    dev = to_dev(A)
    ca.tsqr(dev, ca.make_tree(L))
    beta = -np.copysign(np.linalg.norm(a), a[0])
    v = a.copy()
    v[0] -= beta
    want = C[0] - v[0] * (2.0 / (v @ v)) * (v @ C)
    got = dev[0, 1:].cpu().numpy() / 1e-170
    assert np.all(np.abs(got - want) <= (m + 12) * 2.0 ** -52 * np.linalg.norm(C, axis=0))


def to_dev(A):
    return torch.from_numpy(np.ascontiguousarray(np.asarray(A).T)).cuda().t()


def to_host(T):
    return np.asfortranarray(T.cpu().numpy())


@pytest.mark.parametrize("b", [32, 64, 100])
@pytest.mark.parametrize("delta", [1.0, 1e-2, 1e-4, 1e-8, 1e-12, 1e-40, 1e-200])
def test_lu_keeps_weak_couplings(ca, b, delta):
    """Two groups of unknowns, numbered in turn, coupled by delta: the row of
    L21 is (1, delta, 1, ...), the column of U12 (delta, 1, delta, ...) and the
    element wanted is of size delta.  Every element is good to 1e-12 of its
    first-order rounding scale (|L||U|)_ij, as on the FP64 pipe; no scaling of
    rows and columns undoes this."""
    n, L = 420, 128
    A = inputs.gaussian(n, n, 5 * b)
    k = np.arange(n) % 2
    A = np.asfortranarray(np.where(k[:, None] == k[None, :], A, delta * A))
    LU_o, ipiv_o, info_o, _ = oracle.calu(A, b, oracle.make_tree(L))
    F = to_dev(A)
    before = ca.ca_launch_count(9)
    ipiv, info = ca.calu_factor(F, b, ca.make_tree(L))
    torch.cuda.synchronize()
    assert ca.ca_launch_count(9) > before
    assert info.cpu().tolist() == [info_o, 0]
    assert np.array_equal(ipiv.cpu().numpy(), ipiv_o)
    check(lu_err(to_host(F), LU_o), 1e-12, (b, delta))


@pytest.mark.parametrize("m,n,b", [(190, 190, 64), (333, 421, 48), (421, 333, 32), (385, 513, 128), (300, 161, 128)])
def test_lu_weak_couplings_in_some_blocks(ca, m, n, b):
    """The first panel's unknowns numbered in turn, the others group by group:
    only the blocks that join a group's rows to the other's columns hold
    elements that the digits cannot stand for; ragged tiles on both sides."""
    L, delta = 128, 1e-9
    A = inputs.gaussian(m, n, m + n + b)
    i, K = np.arange(max(m, n)), min(m, n)
    group = np.where((i < b) | (i >= K), i % 2, i >= b + (K - b) // 2)   # as many rows as columns in each
    row, col = group[:m], group[:n]
    A = np.asfortranarray(np.where(row[:, None] == col[None, :], A, delta * A))
    LU_o, ipiv_o, info_o, _ = oracle.calu(A, b, oracle.make_tree(L))
    F = to_dev(A)
    before = ca.ca_launch_count(9)
    ipiv, info = ca.calu_factor(F, b, ca.make_tree(L))
    torch.cuda.synchronize()
    assert (ca.ca_launch_count(9) > before) == (K - b >= 64)
    assert info.cpu().tolist() == [info_o, 0]
    assert np.array_equal(ipiv.cpu().numpy(), ipiv_o)
    check(lu_err(to_host(F), LU_o), 1e-12, (m, n, b))


def qr_run(ca, A, b, tree, work=None):
    F = to_dev(A)
    before = ca.ca_launch_count(9)
    _, info = ca.caqr_factor(F, b, tree, work=work)
    torch.cuda.synchronize()
    assert info.cpu().tolist() == [0, 0]
    return to_host(F), ca.ca_launch_count(9) > before


@pytest.mark.parametrize("w", [0, 4, 8, 12, 20, 30, 40])
@pytest.mark.parametrize("b,L,lv", [(64, 128, [(0, 0)]), (100, 300, [(0, 1)])])
def test_qr_keeps_light_rows_below_heavy_ones(ca, w, b, L, lv):
    """The first b / 2 rows weighted by 2^w (equality-constrained least squares by
    weights), so that the first panel has heavy reflectors and light ones: the
    rows of R below them are those of the light part.  Their distance from the
    oracle, columnwise, is at most 11 times that of the same factorization on
    the FP64 pipe (ten times its error, and the oracle's own is in both)."""
    m, n = 2000, 1400
    A = inputs.gaussian(m, n, 31 + b)
    h = b // 2
    A[:h] *= 2.0 ** w
    QR_o, _ = oracle.caqr(A, b, oracle.make_tree(L, lv))
    t = ca.make_tree(L, lv)
    got, digits = qr_run(ca, A, b, t)
    work = torch.empty(ca.ca_caqr_workspace(m, b, b, t)[1] // 8, dtype=torch.float64, device="cuda")
    pipe, other = qr_run(ca, A, b, t, work)
    assert digits and not other

    def light(X):
        return np.triu(X[:n])[h:, h:]

    scale = np.linalg.norm(light(QR_o), axis=0)
    err = [float((np.abs(light(X) - light(QR_o)) / scale).max()) for X in (got, pipe)]
    assert err[0] <= 11 * max(err[1], 2.0 ** -52), (w, err)
