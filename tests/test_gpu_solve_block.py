"""Triangular solves of one block (up to 128 rows) with given factors: pivots at
the end of the range, triangles with a huge inverse."""
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


def to_dev(A):
    return torch.from_numpy(np.ascontiguousarray(np.asarray(A).T)).cuda().t()



def solve_factors(ca, LU, B):
    """calu_getrs with given factors and no interchanges."""
    n = len(LU)
    F, X = to_dev(LU), to_dev(B)
    ipiv = torch.arange(1, n + 1, dtype=torch.int32, device="cuda")
    ca.calu_getrs(F, ipiv, X)
    torch.cuda.synchronize()
    return X.cpu().numpy()


@pytest.mark.parametrize("n,nrhs", [(2, 2), (31, 1), (33, 3), (96, 16), (128, 5)])
def test_one_block_solve_with_tiny_pivots(ca, n, nrhs):
    """Pivots whose reciprocal overflows: the quotients are ordinary numbers,
    exact for powers of two."""
    X = inputs.gaussian(n, nrhs, n)
    X[::2] = np.ldexp(1.0, np.arange(n)[::2, None] % 9)
    LU = np.eye(n) * np.ldexp(1.0, -1030)
    B = np.ldexp(X, -1030)                    # rounded to a subnormal where X is not a power of two
    assert np.array_equal(solve_factors(ca, LU, B), np.ldexp(B, 1030))


@pytest.mark.parametrize("n,nrhs", [(32, 1), (64, 4), (100, 16), (128, 2)])
@pytest.mark.parametrize("lower", [True, False])
def test_one_block_solve_has_the_residual_of_substitution(ca, n, nrhs, lower):
    """-1 everywhere off the diagonal: the inverse has elements of 2^(n - 2).
    Substitution solves (T + E) x = b with |E| <= 1.1 n u |T|, columnwise."""
    T = np.eye(n) - np.tril(np.ones((n, n)), -1)
    if not lower:
        T = T.T
    b = T @ inputs.gaussian(n, nrhs, n)
    X = solve_factors(ca, T, b)
    r = np.abs(T.astype(np.longdouble) @ X.astype(np.longdouble) - b)
    assert np.all(r <= 1.1 * n * 2.0 ** -53 * (np.abs(T) @ np.abs(X)) + n * 2.0 ** -62 * np.abs(b))
