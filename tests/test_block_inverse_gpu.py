"""The inverses of the diagonal blocks (M^-1 of the block-Jacobi PCG), value for
value: a quotient formed as a product with a reciprocal has one rounding more.

For a block-diagonal system and a right-hand side of one 1 per camera, PCG ends
after its first iteration with x = alpha z, z a column of every camera's M^-1 as
it is stored, alpha one number for the whole system (1 but for rounding).  The reference repeats the factorisation operation by operation in
the same precision, with quotients, and fused multiply-adds where the kernels'
sums have them; it agrees in every value but for the rare ones whose emulated
FP32 multiply-add is rounded twice (2^-29 of them).  With reciprocals and
products about half of the values differ."""
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2307_08383_gb300.build import build
    build()
    import paper_2307_08383_gb300 as mod
    return mod


def blocks(n, c, seed, T):
    rng = np.random.default_rng(seed)
    q, _ = np.linalg.qr(rng.standard_normal((n, c, c)))
    d = 10.0 ** rng.uniform(0, 3, (n, 1, c))
    a = ((q * d) @ q.transpose(0, 2, 1)).astype(T)
    return np.tril(a) + np.tril(a, -1).transpose(0, 2, 1)


def fma32(a, b, c):
    return (a.astype(np.float64) * b + c).astype(np.float32)


def inverse32(A):
    """A^-1 = L^-T L^-1 of n 6x6 blocks in FP32."""
    one, zero = np.float32(1), np.zeros(len(A), np.float32)
    L = np.zeros_like(A)
    for i in range(6):
        for j in range(i + 1):
            s = A[:, i, j].copy()
            for k in range(j):
                s = fma32(-L[:, i, k], L[:, j, k], s)
            L[:, i, j] = np.sqrt(s) if i == j else s / L[:, j, j]
    X = np.zeros_like(A)  # L^-1
    for i in range(6):
        X[:, i, i] = one / L[:, i, i]
        for j in range(i):
            s = zero
            for k in range(j, i):
                s = fma32(L[:, i, k], X[:, k, j], s)
            X[:, i, j] = -s * X[:, i, i]
    M = np.zeros_like(A)
    for i in range(6):
        for j in range(i, 6):
            s = zero
            for k in range(j, 6):
                s = fma32(X[:, k, i], X[:, k, j], s)
            M[:, i, j] = M[:, j, i] = s
    return M


def fma64(a, b, c):
    return float(Fraction(a) * Fraction(b) + Fraction(c))


def column64(A, q):
    """Column q of A^-1 by two substitutions, FP64."""
    c = len(A)
    L = [[0.0] * c for _ in range(c)]
    for i in range(c):
        for j in range(i + 1):
            s = 0.5 * (float(A[i, j]) + float(A[j, i]))
            for k in range(j):
                s = fma64(-L[i][k], L[j][k], s)
            L[i][j] = float(np.sqrt(s)) if i == j else s / L[j][j]
    x = [0.0] * c
    for i in range(c):
        s = 1.0 if i == q else 0.0
        for k in range(i):
            s = fma64(-L[i][k], x[k], s)
        x[i] = s / L[i][i]
    for i in reversed(range(c)):
        s = x[i]
        for k in range(i + 1, c):
            s = fma64(-L[k][i], x[k], s)
        x[i] = s / L[i][i]
    return x


def share_equal(x, z):
    """The largest share of x == alpha z, alpha among the quotients x / z and
    their neighbours."""
    T = z.dtype.type
    q, n = np.unique((x / z).astype(T), return_counts=True)
    a = q[np.argsort(-n)[:20]]
    a = np.unique(np.concatenate([a, np.nextafter(a, T(np.inf)), np.nextafter(a, T(-np.inf))]))
    return max(float(np.mean(x == t * z)) for t in a)


def test_fp32_inverse_of_six(B):
    n = 400
    A = blocks(n, 6, 31, np.float32)
    col = np.arange(n) % 6
    b = np.zeros((n, 6))
    b[np.arange(n), col] = 1.0
    g = B.Problem.from_rcs(np.arange(n + 1, dtype=np.int32), np.arange(n, dtype=np.int32), A.astype(np.float64), b,
                           precision=B.BA_FP32, pcg_rel_tol=0.5, pcg_variant=B.BA_PCG_STANDARD)
    info, conv = g.solve_rcs()
    assert conv and info["pcg_iters"] == 1
    x = g.step()[0].reshape(n, 6).astype(np.float32)
    g.close()
    assert share_equal(x, inverse32(A)[np.arange(n), :, col]) >= 0.999


@pytest.mark.parametrize("c", [6, 11])
def test_fp64_inverse_of_variable_size(B, c):
    n = 60
    A = blocks(n, c, 32 + c, np.float64)
    col = np.arange(n) % c
    b = np.zeros((n, c))
    b[np.arange(n), col] = 1.0
    g = B.VBSMC(np.full(n, c, np.int32), np.arange(n + 1, dtype=np.int32), np.arange(n, dtype=np.int32), A.reshape(-1),
                b.reshape(-1), precision=B.BA_FP64)
    x, its = g.solve(0.5)[:2]
    g.close()
    assert its == 1
    assert share_equal(np.asarray(x).reshape(n, c), np.array([column64(A[i], col[i]) for i in range(n)])) >= 0.999
