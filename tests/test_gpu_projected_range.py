"""The projected solve (tc_tikhonov_gcv) on matrices whose columns are graded,
equal, zero or far from one in scale, at a given lambda, against rational
arithmetic on the same doubles.

Tolerance: one-sided Jacobi in FP64 finds the singular values and the first row of
V to a few k eps relative to the columns' own scales, so that GCV is good to about
1e-13 here and y, by Cholesky of matrices of condition below 1e2 after scaling, to
about 1e-13; 1e-9 is the existing tests' bound on y."""
from fractions import Fraction

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tc():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2103_11847_gb300 import tcprod
    tcprod.lib()
    return tcprod


def solve(A, b):
    """A x = b by elimination with pivots, rational."""
    n = len(A)
    M = [list(r) + [v] for r, v in zip(A, b)]
    for i in range(n):
        p = max(range(i, n), key=lambda r: abs(M[r][i]))
        M[i], M[p] = M[p], M[i]
        for r in range(n):
            if r != i and M[r][i] != 0:
                f = M[r][i] / M[i][i]
                M[r] = [x - f * y for x, y in zip(M[r], M[i])]
    return [M[i][n] / M[i][i] for i in range(n)]


def exact(H, beta, lam):
    """The full GCV ||(I - A) b||^2 / trace(I - A)^2, A = H (H^T H + lam^2 I)^-1 H^T,
    b = beta e_1, and y = (H^T H + lam^2 I)^-1 H^T b."""
    rows, k = H.shape
    F = [[Fraction(float(H[i, j])) for j in range(k)] for i in range(rows)]
    l2, b = Fraction(lam) ** 2, Fraction(beta)
    G = [[sum(F[r][i] * F[r][j] for r in range(rows)) + (l2 if i == j else 0) for j in range(k)]
         for i in range(k)]
    y = solve(G, [b * F[0][j] for j in range(k)])
    res = [(b if r == 0 else 0) - sum(F[r][j] * y[j] for j in range(k)) for r in range(rows)]
    tr = Fraction(rows)
    for r in range(rows):
        tr -= sum(x * z for x, z in zip(F[r], solve(G, F[r])))
    return float(sum(v * v for v in res) / (tr * tr)), np.array([float(v) for v in y])


def hessenberg(k, seed, scale):
    rng = np.random.default_rng(seed)
    return np.triu(rng.standard_normal((k + 1, k)), -1) * scale


CASES = {
    # columns far apart in scale, not orthogonal: the small one's rotation is a
    # tangent near 1e-45
    "graded_2": (np.array([[1.0, 1e-45], [1.0, 0.0], [0.0, 0.0]]), 1.0, 1e-3),
    "graded_4": (hessenberg(4, 1, np.array([1.0, 1e-20, 1e-41, 1e-60])), 1.0, 1e-2),
    # columns of equal norm whose dot product is subnormal
    "subnormal_dot": (1e-100 * np.array([[1.0, 1e-109], [1e-109, 1.0], [0.0, 0.0]]), 1e-100, 3e-101),
    # squared norms whose product is near the smallest normal number and below it
    "small_1e-77": (hessenberg(4, 2, 1e-77), 1e-77, 2e-78),
    "small_1e-100": (hessenberg(3, 3, 1e-100), 1e-100, 2e-101),
    "large_1e70": (hessenberg(4, 4, 1e70), 1e70, 2e69),
    "equal_columns": (np.array([[1.0, 1.0], [0.5, 0.5], [0.0, 0.0]]), 1.3, 0.1),
    "zero_column": (np.array([[1.0, 0.0], [0.5, 0.0], [0.0, 0.0]]), 1.3, 0.1),
    "nearly_parallel": (np.array([[1.0, 1.0, 0.3], [1.0, 1.0 + 2.0 ** -30, 0.2], [0.0, 1e-7, 0.1],
                                  [0.0, 0.0, 0.4]]), 1.0, 0.05),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_given_lambda(tc, name):
    H, beta, lam = CASES[name]
    k = H.shape[1]
    gcv, y = exact(H, beta, lam)
    d = lambda v: torch.from_numpy(np.ascontiguousarray(np.atleast_1d(v), dtype=np.float64)).cuda()
    lo, go, yo = d(0.0), d(0.0), d(np.zeros(k))
    tc.tc_tikhonov_gcv(d(H), k, d(beta), tc.TC_GCV_FULL, lam, lo, yo, go)
    torch.cuda.synchronize()
    assert lo.item() == lam
    assert abs(go.item() - gcv) <= 1e-9 * gcv
    assert np.allclose(yo.cpu().numpy(), y, rtol=1e-9, atol=0.0)
