"""GMRES's Arnoldi step in one cluster against its separate launches' sizes, and the
projected solve over its column-pair groupings, against FP64.

Tolerances: an Arnoldi step orthogonalises in FP32 with FP64 coefficients of
FP32 sums: the iterate after m steps on a well-conditioned operator is within
about m 2^-23 of FP64's, 1e-4 as in the existing GMRES parity test. The
projected solve is FP64: the existing test's bounds."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import krylov as kr
from oracle import regularize as rg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tc():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2103_11847_gb300 import tcprod
    tcprod.lib()
    return tcprod


# n s n3 elements: fewer than one CTA of the cluster's, not a multiple of anything,
# 17 / 33 / 49 virtual CTAs (the next CTA count), the largest that fits the
# cluster and the first that does not
@pytest.mark.parametrize("n,s,n3", [(5, 7, 1), (33, 17, 3), (130, 170, 3), (205, 211, 3),
                                    (250, 269, 3), (256, 256, 4), (257, 255, 4), (260, 256, 4)])
def test_gmres_sizes(tc, n, s, n3):
    from oracle import cproduct as cp
    rng = np.random.default_rng(n + s)
    A = rng.standard_normal((n3, n, n)) * (0.2 / np.sqrt(n))
    A[0] += 2 * np.eye(n)
    A = A.astype(np.float32)
    C = rng.standard_normal((n3, n, s)).astype(np.float32)
    Ad = A.astype(np.float64)
    ref = kr.gmres(lambda X: cp.cprod(Ad, X), C.astype(np.float64), np.zeros((n3, n, s)), m=4,
                   itermax=6, lam=0.05)
    plan = tc.Plan(torch.from_numpy(A).cuda(), s=s)
    X, info = plan.gmres(torch.from_numpy(C).cuda(), 4, 6, lam=0.05)
    inf = tc.read_info(info)
    assert inf["iters"] == 6 and inf["cycles"] == 2
    assert np.linalg.norm(X.cpu().numpy() - ref["X"]) < 1e-4 * np.linalg.norm(ref["X"])
    plan.close()


def test_gmres_exact_breakdown(tc):
    """A = 2 I on a constant C whose norm is a power of two: V_1, h_11 = 2 and W -
    h_11 V_1 = 0 are exact, so the cycle stops after one step with X = C / 2."""
    n = 64
    A = 2.0 * torch.eye(n, device="cuda").reshape(1, n, n).contiguous()
    C = torch.ones((1, n, n), device="cuda")
    plan = tc.Plan(A, s=n)
    X, info = plan.gmres(C, 4, 4, lam=0.0)
    inf = tc.read_info(info)
    assert inf["iters"] == 1 and inf["resid"] < 1e-5
    assert float((X - 0.5 * C).abs().max()) < 1e-6
    plan.close()


@pytest.mark.parametrize("k", [2, 3, 8, 15, 16, 31, 32, 33, 127, 128])
@pytest.mark.parametrize("scale", [1.0, 1e-60, 1e60])
def test_projected_solve_groupings(tc, k, scale):
    """Bidiagonal projections (as in the existing test) at the edges of the lane
    groups, H and beta scaled far from one: the printed GCV scales with beta^2,
    lambda with H, y not at all; and y at a fixed lambda."""
    rng = np.random.default_rng(k)
    alpha = np.abs(rng.standard_normal(k + 1)) + 0.05
    beta = np.abs(rng.standard_normal(k + 1)) * np.logspace(0, -3, k + 1)
    H = kr.bidiagonal(alpha, beta, k)
    _, _, g_ref = rg.tikhonov_gcv(H, 1.3, "paper")
    _, y_fix, _ = rg.tikhonov_gcv(H, 1.3, "paper", lam=0.3)
    d = lambda v: torch.from_numpy(np.ascontiguousarray(np.atleast_1d(v), dtype=np.float64)).cuda()
    lo, go, y = d(0.0), d(0.0), d(np.zeros(k))
    tc.tc_tikhonov_gcv(d(H * scale), k, d(1.3 * scale), 0, None, lo, y, go)
    torch.cuda.synchronize()
    assert abs(go.item() / scale ** 2 - g_ref) <= 1e-8 * abs(g_ref)
    lam = lo.item() / scale
    _, y_ref, _ = rg.tikhonov_gcv(H, 1.3, "paper", lam=lam)
    assert np.allclose(y.cpu().numpy(), y_ref, rtol=1e-6, atol=1e-9 * np.abs(y_ref).max())
    tc.tc_tikhonov_gcv(d(H * scale), k, d(1.3 * scale), 0, 0.3 * scale, lo, y, go)
    torch.cuda.synchronize()
    assert np.allclose(y.cpu().numpy(), y_fix, rtol=1e-9, atol=1e-9 * np.abs(y_fix).max())
