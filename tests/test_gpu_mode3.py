"""The FFMA mode-3 pass at its edges against FP64: every outputs-a-warp form
(n3 up to 8, 16, 32, 64), slots that are not full, pixel counts around its
blocks of 128 (and more blocks than the persistent grid), whole groups of four
and ragged ones, prev and the norm; the TF32 operand stored K-major through
whole products.

Tolerance: each output is a chain of n3 FP32 FMAs, relative Frobenius error at
most about sqrt(n3) 2^-24 times |T| |x| / |T x|; on random data that ratio is
below 2, so 1e-6 bounds n3 <= 64 with room. The norm sums positive FP32 squares
in a two-level tree: 1e-6 relative. A TF32 product rounds both operands to 11
bits: 2^-11 sqrt(2) a term at most, random over K: 1e-3 relative."""
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


def matrices(n3):
    from oracle import cproduct as cp
    M = torch.from_numpy(cp.transform_matrix(n3)).cuda()
    Mi = torch.from_numpy(__import__("numpy").linalg.inv(cp.transform_matrix(n3))).cuda()
    return [M, Mi, Mi.mT.contiguous(), M.mT.contiguous()]


@pytest.mark.parametrize("n3,P", [(5, 128), (8, 131), (9, 129), (16, 4096 * 64), (17, 4), (31, 1000),
                                  (32, 127), (33, 128 * 700), (48, 516), (63, 257), (64, 128 * 1300)])
def test_ffma_pass(tc, n3, P):
    g = torch.Generator(device="cuda")
    g.manual_seed(n3 * 1000 + P)
    A = torch.randn((n3, P, 1), generator=g, device="cuda")
    plan = tc.Plan(A, s=1)
    X = torch.randn((n3, P), generator=g, device="cuda")
    prev = torch.randn((n3, P), generator=g, device="cuda")
    ss = torch.zeros(1, dtype=torch.float64, device="cuda")
    for which, T in enumerate(matrices(n3)):
        Y = torch.full_like(X, float("nan"))
        tc.tc_transform(plan.handle, which, X, Y, prev=prev, sumsq=ss)
        want = T @ X.double()
        assert float((Y.double() - prev.double() - want).norm() / want.norm()) < 1e-6
        assert abs(float(ss) / float(Y.double().pow(2).sum()) - 1) < 1e-6
        tc.tc_transform(plan.handle, which, X, Y)
        assert float((Y.double() - want).norm() / want.norm()) < 1e-6
    plan.close()


@pytest.mark.parametrize("n1,n2,s,n3", [(8, 8, 8, 3), (24, 40, 24, 32), (136, 120, 104, 17), (64, 72, 16, 9)])
def test_tf32_operand_k_major(tc, n1, n2, s, n3):
    g = torch.Generator(device="cuda")
    g.manual_seed(n1 + n3)
    A = torch.randn((n3, n1, n2), generator=g, device="cuda")
    X = torch.randn((n3, n2, s), generator=g, device="cuda")
    Y = torch.randn((n3, n1, s), generator=g, device="cuda")
    M, Mi, MiT, MT = matrices(n3)
    m3 = lambda T, Z: (T @ Z.reshape(n3, -1)).reshape(Z.shape)
    plan = tc.Plan(A, s=s, precision=tc.TC_TF32)
    Ah = m3(M, A.double())
    for got, want in ((plan.cprod(X), m3(Mi, torch.bmm(Ah, m3(M, X.double())))),
                      (plan.adjoint(Y), m3(MT, torch.bmm(Ah.mT, m3(MiT, Y.double()))))):
        assert float((got.double() - want).norm() / want.norm()) < 1e-3
    plan.close()
