"""The FFMA mode-3 pass with prev and the norm where its CTAs have one block each
(prev read ahead of the FMAs up to n3 = 16), at the last such size and past it,
against FP64. Tolerance: at most 16 FP32 FMAs and one addition an output, 1e-6 as in
the pass's other tests; the norm's partials are FP32 sums over 128 pixels, 1e-6."""
import pytest

torch = pytest.importorskip("torch")

from test_gpu_mode3 import matrices, tc  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n3", [1, 3, 8, 9, 12, 16])
@pytest.mark.parametrize("P", [4, 128 * 152, 128 * 912, 128 * 912 + 4, 128 * 1216, 128 * 1216 + 128, 20739])
def test_prev_and_norm(tc, n3, P):
    g = torch.Generator(device="cuda")
    g.manual_seed(n3 * 100003 + P)
    plan = tc.Plan(torch.randn((n3, P, 1), generator=g, device="cuda"), s=1)
    X = torch.randn((n3, P), generator=g, device="cuda")
    prev = torch.randn((n3, P), generator=g, device="cuda")
    ss = torch.zeros(1, dtype=torch.float64, device="cuda")
    T = matrices(n3)[0]
    Y = torch.full_like(X, float("nan"))
    tc.tc_transform(plan.handle, tc.TC_M, X, Y, prev=prev, sumsq=ss)
    want = T @ X.double() + prev.double()
    assert float((Y.double() - want).norm() / want.norm()) < 1e-6
    assert abs(float(ss) / float(Y.double().pow(2).sum()) - 1) < 1e-6
    plan.close()
