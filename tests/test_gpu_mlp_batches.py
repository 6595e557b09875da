"""The network's training passes at the edges of their chunks: batches of one,
around four samples a CTA and 128 samples a chunk, and the largest, against FP64
autograd with the BF16-rounded weights; and a training run that wraps around a
data set whose size the batch does not divide.

Tolerance: a gradient is a chain of at most 1024 FP32 FMAs over activations of
relative error near 64 * 2^-24; relative error at most sqrt(1024) 2^-24 + 4e-6
< 1e-5, and 1e-4 (the existing gradient test's bound) leaves room for
cancellation in single entries."""
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


def reference(theta, X, T):
    ws, o = [], 0
    for a, b in ((36, 64), (64, 64), (64, 2)):
        ws.append(theta[o:o + a * b].to(torch.bfloat16).double().reshape(a, b).requires_grad_())
        ws.append(theta[o + a * b:o + a * b + b].double().clone().requires_grad_())
        o += a * b + b
    h = torch.nn.functional.gelu(X.double() @ ws[0] + ws[1])
    h = torch.nn.functional.gelu(h @ ws[2] + ws[3])
    out = h @ ws[4] + ws[5]
    loss = 0.5 * ((out - T.double()) ** 2).sum() / X.shape[0]
    return out.detach(), loss.detach(), torch.cat([g.reshape(-1) for g in torch.autograd.grad(loss, ws)])


@pytest.mark.parametrize("B", [1, 3, 4, 127, 128, 129, 257, 1024])
def test_forward_loss_and_gradient(tc, B):
    g = torch.Generator(device="cuda")
    g.manual_seed(B)
    X = torch.randn((B + 1, 36), generator=g, device="cuda")[1:]  # starts off a 16-byte row
    T = torch.randn((B, 2), generator=g, device="cuda")
    mlp = tc.Mlp(seed=3)
    theta, _ = mlp.get_params()
    theta += 0.05 * torch.randn(theta.shape, generator=g, device="cuda")
    mlp.set_params(theta=theta)
    out, loss, grad = reference(theta, X, T)
    assert float((mlp.forward(X).double() - out).norm() / out.norm()) < 1e-4
    l, gr = mlp.loss_grad(X, T)
    assert abs(float(l) - float(loss)) < 1e-5 * float(loss)
    assert float((gr.double() - grad).norm() / grad.norm()) < 1e-4
    mlp.close()


def test_training_steps_equal_gradient_and_adam_by_hand(tc):
    """Seven steps over 300 samples in batches of 128 (128, 128, 44, 128, ..): the
    loss history is the loss of each batch at the parameters of that step."""
    g = torch.Generator(device="cuda")
    g.manual_seed(0)
    X = torch.randn((300, 36), generator=g, device="cuda")
    T = torch.randn((300, 2), generator=g, device="cuda")
    a, b = tc.Mlp(seed=5), tc.Mlp(seed=5)
    hist = a.train(X, T, 128, 7, 1e-2)
    off = 0
    for s in range(7):
        n = min(128, 300 - off)
        one = b.train(X[off:off + n], T[off:off + n], 128, 1, 1e-2)
        assert torch.equal(one[0], hist[s])
        off = 0 if off + n >= 300 else off + n
    assert torch.equal(a.get_params()[0], b.get_params()[0])
    a.close()
    b.close()
