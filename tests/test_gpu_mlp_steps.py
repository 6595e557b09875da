"""The network's forward pass on more samples than its launch has CTAs for, and
several training steps against FP64: gradients by autograd at the BF16-rounded
weights, Adam with its moments and bias corrections carried over.

Tolerances. Forward: 1e-4 as in the existing tests. Training: a gradient is within
1e-4 in norm, so Adam's step, lr m / sqrt(v), is within a few 1e-4 of its length;
parameters that round to the other BF16 neighbour (of 6658, a few per 10^4 and step)
move a gradient by less than that. 5e-3 of the distance moved leaves room for
both; a moment or correction that is wrong or not carried is off by over 0.05."""
import pytest

torch = pytest.importorskip("torch")

from test_gpu_mlp_batches import reference, tc  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B", [4 * 1216 - 1, 4 * 1216, 4 * 1216 + 1, 8 * 1216 + 5, 30011])
def test_forward_many_samples(tc, B):
    g = torch.Generator(device="cuda")
    g.manual_seed(B)
    X = torch.randn((B, 36), generator=g, device="cuda")
    T = torch.zeros((B, 2), device="cuda")
    mlp = tc.Mlp(seed=4)
    theta, _ = mlp.get_params()
    out, _, _ = reference(theta, X, T)
    got = mlp.forward(X).double()
    assert float(((got - out).norm(dim=1) / out.norm(dim=1).mean()).max()) < 1e-4
    mlp.close()


def test_training_steps_against_fp64_adam(tc):
    """Seven steps over 300 samples in batches of 128 (128, 128, 44, 128, ..)."""
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    X = torch.randn((300, 36), generator=g, device="cuda")
    T = torch.randn((300, 2), generator=g, device="cuda")
    mlp = tc.Mlp(seed=6)
    th0, _ = mlp.get_params()
    hist = mlp.train(X, T, 128, 7, 1e-2)
    th, m, v, off = th0.double(), 0.0, 0.0, 0
    for t in range(1, 8):
        n = min(128, 300 - off)
        _, loss, gr = reference(th, X[off:off + n], T[off:off + n])
        assert abs(float(hist[t - 1]) - float(loss)) < 1e-4 * float(loss)
        m, v = 0.9 * m + 0.1 * gr, 0.999 * v + 0.001 * gr * gr
        th = th - 1e-2 * (m / (1 - 0.9 ** t)) / ((v / (1 - 0.999 ** t)).sqrt() + 1e-8)
        off = 0 if off + n >= 300 else off + n
    got = mlp.get_params()[0].double()
    assert float((got - th).norm() / (th - th0.double()).norm()) < 5e-3
    mlp.close()
