"""The fused FP32 products: the 32 x 32 tiles with each way of reading their
operands (whole groups of four in both, in the left operand only, in the right
one only, in neither; by their sizes and by where the operands start; K whole and
split), and the 64 x 64 tiles with each split.

The choice follows M = n1 (left, K-major) and N = s (right) for the product and
M = n2 for the adjoint. Tolerance: the FP32 products' 1e-5 bound (K <= 420 FMAs in
one chain are within sqrt(420) 2^-24 = 1.2e-6 relative, K = 832 within 1.8e-6, times the transforms'
condition, at most 4 for n3 <= 4 on random data)."""
import pytest

torch = pytest.importorskip("torch")

from test_gpu_ffma_tiles import reference, rel, tc  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


# n1, n2 in (both whole), (only n2 whole), (only n1 whole); s whole and not
@pytest.mark.parametrize("n3", [1, 2, 3, 4])
@pytest.mark.parametrize("n1,n2,s", [(36, 100, 40), (33, 100, 40), (36, 101, 40), (36, 100, 41),
                                     (33, 35, 31), (130, 420, 200), (132, 418, 202), (1, 20, 4), (4, 15, 1)])
def test_products_by_alignment(tc, n1, n2, s, n3):
    g = torch.Generator(device="cuda")
    g.manual_seed(n1 + 3 * n2 + s + n3)
    rand = lambda *sh: torch.randn(sh, generator=g, device="cuda")
    A, X, Y = rand(n3, n1, n2), rand(n3, n2, s), rand(n3, n1, s)
    plan = tc.Plan(A, s=s)
    assert rel(plan.cprod(X), reference(A, None, X, False)) < 1e-5
    assert rel(plan.adjoint(Y), reference(A, None, Y, True)) < 1e-5
    plan.close()


# The product's form by the rule of gemm.cu (64 x 64 tiles whole, and split over
# 2, 4 and 8 ranks), whole groups and ragged; with a right factor both products of
# the pair, the first stored transposed
@pytest.mark.parametrize("n1,n2,s,n3,two", [
    (512, 130, 832, 3, False), (401, 130, 833, 3, False), (512, 520, 832, 3, False), (257, 520, 833, 3, False),
    (448, 448, 448, 1, False), (257, 521, 259, 3, False), (256, 520, 832, 4, False), (256, 520, 641, 2, False),
    (448, 448, 448, 3, True), (451, 449, 450, 4, True), (256, 520, 832, 2, True), (300, 520, 521, 1, True)])
def test_products_by_form(tc, n1, n2, s, n3, two):
    g = torch.Generator(device="cuda")
    g.manual_seed(n1 + 3 * n2 + s + n3)
    rand = lambda *sh: torch.randn(sh, generator=g, device="cuda")
    A, B = rand(n3, n1, n2), rand(n3, s, s) if two else None
    X, Y = rand(n3, n2, s), rand(n3, n1, s)
    plan = tc.Plan(A, B, s=s)
    assert rel(plan.cprod(X), reference(A, B, X, False)) < 1e-5
    assert rel(plan.adjoint(Y), reference(A, B, Y, True)) < 1e-5
    plan.close()


def test_operand_off_alignment_gives_the_same_bits(tc):
    """An operand one float past an aligned address is read value by value: the
    same chain of FMAs."""
    n3, n1, n2, s = 4, 64, 132, 48
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    A = torch.randn((n3, n1, n2), generator=g, device="cuda")
    X = torch.randn((n3, n2, s), generator=g, device="cuda")
    plan = tc.Plan(A, s=s)
    buf = torch.zeros(X.numel() + 1, device="cuda")
    Xo = buf[1:].view(X.shape)
    Xo.copy_(X)
    assert torch.equal(plan.cprod(Xo), plan.cprod(X))
    plan.close()


@pytest.mark.parametrize("n1,n2,s", [(36, 40, 44), (33, 40, 44), (36, 40, 43), (33, 35, 31)])
def test_grouped_small_tiles_by_alignment(tc, n1, n2, s):
    """The grouped form's 32 x 32 tiles, three problems of one size: three steps
    agree with a single solve to the grouped tests' 1e-5."""
    g = torch.Generator(device="cuda")
    g.manual_seed(n1 + s)
    rand = lambda *sh: torch.randn(sh, generator=g, device="cuda")
    As, Cs = [rand(3, n1, n2) for _ in range(3)], [rand(3, n1, s) for _ in range(3)]
    Xs, Xr = ([torch.empty((3, n2, s), device="cuda") for _ in range(3)] for _ in range(2))
    h = tc.tc_batch_create(As, [s] * 3)
    tc.tc_batch_force_tile(h, 1)
    tc.tc_lsqr_c_batched(h, Cs, Xs, Xr, 3, 0.0, None, tc.new_infos(3))
    for A, C, X in zip(As, Cs, Xs):
        plan = tc.Plan(A, s=s)
        want = plan.lsqr(C, itermax=3, regularize=True)[0]
        assert rel(X, want.double()) < 1e-5
        plan.close()
    tc.tc_batch_destroy(h)
