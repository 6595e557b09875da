"""Norms and inner products that the fused FP32 products reduce in their store, in
solves large enough for whole 64 x 64 tiles (152 of them and more), whole groups
of four and ragged, one- and two-sided (there the first product of the pair is
stored transposed), and the same bits from the grouped form's 64 x 64 and 128 x 64
tiles.

Tolerances: a Golub-Kahan step is two products of K <= 840 FP32 FMAs a value and
FP32 sums of 4096 squares a block, reduced in FP64: alpha and beta are within
sqrt(840) 2^-24 = 2e-6 times the transforms' condition (at most 4); 1e-5 as for
the products. Two steps on well separated data carry it to U and V times a small
factor: 1e-4, the existing solver tests' bound."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from test_gpu_ffma_tiles import mode3, rel, tc, transform  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


class Operator:
    def __init__(self, A, B):
        self.M = transform(A.shape[0])
        self.Mi = torch.from_numpy(np.linalg.inv(self.M.cpu().numpy())).cuda()
        self.A = mode3(self.M, A.double())
        self.B = None if B is None else mode3(self.M, B.double())

    def fwd(self, X):
        Z = torch.bmm(self.A, mode3(self.M, X))
        return mode3(self.Mi, Z if self.B is None else torch.bmm(Z, self.B))

    def adj(self, Y):
        Z = torch.bmm(self.A.mT, mode3(self.Mi.mT.contiguous(), Y))
        return mode3(self.M.mT.contiguous(), Z if self.B is None else torch.bmm(Z, self.B.mT))


def problem(n1, n2, s, n3, two, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    rand = lambda *sh: torch.randn(sh, generator=g, device="cuda")
    A = rand(n3, n1, n2) / n2 ** 0.5
    B = rand(n3, s, s) / s ** 0.5 if two else None
    return A, B, rand(n3, n1, s)


SHAPES = [(832, 832, 832, 3, False), (837, 835, 831, 3, False), (840, 200, 900, 4, False), (834, 40, 835, 1, False),
          (832, 832, 832, 2, True), (835, 833, 837, 3, True)]


@pytest.mark.parametrize("n1,n2,s,n3,two", SHAPES)
def test_golub_kahan_steps(tc, n1, n2, s, n3, two):
    A, B, C = problem(n1, n2, s, n3, two, n1 + n2)
    op, plan = Operator(A, B), tc.Plan(A, B, s=s)
    U, V = torch.empty((3, n3, n1, s), device="cuda"), torch.empty((3, n3, n2, s), device="cuda")
    al, be = (torch.zeros(3, dtype=torch.float64, device="cuda") for _ in range(2))
    tc.tc_gkb_init(plan.handle, C, U, V, al, be, 2)
    for j in (1, 2):
        tc.tc_gkb_step(plan.handle, j, U, V, al, be, 2)
    u = C.double()
    b = [float(u.norm())]
    u = u / b[0]
    v = op.adj(u)
    a = [float(v.norm())]
    v = v / a[0]
    for _ in range(2):
        w = op.fwd(v) - a[-1] * u
        b.append(float(w.norm()))
        u = w / b[-1]
        w = op.adj(u) - b[-1] * v
        a.append(float(w.norm()))
        v = w / a[-1]
    for got, want in ((al, a), (be, b)):
        assert np.allclose(got.cpu().numpy(), want, rtol=1e-5, atol=0)
    assert rel(U[2], u) < 1e-4 and rel(V[2], v) < 1e-4
    plan.close()


@pytest.mark.parametrize("n,s,two", [(832, 832, False), (833, 835, False), (832, 832, True)])
def test_gmres_inner_product_in_the_store(tc, n, s, two):
    """DC-GMRES steps: h_1j = <V_1, W> comes from the product's store."""
    from oracle import krylov as kr
    A, B, C = problem(n, n, s, 3, two, n + s)
    A = (0.2 * A).contiguous()
    A[0] += 2 * torch.eye(n, device="cuda")
    if two:
        B = (0.2 * B).contiguous()
        B[0] += 2 * torch.eye(s, device="cuda")
    op, plan = Operator(A, B), tc.Plan(A, B, s=s)
    fwd = lambda X: op.fwd(torch.from_numpy(X).cuda()).cpu().numpy()
    ref = kr.gmres(fwd, C.double().cpu().numpy(), np.zeros((3, n, s)), m=3, itermax=4, lam=0.05)
    X, info = plan.gmres(C, 3, 4, lam=0.05)
    assert tc.read_info(info)["iters"] == 4
    assert np.linalg.norm(X.cpu().numpy() - ref["X"]) < 1e-4 * np.linalg.norm(ref["X"])
    plan.close()


@pytest.mark.parametrize("n3", [1, 3, 4])
def test_grouped_64_and_128_row_tiles_to_the_bit(tc, n3):
    sizes = [33, 64, 65, 128, 129, 200]
    g = torch.Generator(device="cuda")
    g.manual_seed(n3)
    As = [torch.randn((n3, n, n + 1), generator=g, device="cuda") for n in sizes]
    Cs = [torch.randn((n3, n, n + 3), generator=g, device="cuda") for n in sizes]
    h = tc.tc_batch_create(As, [n + 3 for n in sizes])
    res = []
    for tile in (0, 2):
        X, Xr = ([torch.empty((n3, n + 1, n + 3), device="cuda") for n in sizes] for _ in range(2))
        infos = tc.new_infos(len(sizes))
        tc.tc_batch_force_tile(h, tile)
        tc.tc_lsqr_c_batched(h, Cs, X, Xr, 5, 0.0, None, infos)
        torch.cuda.synchronize()
        res.append((X + Xr, infos))
    for a, b in zip(res[0][0], res[1][0]):
        assert torch.equal(a, b)
    assert torch.equal(res[0][1], res[1][1])
    tc.tc_batch_destroy(h)
