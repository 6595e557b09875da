"""The FP32 products at the edges of their tiles and of the rules that choose
them, against FP64 on the same FP32 inputs.

Tolerance: an output is a sum of K products of FP32 values taken through two
n3 x n3 transforms. With every addition rounded (unit roundoff 2^-24) the
relative Frobenius error of a sum of K random terms is near sqrt(K) 2^-24, at
most 2e-6 for K <= 1100, times the transforms' condition (at most 4 for n3 <=
5 on random data): below the products' bound of 1e-5, which is used here as
everywhere for FP32."""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu
TOL = 1e-5


@pytest.fixture(scope="module")
def tc():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2103_11847_gb300 import tcprod
    tcprod.lib()
    return tcprod


def rel(a, b):
    return float((a.double() - b).norm() / b.norm())


def transform(n3):
    from oracle import cproduct as cp
    return torch.from_numpy(cp.transform_matrix(n3)).cuda()


def mode3(T, X):
    return (T @ X.reshape(X.shape[0], -1)).reshape(X.shape)


def reference(A, B, X, adjoint):
    M = transform(A.shape[0])
    Mi = torch.from_numpy(__import__("numpy").linalg.inv(M.cpu().numpy())).cuda()
    At, pro, epi = mode3(M, A.double()), M, Mi
    Bt = None if B is None else mode3(M, B.double())
    if adjoint:
        At, pro, epi = At.mT, Mi.mT.contiguous(), M.mT.contiguous()
        Bt = None if Bt is None else Bt.mT
    Z = torch.bmm(At, mode3(pro, X.double()))
    return mode3(epi, Z if Bt is None else torch.bmm(Z, Bt))


# n1, n2, s, n3, two_sided: fused 64 x 64 tiles split over 8, 4, 2 ranks and
# whole (with K too short for a split), whole groups of four and ragged rows,
# n3 = 1 .. 4; two-sided past s = 256, whose first product is stored
# transposed; per-slice tiles of each shape, ragged in every dimension
SHAPES = [
    (448, 448, 448, 3, False), (321, 270, 325, 3, False), (512, 100, 520, 1, False),
    (640, 33, 512, 4, False), (768, 20, 770, 2, False), (833, 64, 832, 3, False),
    (1024, 513, 1000, 3, False),
    (260, 300, 272, 3, True), (259, 70, 301, 4, True), (64, 40, 1028, 2, True),
    (389, 301, 257, 9, False), (512, 128, 512, 20, False), (130, 64, 66, 40, False),
    (70, 65, 31, 5, True), (256, 36, 260, 6, True),
]


@pytest.mark.parametrize("n1,n2,s,n3,two", SHAPES)
def test_products_at_tile_edges(tc, n1, n2, s, n3, two):
    g = torch.Generator(device="cuda")
    g.manual_seed(n1 + 7 * n2 + s + n3)
    rand = lambda *sh: torch.randn(sh, generator=g, device="cuda")
    A, B = rand(n3, n1, n2), rand(n3, s, s) if two else None
    X, Y = rand(n3, n2, s), rand(n3, n1, s)
    plan = tc.Plan(A, B, s=s)
    assert rel(plan.cprod(X), reference(A, B, X, False)) < TOL
    assert rel(plan.adjoint(Y), reference(A, B, Y, True)) < TOL
    plan.close()


@pytest.mark.parametrize("offset", [1, 4])
def test_products_of_operands_off_alignment(tc, offset):
    """Operands and results that start `offset` floats past an aligned address:
    the same bits as the aligned call (each output is one chain of FMAs in K order)."""
    n, n3 = 384, 3
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    A = torch.randn((n3, n, n), generator=g, device="cuda")
    X = torch.randn((n3, n, n), generator=g, device="cuda")
    plan = tc.Plan(A, s=n)
    want = plan.cprod(X)
    buf = torch.zeros(X.numel() + offset, device="cuda")
    Xo = buf[offset:].view(X.shape)
    Xo.copy_(X)
    out = torch.full((X.numel() + offset,), float("nan"), device="cuda")
    got = plan.cprod(Xo, out=out[offset:].view(X.shape))
    assert torch.equal(got, want)
    assert bool(torch.isnan(out[:offset]).all())
    plan.close()


@pytest.mark.parametrize("mode", [2, 3, 4])
def test_grouped_tiles_match_single_solves(tc, mode):
    """Each FP32 tile shape of the grouped form, sizes ragged against all of them:
    three steps, where the orders of addition differ by FP32 rounding alone
    (the grouped tests' 1e-5)."""
    sizes = [33, 64, 70, 129, 200]
    g = torch.Generator(device="cuda")
    g.manual_seed(9)
    As = [torch.randn((3, n, n + 1), generator=g, device="cuda") for n in sizes]
    Cs = [torch.randn((3, n, n + 3), generator=g, device="cuda") for n in sizes]
    new = lambda: [torch.empty((3, n + 1, n + 3), device="cuda") for n in sizes]
    h = tc.tc_batch_create(As, [n + 3 for n in sizes])
    tc.tc_batch_info(h, mode=mode)
    X, Xr, infos = new(), new(), tc.new_infos(len(sizes))
    tc.tc_lsqr_c_batched(h, Cs, X, Xr, 3, 0.0, None, infos)
    torch.cuda.synchronize()
    assert tc.tc_batch_info(h)[1] == mode - 2
    for i, n in enumerate(sizes):
        plan = tc.Plan(As[i], s=n + 3)
        want, _, _, _ = plan.lsqr(Cs[i], itermax=3, regularize=True)
        assert rel(X[i], want.double()) < 1e-5
        plan.close()
    tc.tc_batch_destroy(h)
