"""The grouped BF16 products with many tiles a CTA: batches with several times as
many tiles as SMs, long and short contractions, ragged against both tile shapes.
The two shapes give the same bits (the norms are reduced over blocks that do not
follow the tile), and results agree with single solves to the grouped form's
bound (2e-3 of BF16 products whose transforms are rounded at other points)."""
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


@pytest.mark.parametrize("count,n1,n2,s,n3", [(1, 8, 8, 8, 3), (24, 512, 64, 520, 3), (40, 136, 200, 264, 2),
                                              (30, 264, 72, 328, 4), (300, 64, 72, 40, 1)])
def test_tiles_beyond_the_grid(tc, count, n1, n2, s, n3):
    g = torch.Generator(device="cuda")
    g.manual_seed(count + n1)
    shapes = [(n1 + 8 * (i % 5), n2 + 8 * (i % 3), s - 8 * (i % 2) if s > 8 else s) for i in range(count)]
    As = [torch.randn((n3, a, b), generator=g, device="cuda") for a, b, _ in shapes]
    Cs = [torch.randn((n3, a, c), generator=g, device="cuda") for a, _, c in shapes]
    h = tc.tc_batch_create(As, [c for _, _, c in shapes], precision=tc.TC_BF16)
    res = []
    for tile in (0, 1):
        X = [torch.full((n3, b, c), float("nan"), device="cuda") for _, b, c in shapes]
        Xr = [torch.empty_like(x) for x in X]
        infos = tc.new_infos(count)
        tc.tc_batch_force_tile(h, tile)
        tc.tc_lsqr_c_batched(h, Cs, X, Xr, 3, 0.0, None, infos)
        torch.cuda.synchronize()
        assert tc.tc_batch_info(h)[:2] == (True, tile)
        assert all(i["iters"] == 3 and i["status"] == "maxiter" for i in tc.read_infos(infos, count))
        res.append((X, Xr, infos))
    for a, b in zip(res[0][0] + res[0][1], res[1][0] + res[1][1]):
        assert torch.equal(a, b)
    assert torch.equal(res[0][2], res[1][2])
    for i in range(0, count, max(1, count // 6)):
        plan = tc.Plan(As[i], s=shapes[i][2], precision=tc.TC_BF16)
        want, _, _, _ = plan.lsqr(Cs[i], itermax=3, regularize=True)
        assert float((res[0][0][i] - want).norm() / want.norm()) < 2e-3
        plan.close()
    tc.tc_batch_destroy(h)
