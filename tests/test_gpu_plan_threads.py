"""Plans created by several threads at once, each on a stream of its own: the
kernels' attributes are set once a device before any of them launches."""
import threading

import pytest

torch = pytest.importorskip("torch")

from test_gpu_ffma_tiles import reference, rel, tc  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def test_plans_from_threads(tc):
    out, errors = [None] * 6, []

    def work(i):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                g = torch.Generator(device="cuda")
                g.manual_seed(i)
                n = 448 + 8 * i  # 64 x 64 tiles: shared memory beyond 48 KB
                A = torch.randn((3, n, n), generator=g, device="cuda")
                X = torch.randn((3, n, n), generator=g, device="cuda")
                plan = tc.Plan(A, s=n)
                Y = plan.cprod(X)
                torch.cuda.current_stream().synchronize()
                out[i] = rel(Y, reference(A, None, X, False))
                plan.close()
        except Exception as e:  # reported by the main thread
            errors.append(repr(e))

    ts = [threading.Thread(target=work, args=(i,)) for i in range(len(out))]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not errors, errors
    assert max(out) < 1e-5
