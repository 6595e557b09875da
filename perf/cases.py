"""What is measured: the work a user of this library has it do, through its
public entry points.

Kinds of case:
  product   Y = A *c X [*c B] and the adjoint of a second operand: the two
            directions of the operator, one call each (tc_cprod,
            tc_cprod_adjoint), as a user's own iteration calls them.
  lsqr      a whole c-LSQR solve with the Tikhonov/GCV projection (tc_lsqr_c).
  batch     c-LSQR of many independent problems of uneven sizes in one call.
  gmres     restarted DC-GMRES(m) with GCV.
  mlp       training steps of the learned-lambda network from given parameters.

Sizes are the workloads of the benchmark (64x64x3, 256x256x3 two-sided,
512x512x64 video, the batch of 64..512, 512x512x32 of the learned form), the
paper's shapes (256x256x3, 1024x1024x3) and odd ones like those of the tests.
Operators are Gaussian blurs, operands are images in [0, 1], observations
carry Gaussian noise. Iteration counts of the FP32 and batched solves stay where
FP32 still follows the FP64 iteration, so that results can be compared; the GCV
variant is the full one, whose minimum is interior.
"""
import math

import numpy as np
import torch

from paper_2103_11847_gb300 import tcprod as tc

PREC = {"fp32": tc.TC_FP32, "tf32": tc.TC_TF32, "bf16": tc.TC_BF16, "bf16x3": tc.TC_BF16X3}
ELEM = {"fp32": 4, "tf32": 4, "bf16": 2, "bf16x3": 6}  # bytes of an operator element


def listed():
    return [
        # the smallest call: a 64x64 colour image, latency and launches
        dict(name="product_64x64x3_fp32", kind="product", n1=64, n2=64, s=64, n3=3, two=False,
             prec="fp32", store="f32"),
        # rectangular and odd in every dimension: no aligned rows, n3 past the fused form
        dict(name="product_389x301x257x9_fp32", kind="product", n1=389, n2=301, s=257, n3=9,
             two=False, prec="fp32", store="f32"),
        # the paper's first image, blurred on both sides (Tables 1-2): an ordinary call
        dict(name="two_sided_256x256x3_fp32", kind="product", n1=256, n2=256, s=256, n3=3,
             two=True, prec="fp32", store="f32"),
        # the paper's second image (Tables 3-4)
        dict(name="two_sided_1024x1024x3_fp32", kind="product", n1=1024, n2=1024, s=1024, n3=3,
             two=True, prec="fp32", store="f32"),
        # the video operator in the default precision
        dict(name="video_512x512x64_fp32", kind="product", n1=512, n2=512, s=512, n3=64,
             two=False, prec="fp32", store="f32"),
        # the same with FP32-level products on the tensor cores
        dict(name="video_512x512x64_bf16x3", kind="product", n1=512, n2=512, s=512, n3=64,
             two=False, prec="bf16x3", store="f32"),
        # the learned form's second size, in TF32: transforms at n3 = 32
        dict(name="product_512x512x32_tf32", kind="product", n1=512, n2=512, s=512, n3=32,
             two=False, prec="tf32", store="f32"),
        # the benchmark's headline: a whole video solve, BF16 with BF16-stored products
        dict(name="lsqr_video_512x512x64_bf16", kind="lsqr", n=512, n3=64, iters=50, prec="bf16",
             store="bf16"),
        # the batched form, both precisions it groups
        dict(name="batch_128_fp32", kind="batch", count=128, lo=64, hi=512, step=32, iters=12,
             prec="fp32"),
        dict(name="batch_128_bf16", kind="batch", count=128, lo=64, hi=512, step=32, iters=20,
             prec="bf16"),
        # DC-GMRES(10) on the paper's first image
        dict(name="gmres_256x256x3_fp32", kind="gmres", n=256, n3=3, two=True, m=10, iters=10),
        # training the learned-lambda network
        dict(name="mlp_train_256", kind="mlp", rows=4096, batch=256, steps=16),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["product"] * 6 + ["lsqr", "lsqr", "batch", "batch", "gmres", "mlp"])
    if kind == "product":
        two = rng.random() < 0.35
        prec = rng.choice(["fp32", "fp32", "fp32", "tf32", "bf16", "bf16x3"])
        while True:
            if two:
                n3 = rng.choice([1, 2, 3, 3, 3, 4, 7])
                n1, n2, s = (_logint(rng, 32, 1024) for _ in range(3))
            else:
                n3 = rng.choice([3, 3, 3, 4, 9, 32, 64, _logint(rng, 1, 64)])
                n1, n2, s = (_logint(rng, 32, 768) for _ in range(3))
            if prec != "fp32":  # the tensor-core forms take multiples of 8
                n1, n2, s = (max(8, 8 * (v // 8)) for v in (n1, n2, s))
            store = "f32"
            if prec == "bf16" and not two and n3 > 32 and rng.random() < 0.5:
                store = "bf16"
            c = dict(kind=kind, n1=n1, n2=n2, s=s, n3=n3, two=two, prec=prec, store=store)
            if work(c)["flops"] <= 3.0e10 and n1 * n2 * n3 <= 1.6e7:
                return c
    if kind == "lsqr":
        prec = rng.choice(["fp32", "tf32", "bf16", "bf16x3"])
        n3 = rng.choice([3, 3, 9, 32, 40, 64])
        n = _logint(rng, 48, 448)
        if prec != "fp32":
            n = 8 * (n // 8)
        store = "bf16" if prec == "bf16" and n3 > 32 and rng.random() < 0.6 else "f32"
        return dict(kind=kind, n=n, n3=n3, iters=rng.randint(6, 12), prec=prec, store=store)
    if kind == "batch":
        prec = rng.choice(["fp32", "bf16"])
        step = 8 if prec == "bf16" else rng.choice([1, 8, 32])
        return dict(kind=kind, count=_logint(rng, 8, 100), lo=64, hi=rng.choice([128, 256, 448]),
                    step=step, iters=rng.randint(6, 12), prec=prec)
    if kind == "gmres":
        return dict(kind=kind, n=_logint(rng, 48, 400), n3=rng.choice([2, 3, 3, 4]),
                    two=rng.random() < 0.6, m=rng.randint(4, 10), iters=rng.randint(4, 12))
    return dict(kind=kind, rows=_logint(rng, 500, 8192), batch=_logint(rng, 32, 1024),
                steps=rng.randint(4, 16))


# ------------------------------------------------------------------- inputs --

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _uniform(g, n, lo, hi):
    return [lo + (hi - lo) * v for v in torch.rand(n, generator=g, device="cuda",
                                                   dtype=torch.float64).tolist()]


def _blur(rows, cols, sigma):
    """Banded Gaussian Toeplitz factor, half-band ceil(3 sigma), interior rows sum to 1."""
    r = int(math.ceil(3 * sigma))
    d = (torch.arange(rows, device="cuda", dtype=torch.float64)[:, None] * (cols / rows)).round() \
        - torch.arange(cols, device="cuda", dtype=torch.float64)[None, :]
    w = torch.exp(-d * d / (2 * sigma * sigma)) * (d.abs() <= r)
    k = torch.arange(-r, r + 1, device="cuda", dtype=torch.float64)
    return w / torch.exp(-k * k / (2 * sigma * sigma)).sum()


def _image(g, n3, rows, cols):
    """A smooth field a slice with 12 constant rectangles over all slices, in [0, 1]."""
    i = torch.arange(rows, device="cuda", dtype=torch.float64)[:, None] / rows
    j = torch.arange(cols, device="cuda", dtype=torch.float64)[None, :] / cols
    p = torch.rand((n3, 4), generator=g, device="cuda", dtype=torch.float64)
    X = (0.1 + 0.4 * p[:, 0, None, None] + (p[:, 1, None, None] - 0.5) * 0.6 * i
         + (p[:, 2, None, None] - 0.5) * 0.6 * j
         + 0.2 * p[:, 3, None, None] * torch.sin(6.283185307179586 * i)
         * torch.cos(6.283185307179586 * 2 * j))
    u = _uniform(g, 12 * 4, 0.0, 1.0)
    val = torch.rand((12, n3), generator=g, device="cuda", dtype=torch.float64)
    for t in range(12):
        h, w = max(1, int(rows * (0.05 + 0.35 * u[4 * t]))), max(1, int(cols * (0.05 + 0.35 * u[4 * t + 1])))
        a, b = int((rows - h) * u[4 * t + 2]), int((cols - w) * u[4 * t + 3])
        X[:, a:a + h, b:b + w] = val[t, :, None, None]
    return X.clamp(0.0, 1.0)


def _weights(n3):
    if n3 <= 4:
        return [1.0, 0.7, 0.4, 0.2][:n3]
    return [1.0 - 0.6 * k / (n3 - 1) for k in range(n3)]


def _problem(seed, n1, n2, s, n3, two):
    """FP32 A (and B), X, Y of the given sizes, float32 on the GPU."""
    g = _gen(seed)
    sg = _uniform(g, 2, 1.5, 3.5)
    if n3 <= 4:
        blur = _blur(n1, n2, sg[0])
        A = torch.stack([w * blur for w in _weights(n3)])
    else:  # a video: the blur widens over the frames
        A = torch.stack([_blur(n1, n2, 1.5 + (sg[0] - 0.5) * k / (n3 - 1)) for k in range(n3)])
    B = torch.stack([_blur(s, s, sg[1])] * n3) if two else None
    X = _image(g, n3, n2, s)
    Y = _image(g, n3, n1, s) + 0.01 * torch.randn((n3, n1, s), generator=g, device="cuda",
                                                  dtype=torch.float64)
    f = lambda t: None if t is None else t.float().contiguous()
    return f(A), f(B), f(X), f(Y)


def _observe(A, B, X, nu, seed):
    """C = A *c X [*c B] + noise of relative level nu, in FP64, rounded to FP32."""
    C = _op(A.double(), None if B is None else B.double(), X.double())
    N = torch.randn(C.shape, generator=_gen(seed + 7), device="cuda", dtype=torch.float64)
    return (C + nu * C.norm() / N.norm() * N).float().contiguous()


def _batch_inputs(case, seed):
    steps = (case["hi"] - case["lo"]) // case["step"]  # the sizes are the case's, not the seed's
    sizes = [case["lo"] + case["step"] * min(steps, int(v))
             for v in _uniform(_gen(case["count"]), case["count"], 0.0, steps + 1.0)]
    out = []
    for i, n in enumerate(sizes):
        A, _, X, _ = _problem(seed * 131 + i, n, n, n, 3, False)
        nu = 10.0 ** (-4.0 + 2.0 * ((i * 37) % 100) / 100.0)
        out.append((A, _observe(A, None, X, nu, seed * 131 + i)))
    return sizes, out


def _solve_inputs(case, seed):
    n, n3, two = case["n"], case["n3"], case.get("two", False)
    A, B, X, _ = _problem(seed, n, n, n, n3, two)
    return A, B, _observe(A, B, X, 1e-3, seed)


def _mlp_inputs(case, seed):
    g = _gen(seed)
    X = torch.randn((case["rows"], 36), generator=g, device="cuda")
    W = torch.randn((36, 2), generator=g, device="cuda") / 6.0
    T = torch.tanh(X @ W) + 0.05 * torch.randn((case["rows"], 2), generator=g, device="cuda")
    th = []
    for a, b in ((36, 64), (64, 64), (64, 2)):
        th.append((torch.randn((a, b), generator=g, device="cuda") / math.sqrt(a)).reshape(-1))
        th.append(torch.zeros(b, device="cuda"))
    return X.contiguous(), T.contiguous(), torch.cat(th).contiguous()


def prepare(case, seed):
    k = case["kind"]
    if k == "product":
        A, B, X, Y = _problem(seed, case["n1"], case["n2"], case["s"], case["n3"], case["two"])
        plan = tc.Plan(A, B, s=case["s"], precision=PREC[case["prec"]],
                       store=tc.TC_STORE_BF16 if case["store"] == "bf16" else tc.TC_STORE_F32)
        return dict(kind=k, plan=plan, X=X, Y=Y)
    if k == "lsqr":
        A, B, C = _solve_inputs(case, seed)
        plan = tc.Plan(A, B, s=case["n"], precision=PREC[case["prec"]], gcv_variant=tc.TC_GCV_FULL,
                       store=tc.TC_STORE_BF16 if case["store"] == "bf16" else tc.TC_STORE_F32)
        return dict(kind=k, plan=plan, C=C, X=torch.empty_like(C), Xr=torch.empty_like(C),
                    hist=torch.empty(case["iters"], dtype=torch.float64, device="cuda"),
                    info=tc.new_info(), iters=case["iters"])
    if k == "batch":
        sizes, ps = _batch_inputs(case, seed)
        As = [p[0] for p in ps]
        h = _Batch(As, sizes, PREC[case["prec"]])
        Cs = [p[1] for p in ps]
        X, Xs = _arena(Cs)
        Xr, Xrs = _arena(Cs)
        return dict(kind=k, batch=h, Cs=Cs, X=X, Xs=Xs, Xr=Xr, Xrs=Xrs,
                    infos=tc.new_infos(len(Cs)), iters=case["iters"])
    if k == "gmres":
        A, B, C = _solve_inputs(case, seed)
        plan = tc.Plan(A, B, s=case["n"], gcv_variant=tc.TC_GCV_FULL)
        return dict(kind=k, plan=plan, C=C, X=torch.empty_like(C), info=tc.new_info(),
                    m=case["m"], iters=case["iters"])
    X, T, theta = _mlp_inputs(case, seed)
    return dict(kind=k, mlp=tc.Mlp(seed=1), X=X, T=T, theta=theta, batch=case["batch"],
                steps=case["steps"])


def _arena(ts):
    """One zeroed buffer and a view of it for each of ts, 256-byte aligned."""
    offs = [0]
    for t in ts:
        offs.append(offs[-1] + (t.numel() + 63) // 64 * 64)
    flat = torch.zeros(offs[-1], dtype=ts[0].dtype, device="cuda")
    return flat, [flat[o:o + t.numel()].view(t.shape) for o, t in zip(offs, ts)]


class _Batch:
    def __init__(self, As, sizes, precision):
        self.handle = tc.tc_batch_create(As, sizes, precision=precision,
                                         gcv_variant=tc.TC_GCV_FULL)

    def __del__(self):
        try:
            tc.tc_batch_destroy(self.handle)
        except Exception:
            pass


def run(state):
    k = state["kind"]
    if k == "product":
        return state["plan"].cprod(state["X"]), state["plan"].adjoint(state["Y"])
    if k == "lsqr":
        tc.tc_lsqr_c(state["plan"].handle, state["C"], state["X"], state["Xr"], state["iters"], 0.0,
                     None, state["hist"], state["info"])
        return [state["X"], state["Xr"], state["hist"], *_info(state["info"])]
    if k == "batch":
        tc.tc_lsqr_c_batched(state["batch"].handle, state["Cs"], state["Xs"], state["Xrs"],
                             state["iters"], 0.0, None, state["infos"])
        return [state["X"], state["Xr"], *_info(state["infos"].view(len(state["Cs"]), -1))]
    if k == "gmres":
        tc.tc_gmres_c(state["plan"].handle, state["C"], None, state["X"], state["m"],
                      state["iters"], 0.0, None, state["info"])
        return [state["X"], *_info(state["info"])]
    state["mlp"].set_params(theta=state["theta"])
    hist = state["mlp"].train(state["X"], state["T"], state["batch"], state["steps"], 2e-3)
    return state["mlp"].get_params()[0], hist


def _info(buf):
    """The record's whole numbers (iterations, status, cycles, fallback) and its
    computed ones (residual, lambda, GCV, ||C||)."""
    return buf.view(torch.int32)[..., :4], buf.view(torch.float64)[..., 2:6]


# --------------------------------------------------------------------- work --

def work(case):
    """Slice-product flops (dense operators), and bytes: operator and operand in,
    result out for each call; for a solve, every iteration's operator reads
    (forward and adjoint) and the two Krylov vectors read and written."""
    k = case["kind"]
    if k == "product":
        n1, n2, s, n3 = case["n1"], case["n2"], case["s"], case["n3"]
        fl = 2.0 * (2.0 * n1 * n2 * s * n3)
        by = 2.0 * ELEM[case["prec"]] * n1 * n2 * n3 + 2.0 * 4.0 * n3 * s * (n1 + n2)
        if case["two"]:
            fl += 2.0 * s * s * n3 * (n1 + n2)
            by += 2.0 * ELEM[case["prec"]] * s * s * n3
        return dict(bytes=by, flops=fl)
    if k == "mlp":
        per = 2.0 * (36 * 64 + 64 * 64 + 64 * 2) * case["batch"]
        return dict(bytes=case["steps"] * case["batch"] * 38 * 4.0 + 2 * 6658 * 4.0,
                    flops=case["steps"] * 3.0 * per)
    if k == "gmres":
        n, n3 = case["n"], case["n3"]
        per = 2.0 * n ** 3 * n3 * (2 if case["two"] else 1)
        return dict(bytes=4.0 * n * n * n3 * ((2 if case["two"] else 1) + 2), flops=case["iters"] * per)
    if k == "lsqr":
        t = float(case["n"]) ** 2 * case["n3"]
        return dict(bytes=case["iters"] * (2.0 * ELEM[case["prec"]] * t + 4.0 * 4.0 * t) + 12.0 * t,
                    flops=case["iters"] * 4.0 * t * case["n"])
    ns = [case["lo"] + (case["hi"] - case["lo"]) * (i + 0.5) / case["count"] for i in range(case["count"])]
    t2, t3 = sum(3.0 * n ** 2 for n in ns), sum(3.0 * n ** 3 for n in ns)
    return dict(bytes=case["iters"] * (2.0 * ELEM[case["prec"]] + 16.0) * t2 + 12.0 * t2,
                flops=case["iters"] * 4.0 * t3)


# -------------------------------------------------------------------- exact --

def _transform(n):
    """M = W^{-1} C (I + Z) of the cosine product, FP64."""
    i = torch.arange(n, dtype=torch.float64)
    C = torch.cos(math.pi * i[:, None] * (2 * i[None, :] + 1) / (2 * n)) * math.sqrt(2.0 / n)
    C[0] = math.sqrt(1.0 / n)
    IZ = torch.eye(n, dtype=torch.float64) + torch.diag(torch.ones(n - 1, dtype=torch.float64), 1)
    return ((C @ IZ) / C[:, :1]).cuda()


def _inverse(M):
    return torch.from_numpy(np.linalg.inv(M.cpu().numpy())).cuda()


def _m3(T, X):
    return (T @ X.reshape(X.shape[0], -1)).reshape(X.shape)


def _op(A, B, X):
    M = _transform(A.shape[0])
    Z = torch.bmm(_m3(M, A), _m3(M, X))
    if B is not None:
        Z = torch.bmm(Z, _m3(M, B))
    return _m3(_inverse(M), Z)


class _Operator:
    """The operator and its adjoint in FP64, factors transformed once."""

    def __init__(self, A, B):
        self.M = _transform(A.shape[0])
        self.Mi = _inverse(self.M)
        self.A = _m3(self.M, A.double())
        self.B = None if B is None else _m3(self.M, B.double())

    def fwd(self, X):
        Z = torch.bmm(self.A, _m3(self.M, X))
        return _m3(self.Mi, Z if self.B is None else torch.bmm(Z, self.B))

    def adj(self, Y):
        Z = torch.bmm(self.A.mT, _m3(self.Mi.mT.contiguous(), Y))
        return _m3(self.M.mT.contiguous(), Z if self.B is None else torch.bmm(Z, self.B.mT))


def _projected(H, beta):
    """lambda by the full GCV on three nested 200-point log grids from ||H||_F
    down ten decades, and the Tikhonov solution; NumPy FP64."""
    U, s, _ = np.linalg.svd(H, full_matrices=True)
    g, k = beta * U[0], H.shape[1]

    def gcv(lam):
        d = s ** 2 + lam ** 2
        return (np.sum((lam ** 2 * g[:k] / d) ** 2) + np.sum(g[k:] ** 2)) / (1.0 + np.sum(lam ** 2 / d)) ** 2

    hi = math.log(np.linalg.norm(H))
    lo = hi - 10.0 * math.log(10.0)
    for _ in range(3):
        lams = np.exp(np.linspace(lo, hi, 200))
        vals = np.array([gcv(t) for t in lams])
        b = int(np.argmin(vals))
        lo, hi = math.log(lams[max(b - 1, 0)]), math.log(lams[min(b + 1, 199)])
    y = np.linalg.lstsq(np.vstack([H, lams[b] * np.eye(k)]),
                        np.concatenate([[beta], np.zeros(2 * k)]), rcond=None)[0]
    return float(lams[b]), float(vals[b]), y


def _combine(V, y):
    out = torch.zeros_like(V[0])
    for v, c in zip(V, y):
        out += float(c) * v
    return out


def _doubles(*v):
    return torch.tensor(v, dtype=torch.float64)


def _lsqr_exact(A, C, iters):
    op, C = _Operator(A, None), C.double()
    beta = [float(C.norm())]
    U = C / beta[0]
    V = [op.adj(U)]
    alpha = [float(V[0].norm())]
    V[0] /= alpha[0]
    for j in range(iters):
        U = op.fwd(V[j]) - alpha[j] * U
        beta.append(float(U.norm()))
        U /= beta[-1]
        W = op.adj(U) - beta[-1] * V[j]
        alpha.append(float(W.norm()))
        V.append(W / alpha[-1])
    H = np.zeros((iters + 1, iters))
    for j in range(iters):
        H[j, j], H[j + 1, j] = alpha[j], beta[j + 1]
    hist, rb, pb = [], alpha[0], beta[0]
    for j in range(iters):
        rho = math.hypot(rb, beta[j + 1])
        pb, rb = pb * beta[j + 1] / rho, rb / rho * alpha[j + 1]
        hist.append(pb)
    y0 = np.linalg.lstsq(H, np.concatenate([[beta[0]], np.zeros(iters)]), rcond=None)[0]
    lam, gv, y = _projected(H, beta[0])
    V = V[:iters]
    return (_combine(V, y0), _combine(V, y), _doubles(*hist), None,
            _doubles(hist[-1], lam, gv, beta[0]))


def _gmres_exact(A, B, C, m, iters):
    op, C = _Operator(A, B), C.double()
    X, done, beta1 = torch.zeros_like(C), 0, float(C.norm())
    while done < iters:
        R = C - op.fwd(X)
        beta, mj = float(R.norm()), min(m, iters - done)
        V, H = [R / beta], np.zeros((mj + 1, mj))
        for j in range(mj):
            W = op.fwd(V[j])
            for i in range(j + 1):
                H[i, j] = float((V[i] * W).sum())
                W = W - H[i, j] * V[i]
            H[j + 1, j] = float(W.norm())
            V.append(W / H[j + 1, j])
        lam, gv, y = _projected(H, beta)
        X = X + _combine(V[:mj], y)
        done += mj
    return [X, None, _doubles(float((C - op.fwd(X)).norm()), lam, gv, beta1)]


def _mlp_exact(case, X, T, theta):
    X, T, th = X.double(), T.double(), theta.double()
    m, v, off, losses = torch.zeros_like(th), torch.zeros_like(th), 0, []
    for t in range(1, case["steps"] + 1):
        n = min(case["batch"], case["rows"] - off)
        x, y = X[off:off + n], T[off:off + n]
        off = 0 if off + n >= case["rows"] else off + n
        ws, o = [], 0
        for a, b in ((36, 64), (64, 64), (64, 2)):  # the pass reads BF16 copies of the weights
            ws.append(th[o:o + a * b].to(torch.bfloat16).double().reshape(a, b).requires_grad_())
            ws.append(th[o + a * b:o + a * b + b].clone().requires_grad_())
            o += a * b + b
        h = torch.nn.functional.gelu(x @ ws[0] + ws[1])
        h = torch.nn.functional.gelu(h @ ws[2] + ws[3])
        loss = 0.5 * ((h @ ws[4] + ws[5] - y) ** 2).sum() / n
        g = torch.cat([w.reshape(-1) for w in torch.autograd.grad(loss, ws)])
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        th = th - 2e-3 * (m / (1 - 0.9 ** t)) / ((v / (1 - 0.999 ** t)).sqrt() + 1e-8)
        losses.append(loss.detach())
    return th, torch.stack(losses)


def exact(case, seed):
    k = case["kind"]
    if k == "product":
        A, B, X, Y = _problem(seed, case["n1"], case["n2"], case["s"], case["n3"], case["two"])
        op = _Operator(A, B)
        return op.fwd(X.double()), op.adj(Y.double())
    if k == "lsqr":
        A, _, C = _solve_inputs(case, seed)
        return list(_lsqr_exact(A, C, case["iters"]))
    if k == "batch":
        _, ps = _batch_inputs(case, seed)
        rs = [_lsqr_exact(A, C, case["iters"]) for A, C in ps]
        flats = []
        for i in (0, 1):
            flat, views = _arena([r[i] for r in rs])
            for v, r in zip(views, rs):
                v.copy_(r[i])
            flats.append(flat)
        return [*flats, None, torch.stack([r[4] for r in rs])]
    if k == "gmres":
        A, B, C = _solve_inputs(case, seed)
        return _gmres_exact(A, B, C, case["m"], case["iters"])
    X, T, theta = _mlp_inputs(case, seed)
    return _mlp_exact(case, X, T, theta)
