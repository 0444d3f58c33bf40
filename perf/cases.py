"""What a user of the FIRLS library has it do, as cases to be timed.

Reconstructions (one slice, a batch, multi-contrast images, tree groups, several
sizes in one call), dense random projections with an own or a shared matrix, the
operator-level calls, and the learned warm start in training and in use.  Sizes
come from the library's own workloads; drawn cases spread over the ranges around
them.  `exact` restates each path in 64 bits with plain torch.
"""
import math

import numpy as np
import torch

import paper_1411_5057_gb300 as F
from paper_1411_5057_gb300 import binding as B

SIZES = (16, 32, 48, 64, 80, 96, 128, 160, 192, 256, 320, 384, 512)
EPS = 1e-10  # the library's default smoothing of the weights
# A solve with both regularisers is smoothed at a tenth of the noise level: with
# the default, single wavelet coefficients of an otherwise settled slice are
# weighted by rounding, and two correct programs part after a few PCG steps.
SMOOTH = 1e-6
CNN = (3, 32, 32, 32, 32, 32, 2)
_stream = None


def stream():
    """The program's one side stream (the library captures its graphs on it)."""
    global _stream
    if _stream is None:
        _stream = torch.cuda.Stream()
    return _stream


# ------------------------------------------------------------------- cases --

def fourier(op, n, batch, wavelet="", levels=0, tv="", outer=2, pcg=60, precond="paper", real=False, channels=1,
            tree=False, ratio=0.2, eps=EPS):
    return dict(op=op, n=n, batch=batch, wavelet=wavelet, levels=levels, tv=tv, outer=outer, pcg=pcg,
                precond=precond, real=real, channels=channels, tree=tree, ratio=ratio, eps=eps)


def listed():
    def named(name, c):
        return dict(c, name=name)

    return [
        # one operator application on one small real image: a user's own
        # iteration around A^H A, where launches and latency count
        named("aha_real_64_b1", fourier("aha", 64, 1, wavelet="haar", levels=3, real=True, ratio=0.25)),
        # weights, S d and P^-1 r of an odd batch at a radix-5 size with the l1
        # form of TV, Haar and the ILU(0) factors: the operators used singly
        named("sp_l1tv_haar_320_b5", fourier("sp", 320, 5, "haar", 3, "l1", precond="ilu0")),
        # the small real l1 workload (64^2 Haar, 20 PCG steps per outer step):
        # many short launches
        named("solve_haar_64_b1", fourier("solve", 64, 1, "haar", 3, outer=3, pcg=20, real=True, ratio=0.25)),
        # one outer step of one 256^2 TV + D4 slice: the latency of a
        # reconstruction, and of the end of a served queue
        named("solve_tv_db4_256_b1", fourier("solve", 256, 1, "db4", 4, "iso", outer=1, pcg=20, eps=SMOOTH)),
        # the same slices at the batch a server runs: throughput
        named("solve_tv_db4_256_b304", fourier("solve", 256, 304, "db4", 4, "iso", outer=1, pcg=20, eps=SMOOTH)),
        # multi-contrast cross sections (joint D4 sparsity)
        named("solve_mt_db4_256_b60", fourier("solve", 256, 60, "db4", 4, outer=2, pcg=10, channels=3, ratio=0.25)),
        # overlapping tree groups at 512^2, the largest image
        named("solve_tree_db4_512_b8", fourier("solve", 512, 8, "db4", 5, outer=2, pcg=20, tree=True, ratio=0.25)),
        # slices of four sizes in one call
        named("multi_tv_db4_b4x4", dict(op="multi", sizes="128,192,256,320", batch=4, levels=4, outer=1, pcg=20)),
        # dense random projections, 4000 unknowns and 800 measurements: a
        # matrix per problem, and one matrix for many signals
        named("dense_own_800x4000_p152", dict(op="dense", M=800, N=4000, problems=152, shared=False, outer=2, pcg=5,
                                              precond="paper")),
        named("dense_shared_800x4000_p256", dict(op="dense", M=800, N=4000, problems=256, shared=True, outer=2,
                                                 pcg=5, precond="paper")),
        # one training step of the warm-start network, and its use on a batch
        # (network, data consistency, guard)
        named("cnn_train_256_b16", dict(op="train", n=256, batch=16, lr=1e-3)),
        named("warm_256_b64", dict(op="warm", n=256, batch=64)),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["aha", "sp", "sp", "solve", "solve", "solve", "solve", "multi", "dense", "dense", "train",
                     "warm"])
    if op == "multi":
        sizes = rng.sample([64, 96, 128, 160, 192, 256, 320], rng.randint(2, 4))
        return dict(op=op, sizes=",".join(map(str, sizes)), batch=_log(rng, 1, 12), levels=rng.randint(2, 4), outer=1,
                    pcg=rng.randint(10, 20))
    if op == "dense":
        shared = rng.random() < 0.5
        N = 4 * _log(rng, 64, 2000)  # a tenth to a half as many measurements
        M = min(1600, _log(rng, N // 10, N // 2))
        P = _log(rng, 1, 400)
        if not shared:  # a matrix per problem: at most the listed case's bytes
            P = max(1, min(P, 152 * 800 * 4000 // (M * N)))
        else:
            P = max(1, min(P, 256 * 800 * 4000 * 2 // (M * N)))
        return dict(op=op, M=M, N=N, problems=P, shared=shared, outer=rng.randint(1, 2), pcg=rng.randint(3, 5),
                    precond=rng.choice(["paper", "paper", "jacobi"]))
    if op in ("train", "warm"):
        n = rng.choice([64, 96, 128, 192, 256, 320, 384])
        most = (16 if op == "train" else 64) * 65536 // (n * n)
        return dict(op=op, n=n, batch=_log(rng, 1, max(1, most)), **({"lr": rng.choice([1e-3, 3e-4])}
                                                                     if op == "train" else {}))
    n = rng.choice(SIZES[2:] if op == "solve" else SIZES)
    batch = _log(rng, 1, max(2, min(1500, 200 * 65536 // (n * n))))
    tv = rng.choice(["", "iso", "iso", "l1"])
    wavelet = rng.choice(["haar", "db4", "db4"] + ([""] if tv else []))
    most = 1
    while most < 5 and n % (1 << (most + 1)) == 0 and n >> most >= 4:
        most += 1
    levels = rng.randint(1, most) if wavelet else 0
    precond = rng.choice(["paper", "paper", "jacobi"] + (["ilu0"] if tv else []))
    tree = bool(wavelet and not tv and levels >= 2 and rng.random() < 0.4)
    channels = 1
    if wavelet and not tree and tv != "l1" and rng.random() < 0.25:
        channels = rng.randint(2, 3)
        batch = max(1, batch // channels) * channels
    real = rng.random() < 0.3 and channels == 1
    pcg = rng.randint(8, 10 if n < 64 else 20)
    eps = SMOOTH if op == "solve" and tv and wavelet else EPS
    return fourier(op, n, batch, wavelet, levels, tv, outer=1 if tv else rng.randint(1, 2), pcg=pcg, precond=precond,
                   real=real, channels=channels, tree=tree, ratio=round(rng.uniform(0.15, 0.35), 3), eps=eps)


# ------------------------------------------------------------------ inputs --

def _gen(seed, k):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 1009 + k)
    return g


def _rand(g, *shape, lo=0.0, hi=1.0):
    return torch.rand(*shape, generator=g, device="cuda", dtype=torch.float64) * (hi - lo) + lo


def phantoms(n, images, channels, real, seed):
    """[images * channels][n][n] ellipse phantoms; the contrasts of an image
    share their ellipses, complex ones carry a smooth phase."""
    g = _gen(seed, 1)
    t = (2.0 * (torch.arange(n, device="cuda", dtype=torch.float64) + 0.5) / n) - 1.0
    v, u = t[:, None], t[None, :]
    x = torch.zeros(images, channels, n, n, dtype=torch.float32, device="cuda")
    for _ in range(10):
        cx, cy = (_rand(g, images, 1, 1, lo=-0.7, hi=0.7) for _ in range(2))
        ax, ay = (_rand(g, images, 1, 1, lo=0.05, hi=0.45) for _ in range(2))
        th = _rand(g, images, 1, 1, hi=math.pi)
        level = _rand(g, images, channels).float()
        du, dv = u - cx, v - cy
        inside = ((torch.cos(th) * du + torch.sin(th) * dv) / ax) ** 2 \
            + ((torch.cos(th) * dv - torch.sin(th) * du) / ay) ** 2 <= 1.0
        x += inside[:, None].float() * level[:, :, None, None]
    x = x.reshape(images * channels, n, n)
    if real:
        return x.to(torch.complex64)
    a = _rand(g, images * channels, 6, 1, 1, lo=-0.5, hi=0.5).float()
    ps = [u ** p * v ** q for p in range(3) for q in range(3 - p)]
    phi = sum(a[:, i] * p.float() for i, p in enumerate(ps)) * math.pi
    return torch.polar(x, phi)


def masks(n, batch, ratio, seed):
    """uint8 [batch][n][n]: variable-density sampling, DC kept."""
    g = _gen(seed, 2)
    k = torch.arange(n, device="cuda", dtype=torch.float64)
    k = torch.where(k >= n // 2, k - n, k)
    r = torch.sqrt(k[:, None] ** 2 + k[None, :] ** 2)
    w = (1.0 - r / r.max()) ** 4 + 0.02
    m = max(1, int(round(ratio * n * n)))
    out = torch.zeros(batch, n * n, dtype=torch.uint8, device="cuda")
    for s in range(0, batch, 64):
        e = min(batch, s + 64)
        keys = torch.log(_rand(g, e - s, n * n, lo=1e-12)) / w.reshape(-1)
        keys[:, 0] = 0.0
        out[s:e].scatter_(1, keys.topk(m, dim=1).indices, 1)
    return out.reshape(batch, n, n)


def measure(x, mask, seed):
    g = _gen(seed, 3)
    noise = torch.view_as_complex(torch.randn(*x.shape, 2, generator=g, device="cuda") * 0.01)
    return (mask * (torch.fft.fft2(x, norm="ortho") + noise)).contiguous()


def tree_map(n, levels):
    """int32 [groups][2]: each detail coefficient with its parent."""
    rows = []
    for l in range(1, levels + 1):
        h = n >> l
        i, j = torch.meshgrid(torch.arange(h), torch.arange(h), indexing="ij")
        for br, bc in ((0, 1), (1, 0), (1, 1)):
            r, c = br * h + i, bc * h + j
            pr, pc = (r // 2, c // 2) if l < levels else (i, j)
            rows.append(torch.stack([(r * n + c).reshape(-1), (pr * n + pc).reshape(-1)], dim=1))
    return torch.cat(rows).to(torch.int32).contiguous().cuda()


def slices(case, seed):
    n, b, C = case["n"], case["batch"], case["channels"]
    x = phantoms(n, b // C, C, case["real"], seed)
    mask = masks(n, b, case["ratio"], seed)
    return x, mask, measure(x, mask, seed)


def lambdas(case):
    if case["tv"] and case["wavelet"]:
        return 5e-4, 1e-3
    return (0.0, 1e-3) if case["tv"] else (1e-3, 0.0)


def psi_of(case):
    w = {"": 0, "haar": B.PSI_HAAR, "db4": B.PSI_DB4}[case["wavelet"]]
    return w | {"": 0, "iso": B.PSI_TV, "l1": B.PSI_TV_ANISO}[case["tv"]]


def context(case, mask):
    ctx = F.Context(case["n"], batch=case["batch"], real=case["real"], stream=stream())
    if case["channels"] > 1:
        ctx.set_channels(case["channels"])
    ctx.set_operator(mask, psi_of(case), case["levels"],
                     groups=tree_map(case["n"], case["levels"]) if case["tree"] else None)
    return ctx


def params(case, outer=None):
    lam, lam_tv = lambdas(case)
    return F.make_params(outer or case["outer"], case["pcg"], lam=lam, lam_tv=lam_tv, precond=case["precond"],
                         eps=case["eps"])


def multi_cases(case):
    return [fourier("solve", int(n), case["batch"], "db4", case["levels"], "iso", case["outer"], case["pcg"],
                    eps=SMOOTH)
            for n in case["sizes"].split(",")]


def sp_inputs(case, x, seed):
    """An iterate near the image, and a direction and a residual as PCG has them."""
    g = _gen(seed, 4)
    n = case["n"]

    def noise(scale):
        v = torch.view_as_complex(torch.randn(case["batch"], n, n, 2, generator=g, device="cuda") * scale)
        return v.real.to(torch.complex64) if case["real"] else v

    return (x + noise(0.02)).contiguous(), noise(0.1).contiguous(), noise(0.05).contiguous()


def dense_inputs(case, seed):
    g = _gen(seed, 5)
    M, N, P = case["M"], case["N"], case["problems"]
    nA = 1 if case["shared"] else P
    A = torch.randn(nA, M, N, generator=g, device="cuda") / math.sqrt(M)
    keep = torch.rand(P, N, generator=g, device="cuda").argsort(dim=1) < max(1, N // 10)
    x = torch.randn(P, N, generator=g, device="cuda") * keep
    b = x @ A[0].T if case["shared"] else torch.bmm(A, x[:, :, None])[:, :, 0]
    return A, (b + 0.01 * torch.randn(P, M, generator=g, device="cuda")).contiguous()


def cnn_weights(seed):
    """A partly trained network: He-normal layers, a small last one, biases."""
    rng = np.random.default_rng([int(seed), 6])
    out = []
    for l in range(6):
        std = math.sqrt(2.0 / (9 * CNN[l])) * (0.1 if l == 5 else 1.0)
        out.append(((rng.standard_normal((3, 3, CNN[l], CNN[l + 1])) * std).astype(np.float32),
                    (rng.standard_normal(CNN[l + 1]) * 0.01).astype(np.float32)))
    return out


def cnn_case(case):
    return fourier("solve", case["n"], case["batch"], "db4", 4 if case["n"] % 16 == 0 else 3, "iso")


def cnn_inputs(case, seed):
    c = cnn_case(case)
    x, mask, b = slices(c, seed)
    y = b.real.to(torch.complex64) if c["real"] else b
    atb = torch.fft.ifft2(mask * y, norm="ortho").contiguous()
    return c, x, mask, b, atb


def prepare(case, seed):
    with torch.cuda.stream(stream()):
        state = _prepare(dict(case), seed)
    stream().synchronize()
    return state


def _prepare(case, seed):
    op = case["op"]
    if op == "dense":
        A, b = dense_inputs(case, seed)
        ctx = F.DenseContext(case["M"], case["N"], case["problems"], shared=case["shared"], stream=stream())
        ctx.set_matrix(A[0].contiguous() if case["shared"] else A)
        return dict(op=op, ctx=ctx, b=b, out=torch.empty(case["problems"], case["N"], device="cuda"),
                    params=F.make_params(case["outer"], case["pcg"], lam=0.05, precond=case["precond"]))
    if op == "multi":
        subs = [(c, *slices(c, seed + 17 * i)) for i, c in enumerate(multi_cases(case))]
        # a stream per size, so that the sizes run side by side
        ctxs = []
        for i, (c, _, mask, _) in enumerate(subs):
            ctx = F.Context(c["n"], batch=c["batch"], stream=stream() if i == 0 else torch.cuda.Stream())
            ctx.set_operator(mask, psi_of(c), c["levels"])
            ctxs.append(ctx)
        torch.cuda.synchronize()
        return dict(op=op, ctxs=ctxs, bs=[s[3] for s in subs], params=[params(c) for c, *_ in subs],
                    outs=[torch.empty_like(s[3]) for s in subs])
    if op in ("train", "warm"):
        c, x, mask, b, atb = cnn_inputs(case, seed)
        net = F.Cnn(case["n"], case["batch"], stream=stream())
        net.set_params(cnn_weights(seed))
        st = dict(op=op, net=net, mask=mask, b=b, atb=atb, x1=torch.empty_like(atb))
        if op == "train":
            return dict(st, target=x.contiguous(), lr=case["lr"])
        return dict(st, ctx=context(c, mask), params=params(c), x2=torch.empty_like(atb), x0=torch.empty_like(atb))
    x, mask, b = slices(case, seed)
    st = dict(op=op, ctx=context(case, mask), b=b, params=params(case), out=torch.empty_like(b))
    if op == "aha":
        return dict(st, d=sp_inputs(case, x, seed)[1])
    if op == "sp":
        xk, d, r = sp_inputs(case, x, seed)
        return dict(st, x=xk, d=d, r=r, z=torch.empty_like(b))
    return st


# --------------------------------------------------------------------- run --

def run(state):
    with torch.cuda.stream(stream()):
        op = state["op"]
        if op == "aha":
            state["ctx"].apply_AHA(state["d"], state["out"])
            return state["out"]
        if op == "sp":
            state["ctx"].apply_S_P(state["params"], state["x"], state["d"], state["out"], state["r"], state["z"])
            return [state["out"], state["z"]]
        if op in ("solve", "dense"):
            return state["ctx"].solve(state["b"], state["params"], out=state["out"])
        if op == "multi":
            B.solve_multi(state["ctxs"], state["bs"], state["params"], state["outs"])
            return state["outs"]
        if op == "train":
            net = state["net"]
            loss = net.train_step(state["atb"], state["mask"], state["target"], state["lr"], out=state["x1"])
            return dict(x1=state["x1"], loss=loss, grads=net.get_grads(), weights=net.get_params())
        x1 = state["net"].forward(state["atb"], state["mask"], out=state["x1"])
        x2 = state["ctx"].data_consistency(state["b"], x1, out=state["x2"])
        kept = state["ctx"].warm_start_guard(state["b"], state["params"], x2, state["x0"])
        return dict(x1=x1, x2=x2, x0=state["x0"], kept=np.array(kept))


def work(case):
    """Bytes: inputs and results once per pass over the data that cannot stay
    on the chip; operations of the transforms, stencils, sweeps and products."""
    op = case["op"]
    if op == "multi":
        ws = [work(c) for c in multi_cases(case)]
        return {k: sum(w[k] for w in ws) for k in ("bytes", "flops")}
    if op == "dense":
        M, N, P = case["M"], case["N"], case["problems"]
        steps = case["outer"] * (case["pcg"] + 1)
        nA = 1 if case["shared"] else P
        # a private matrix is read in every step; a shared one stays in the cache
        return dict(bytes=4.0 * nA * M * N * (1 if case["shared"] else steps) + 4.0 * P * (M + N),
                    flops=4.0 * P * M * N * steps)
    px = float(case["batch"]) * case["n"] ** 2
    if op in ("train", "warm"):
        mac = 9 * sum(CNN[l] * CNN[l + 1] for l in range(6))
        act = 2 * (sum(CNN[:6]) + sum(CNN[1:6]))  # each activation written and read once, 16 bits
        if op == "warm":
            return dict(bytes=px * (act + 17 + 25 + 40), flops=px * (2 * mac + 200))
        return dict(bytes=px * (3 * act + 25), flops=px * 6 * mac)
    log = math.log2(case["n"])
    fft = 20 * log  # a forward and an inverse 2-D transform per pixel
    if op == "aha":
        return dict(bytes=17 * px, flops=fft * px)
    wav, tv = bool(case["wavelet"]), bool(case["tv"])
    # a PCG step: d, r, dx read and written, q and z once each, the weights and
    # the mask read, in the two passes that its inner products part
    step = 8 * 8 + 1 + (4 if wav else 0) + (8 if tv else 0)
    flops = fft + 30 + (110 if wav else 0) + (60 if tv else 0)
    if op == "sp":
        return dict(bytes=(5 * 8 + 1) * px, flops=(2 * flops) * px)
    steps = case["outer"] * (case["pcg"] + 1)
    return dict(bytes=px * (steps * step + 17), flops=px * steps * flops)


# ------------------------------------------------------------------- exact --
# FIRLS in 64 bits: the unitary FFT, a filter bank, the penta-diagonal factors
# solved along anti-diagonals, textbook PCG.

def taps(wavelet):
    if wavelet == "haar":
        h = [1 / math.sqrt(2)] * 2
    else:
        s, q = math.sqrt(3.0), 4 * math.sqrt(2.0)
        h = [(1 + s) / q, (3 + s) / q, (3 - s) / q, (1 - s) / q]
    return h, [(-1) ** t * h[len(h) - 1 - t] for t in range(len(h))]


def split1(x, wavelet, dim):
    h, g = taps(wavelet)
    rolled = [torch.roll(x, -t, dim) for t in range(len(h))]
    at = [slice(None)] * x.dim()
    at[dim] = slice(0, None, 2)
    return torch.cat([sum(c * r[tuple(at)] for c, r in zip(f, rolled)) for f in (h, g)], dim)


def join1(c, wavelet, dim):
    h, g = taps(wavelet)
    a, d = c.chunk(2, dim)
    at = [slice(None)] * c.dim()
    at[dim] = slice(0, None, 2)
    out = torch.zeros_like(c)
    for t in range(len(h)):
        up = torch.zeros_like(c)
        up[tuple(at)] = h[t] * a + g[t] * d
        out += torch.roll(up, t, dim)
    return out


def phi(x, wavelet, levels):
    c = x.clone()
    for l in range(levels):
        m = x.shape[-1] >> l
        c[..., :m, :m] = split1(split1(c[..., :m, :m], wavelet, -1), wavelet, -2)
    return c


def phi_t(c, wavelet, levels):
    x = c.clone()
    for l in reversed(range(levels)):
        m = c.shape[-1] >> l
        x[..., :m, :m] = join1(join1(x[..., :m, :m], wavelet, -2), wavelet, -1)
    return x


def diag_phi(w, wavelet, levels):
    """diag(Phi^T diag(w) Phi): squared basis functions, band by band."""
    n = w.shape[-1]
    low, out = torch.eye(n, dtype=w.dtype, device=w.device), torch.zeros_like(w)
    for l in range(1, levels + 1):
        both = split1(low, wavelet, 0)
        h = n >> l
        f = (both[:h] ** 2, both[h:2 * h] ** 2)
        for br, bc in ((0, 1), (1, 0), (1, 1)) + (((0, 0),) if l == levels else ()):
            out += f[br].T @ w[..., br * h:(br + 1) * h, bc * h:(bc + 1) * h] @ f[bc]
        low = both[:h]
    return out


def ahead(x, dim):
    """x at the next pixel along dim, zero past the border."""
    y = torch.zeros_like(x)
    n = x.shape[dim]
    y.narrow(dim, 0, n - 1).copy_(x.narrow(dim, 1, n - 1))
    return y


def behind(x, dim):
    y = torch.zeros_like(x)
    n = x.shape[dim]
    y.narrow(dim, 1, n - 1).copy_(x.narrow(dim, 0, n - 1))
    return y


class System:
    """S and P of one reweighting of a batch, for the iterate x."""

    def __init__(self, case, mask, x):
        self.c, self.mask = case, mask.to(torch.float64)
        lam, lam_tv = lambdas(case)
        # the library takes its parameters in 32 bits
        self.lam, self.lam_tv = float(np.float32(lam)), float(np.float32(lam_tv))
        eps = float(np.float32(case["eps"]))
        self.abar = self.mask.mean(dim=(-2, -1), keepdim=True)
        C, n = case["channels"], case["n"]

        def over_images(v):
            s = v.reshape(-1, C, n, n).sum(1, keepdim=True).expand(-1, C, n, n)
            return s.reshape(-1, n, n)

        if case["wavelet"]:
            p = phi(x, case["wavelet"], case["levels"]).abs() ** 2
            if case["tree"]:
                g = tree_map(n, case["levels"]).long()
                p = p.reshape(p.shape[0], -1)
                wg = (p[:, g[:, 0]] + p[:, g[:, 1]] + eps) ** -0.5
                w = torch.zeros_like(p)
                w.index_add_(1, g[:, 0], wg)
                w.index_add_(1, g[:, 1], wg)
                self.w = w.reshape(-1, n, n)
            else:
                self.w = (over_images(p) + eps) ** -0.5
        if case["tv"]:
            g1, g2 = (x - behind(x, -1)).abs() ** 2, (x - behind(x, -2)).abs() ** 2
            if case["tv"] == "iso":
                self.w1 = self.w2 = (over_images(g1 + g2) + eps) ** -0.5
            else:
                self.w1, self.w2 = (g1 + eps) ** -0.5, (g2 + eps) ** -0.5
        self._factor()

    def aha(self, d):
        q = torch.fft.ifft2(self.mask * torch.fft.fft2(d, norm="ortho"), norm="ortho")
        return q.real.to(q.dtype) if self.c["real"] else q

    def S(self, d):
        c = self.c
        q = self.aha(d)
        if c["wavelet"]:
            u = phi_t(self.w * phi(d, c["wavelet"], c["levels"]), c["wavelet"], c["levels"])
            q = q + self.lam * u
        if c["tv"]:
            e1, e2 = self.w1 * (d - behind(d, -1)), self.w2 * (d - behind(d, -2))
            q = q + self.lam_tv * (e1 - ahead(e1, -1) + e2 - ahead(e2, -2))
        return q

    def _factor(self):
        c = self.c
        if c["precond"] == "none":
            return
        if not c["tv"] and c["precond"] == "paper":
            self.pinv = 1.0 / (self.abar + self.lam * self.w)
            return
        a = self.abar.expand(c["batch"], c["n"], c["n"]).clone()
        if c["wavelet"]:
            a += self.lam * diag_phi(self.w, c["wavelet"], c["levels"])
        if c["tv"]:
            a += self.lam_tv * (self.w1 + ahead(self.w1, -1) + self.w2 + ahead(self.w2, -2))
        if c["precond"] == "jacobi":
            self.ia = 1.0 / a
            return
        # couplings to the left and upper neighbour (zero on the border), by
        # anti-diagonal: [2n-1][batch][n rows]
        n = c["n"]
        i = torch.arange(n, device=a.device)
        self.at = ((i[:, None] + i[None, :]) * n + i[:, None]).reshape(-1)
        left, up = self.lam_tv * self.w1, self.lam_tv * self.w2
        left[..., 0], up[..., 0, :] = 0.0, 0.0
        A, L, U = (self._skew(v) for v in (a, left, up))
        D = A.clone()
        if c["precond"] == "ilu0":
            for k in range(1, 2 * n - 1):
                prev = D[k - 1]
                t = L[k] ** 2 / torch.where(prev == 0, 1.0, prev)
                t[:, 1:] += U[k][:, 1:] ** 2 / torch.where(prev == 0, 1.0, prev)[:, :-1]
                D[k] -= t
        inv = torch.where(D == 0, 0.0, 1.0 / torch.where(D == 0, 1.0, D))
        self.inv, self.gl, self.gu = inv, torch.zeros_like(L), torch.zeros_like(U)
        self.gl[1:] = L[1:] * inv[:-1]
        self.gu[1:, :, 1:] = U[1:, :, 1:] * inv[:-1, :, :-1]
        self.bl, self.bu = torch.zeros_like(L), torch.zeros_like(U)
        self.bl[:-1] = inv[:-1] * L[1:]
        self.bu[:-1, :, :-1] = inv[:-1, :, :-1] * U[1:, :, 1:]

    def _skew(self, v):
        n = self.c["n"]
        s = torch.zeros((2 * n - 1) * n, v.shape[0], *v.shape[3:], dtype=v.dtype, device=v.device)
        s[self.at] = v.reshape(v.shape[0], n * n, *v.shape[3:]).transpose(0, 1)
        return s.reshape(2 * n - 1, n, v.shape[0], *v.shape[3:]).transpose(1, 2).contiguous()

    def P(self, r):
        c = self.c
        if c["precond"] == "none":
            return r
        if c["precond"] == "jacobi":
            return self.ia * r
        if not c["tv"]:
            z = phi_t(self.pinv * phi(r, c["wavelet"], c["levels"]), c["wavelet"], c["levels"])
            return z.real.to(z.dtype) if c["real"] else z
        n = c["n"]
        y = self._skew(torch.view_as_real(r))
        for k in range(1, 2 * n - 1):
            y[k].addcmul_(self.gl[k][..., None], y[k - 1])
            y[k][:, 1:].addcmul_(self.gu[k][:, 1:, None], y[k - 1][:, :-1])
        y *= self.inv[..., None]
        for k in range(2 * n - 3, -1, -1):
            y[k].addcmul_(self.bl[k][..., None], y[k + 1])
            y[k][:, :-1].addcmul_(self.bu[k][:, :-1, None], y[k + 1][:, 1:])
        z = y.transpose(1, 2).reshape((2 * n - 1) * n, -1, 2)[self.at].transpose(0, 1)
        return torch.view_as_complex(z.reshape(-1, n, n, 2).contiguous())


def solve64(case, mask, b):
    C = case["channels"]

    def dot(u, v):
        s = (u.real * v.real + u.imag * v.imag).sum((-2, -1)).reshape(-1, C).sum(1, keepdim=True)
        return s.expand(-1, C).reshape(-1, 1, 1)

    atb = torch.fft.ifft2(mask * b.to(torch.complex128), norm="ortho")
    atb = atb.real.to(atb.dtype) if case["real"] else atb
    x = atb.clone()
    for _ in range(case["outer"]):
        A = System(case, mask, x)
        r = atb - A.S(x)
        d = A.P(r)
        rho, dx = dot(r, d), torch.zeros_like(x)
        for j in range(case["pcg"]):
            q = A.S(d)
            alpha = rho / dot(d, q)
            dx += alpha * d
            if j + 1 == case["pcg"]:
                break
            r -= alpha * q
            z = A.P(r)
            new = dot(r, z)
            d = z + (new / rho) * d
            rho = new
        x = x + dx
    return x


def dense64(case, A, b):
    A, b = A.double(), b.double()
    lam, eps = float(np.float32(0.05)), float(np.float32(EPS))
    if case["shared"]:
        ata, atb = (lambda v: (v @ A[0].T) @ A[0]), b @ A[0]
    else:
        ata = lambda v: torch.bmm(torch.bmm(A, v[:, :, None]).transpose(1, 2), A)[:, 0]  # noqa: E731
        atb = torch.bmm(b[:, None], A)[:, 0]
    sq = (A * A).sum(1)
    abar = sq.mean(1, keepdim=True)
    x = atb.clone()
    for _ in range(case["outer"]):
        w = (x * x + eps) ** -0.5
        P = {"paper": abar + lam * w, "jacobi": sq + lam * w, "none": torch.ones_like(w)}[case["precond"]]
        r = atb - (ata(x) + lam * w * x)
        d = r / P
        rho, dx = (r * d).sum(1, keepdim=True), torch.zeros_like(x)
        for _ in range(case["pcg"]):
            q = ata(d) + lam * w * d
            alpha = rho / (d * q).sum(1, keepdim=True)
            dx += alpha * d
            r = r - alpha * q
            z = r / P
            new = (r * z).sum(1, keepdim=True)
            d = z + (new / rho) * d
            rho = new
        x = x + dx
    return x


def net64(ws, atb, mask):
    """x1 = atb + CNN(.): a 3x3 convolution is a product per tap."""
    n = atb.shape[-1]
    a = torch.stack([atb.real, atb.imag, mask.to(torch.float64)], -1)
    for l, (w, b) in enumerate(ws):
        p = torch.nn.functional.pad(a, (0, 0, 1, 1, 1, 1))
        z = b
        for dy in range(3):
            for dx in range(3):
                z = z + p[:, dy:dy + n, dx:dx + n] @ w[dy, dx]
        a = torch.relu(z) if l < 5 else z
    return torch.complex(atb.real + a[..., 0], atb.imag + a[..., 1])


def exact(case, seed):
    op = case["op"]
    if op == "dense":
        return dense64(case, *dense_inputs(case, seed))
    if op == "multi":
        return [solve64(c, *slices(c, seed + 17 * i)[1:]) for i, c in enumerate(multi_cases(case))]
    if op in ("train", "warm"):
        c, x, mask, b, atb = cnn_inputs(case, seed)
        atb = atb.to(torch.complex128)
        ws = [tuple(torch.from_numpy(v).cuda().double() for v in wb) for wb in cnn_weights(seed)]
        if op == "warm":
            with torch.no_grad():
                x1 = net64(ws, atb, mask)
                k = torch.fft.fft2(x1, norm="ortho")
                x2 = torch.fft.ifft2(torch.where(mask.bool(), b.to(k.dtype), k), norm="ortho")
            return dict(x1=x1, x2=x2, x0=None, kept=None)  # the guard chooses by two near values
        for wb in ws:
            for v in wb:
                v.requires_grad_(True)
        x1 = net64(ws, atb, mask)
        e = x1 - x.to(torch.complex128)
        loss = (e.real ** 2 + e.imag ** 2).sum()
        flat = [v for wb in ws for v in wb]
        grads = torch.autograd.grad(loss, flat)
        # Adam's first step: m / c1 = g, v / c2 = g^2
        new = [(v - case["lr"] * g / (g.abs() + 1e-8)).detach() for v, g in zip(flat, grads)]

        def pairs(v):
            return [tuple(v[i:i + 2]) for i in range(0, 12, 2)]

        return dict(x1=x1.detach(), loss=float(loss), grads=pairs(grads), weights=pairs(new))
    x, mask, b = slices(case, seed)
    if op == "aha":
        d = sp_inputs(case, x, seed)[1].to(torch.complex128)
        q = torch.fft.ifft2(mask * torch.fft.fft2(d, norm="ortho"), norm="ortho")
        return q.real.to(q.dtype) if case["real"] else q
    if op == "sp":
        xk, d, r = (v.to(torch.complex128) for v in sp_inputs(case, x, seed))
        A = System(case, mask, xk)
        return [A.S(d), A.P(r)]
    return solve64(case, mask, b)
