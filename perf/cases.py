"""What a user of the solver has it do, as measurable cases.

A case is one call sequence through the public entry points, on inputs that are already on the GPU, as they are
between the steps of a refinement: back-projection of a batch of images, the reweighted solve of a new data volume
(one map, several maps at once, real-space or Fourier-domain data term), its monitoring, the differentiable solve,
and the shell correlation of two half-maps. Inputs are drawn on the GPU from the seed: Gaussian blobs, a smooth
positive weight field and white noise, the distributions of ``synth.py``.
"""
import math

import torch

from paper_1905_13408_gb300 import spg

HYPER = dict(lambda_l1=0.05, lambda_tv=0.1, mu=1e-3, eps=1e-3, eps_tv=1e-3)
L2_BYTES = 126 << 20
STEP_FLOPS = 60  # of one voxel in one iteration (differences, clip, divergence, step, threshold, objective)


# ---------------------------------------------------------------- the cases

def listed():
    return [
        # a class average or a masked sub-volume: a handful of iterations, where launches and host calls count
        dict(name="solve-small", kind="solve", nz=28, ny=32, nx=40, rounds=1, iters=20),
        # the smallest workload of the repository, its full schedule
        dict(name="solve-64", kind="solve", nz=64, ny=64, nx=64, rounds=3, iters=200),
        # a map cropped to its particle: odd extents, rows that are no multiple of the pitch, gradient restart on
        dict(name="solve-ragged", kind="solve", nz=101, ny=147, nx=183, rounds=2, iters=60, restart=True),
        # the M step of an ordinary box, anchored to the previous step's map (the implicit-gradient term)
        dict(name="solve-256", kind="solve", nz=256, ny=256, nx=256, rounds=2, iters=50, gamma=0.1),
        # a larger box with b and w kept in bfloat16 and the storage form of fewest bytes
        dict(name="solve-384-bf16", kind="solve", nz=384, ny=384, nx=384, rounds=1, iters=40, dtype="bf16",
             storage="prev"),
        # the paper's own size
        dict(name="solve-512", kind="solve", nz=512, ny=512, nx=512, rounds=2, iters=15),
        # classes and half-maps of one refinement, advanced together (the 24 volumes of the batched workload)
        dict(name="batch-24", kind="batch", volumes=24, smallest=96, largest=256, rounds=1, iters=30),
        # learning the data, weights and regularisation: forward and backward of the unrolled solve
        dict(name="unrolled-128", kind="unrolled", nz=128, ny=128, nx=128, K=50, ckpt=10),
        # Fourier-domain data term, power-of-two box and one of the usual boxes that is not
        dict(name="fourier-256", kind="fourier", nz=256, ny=256, nx=256, iters=30),
        dict(name="fourier-180", kind="fourier", nz=180, ny=180, nx=180, iters=30),
        # a batch of particle images into the gridded spectrum, and its conversion to the data term
        dict(name="grid-256", kind="grid", n=256, images=2048, kernel="gauss", posterior=True),
        # the gold-standard resolution estimate after each refinement step
        dict(name="fsc-256", kind="fsc", n=256),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "batch", "unrolled", "fourier", "grid", "fsc"])
    if kind == "solve":
        edge = [_log(rng, 24, 400) for _ in range(3)]
        while edge[0] * edge[1] * edge[2] > 320 ** 3:
            edge[rng.randrange(3)] //= 2
        nz, ny, nx = edge
        rounds = rng.randint(1, 3)
        iters = min(_log(rng, 10, 200), max(5, int(4e9 / (rounds * nz * ny * nx))))
        c = dict(kind=kind, nz=nz, ny=ny, nx=nx, rounds=rounds, iters=iters)
        c["dtype"] = rng.choice(["f32", "f32", "bf16"])
        c["storage"] = rng.choice(["delta", "delta", "prev"])
        c["restart"] = rng.random() < 0.25
        c["gamma"] = rng.choice([0.0, 0.0, 0.05, 0.2])
        return c
    if kind == "batch":
        lo = _log(rng, 32, 128)
        return dict(kind=kind, volumes=rng.randint(2, 16), smallest=lo, largest=rng.randint(lo, 224), rounds=1,
                    iters=rng.randint(10, 30))
    if kind == "unrolled":
        nz, ny, nx = (_log(rng, 24, 144) for _ in range(3))
        return dict(kind=kind, nz=nz, ny=ny, nx=nx, K=rng.randint(10, 50), ckpt=rng.randint(4, 12))
    if kind == "fourier":
        if rng.random() < 0.5:
            nz, ny, nx = (2 ** rng.randint(6, 8) for _ in range(3))
        else:
            nz, ny, nx = (2 * _log(rng, 20, 110) for _ in range(3))
        return dict(kind=kind, nz=nz, ny=ny, nx=nx, iters=rng.randint(10, 30))
    if kind == "grid":
        n = 2 * _log(rng, 16, 144)
        images = min(_log(rng, 32, 4096), 2048 * 65536 // (n * n))
        return dict(kind=kind, n=n, images=images, kernel=rng.choice(["gauss", "gauss", "trilinear"]),
                    posterior=rng.random() < 0.5)
    return dict(kind=kind, n=_log(rng, 32, 288))


# ---------------------------------------------------------------- inputs

def _gen(seed, salt=0):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1000003 + salt) % (1 << 62))
    return g


def _smooth(a, sigma):
    """Periodic Gaussian smoothing through the transform."""
    k2 = 0.0
    for i, n in enumerate(a.shape):
        f = torch.fft.rfftfreq(n, device="cuda") if i == 2 else torch.fft.fftfreq(n, device="cuda")
        k2 = k2 + (f * f).reshape([-1 if j == i else 1 for j in range(3)])
    return torch.fft.irfftn(torch.fft.rfftn(a) * torch.exp(-2.0 * math.pi ** 2 * sigma ** 2 * k2), s=a.shape)


def _phantom(shape, g):
    """About one blob of sigma 1.5 .. 3 per 10 000 voxels, amplitudes 0.5 .. 1, inside the central ball."""
    n = shape[0] * shape[1] * shape[2]
    out = torch.zeros(shape, device="cuda")
    r = torch.rand(4, max(2, n // 20000), generator=g, device="cuda")
    for s in (1.7, 2.6):
        pts = [((r[i].sub(0.5) * 0.75 + 0.5) * shape[i]).long().clamp_(0, shape[i] - 1) for i in range(3)]
        spikes = torch.zeros(shape, device="cuda")
        spikes[pts[0], pts[1], pts[2]] = (0.5 + 0.5 * r[3]) * (2 * math.pi * s * s) ** 1.5
        out += _smooth(spikes, s)
        r = torch.rand(r.shape, generator=g, device="cuda")
    return out


def _volume(shape, seed, salt=0):
    """(b, w, start, phantom): data, weights, the previous step's map and the truth, float32."""
    g = _gen(seed, salt)
    ph = _phantom(shape, g)
    f = _smooth(torch.randn(shape, generator=g, device="cuda"), 4.0)
    f = (f - f.mean()) / f.std()
    w = torch.exp(0.5 * f)
    b = ph + 0.3 * torch.randn(shape, generator=g, device="cuda") / torch.sqrt(w)
    x0 = 0.9 * ph * (ph > 0.05) + 0.02 * torch.randn(shape, generator=g, device="cuda") * (ph > 0.05)
    return b.contiguous(), w.contiguous(), x0.contiguous(), ph


def _shape(c):
    return (c["nz"], c["ny"], c["nx"])


def _batch_shapes(c):
    """Cubes from the smallest to the largest edge, in as many equal groups of sizes as there are (up to 4)."""
    n, lo, hi = c["volumes"], c["smallest"], c["largest"]
    edges = [int(round(lo * (hi / lo) ** (q / 3.0))) for q in range(4)]
    return [(edges[4 * j // n],) * 3 for j in range(n)]


def _solve_inputs(c, seed):
    b, w, x0, _ = _volume(_shape(c), seed)
    if c.get("dtype") == "bf16":
        b, w = b.bfloat16(), w.bfloat16()
    return b, w, x0


def _batch_inputs(c, seed):
    g = _gen(seed, 99)
    lam = (0.05 + 0.15 * torch.rand(c["volumes"], generator=g, device="cuda")).cpu().tolist()
    return [_volume(s, seed, 1 + j)[:3] for j, s in enumerate(_batch_shapes(c))], [round(v, 4) for v in lam]


def _fourier_inputs(c, seed):
    """(y, N, start): half spectra of Eq. 31 with an N that falls off with resolution and direction."""
    shape = _shape(c)
    g = _gen(seed)
    ph = _phantom(shape, g)
    kz = torch.fft.fftfreq(shape[0], device="cuda")[:, None, None]
    ky = torch.fft.fftfreq(shape[1], device="cuda")[None, :, None]
    kx = torch.fft.rfftfreq(shape[2], device="cuda")[None, None, :]
    k2 = kz * kz + ky * ky + kx * kx
    N = 4.0 * torch.exp(-k2 / (2 * 0.15 ** 2)) * (0.25 + 0.75 * kz.abs() / k2.clamp(min=1e-12).sqrt()) + 0.05
    y = torch.sqrt(N) * torch.fft.rfftn(ph, norm="ortho")
    y = y + 0.3 * torch.fft.rfftn(torch.randn(shape, generator=g, device="cuda"), norm="ortho")
    return y.contiguous(), N.contiguous(), (0.9 * ph * (ph > 0.05)).contiguous()


def _grid_inputs(c, seed):
    """Rotations, image spectra (Hermitian, signal falling off with frequency), CTFs and posterior weights."""
    n, m = c["n"], c["images"]
    g = _gen(seed)
    q = torch.randn(m, 4, generator=g, device="cuda", dtype=torch.float64)
    w, x, y, z = (q / q.norm(dim=1, keepdim=True)).T
    rot = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - z * w), 2 * (x * z + y * w),
                       2 * (x * y + z * w), 1 - 2 * (x * x + z * z), 2 * (y * z - x * w),
                       2 * (x * z - y * w), 2 * (y * z + x * w), 1 - 2 * (x * x + y * y)], 1).float().contiguous()
    f = torch.fft.fftfreq(n, device="cuda")
    s2 = f[:, None] ** 2 + f[None, :] ** 2
    X = torch.empty(m, n, n, dtype=torch.complex64, device="cuda")
    ctf = torch.empty(m, n, n, device="cuda")
    defocus = 0.5 + torch.rand(m, 1, 1, generator=g, device="cuda")
    fall = 1.0 + 20.0 * torch.exp(-40.0 * s2)
    step = max(1, (1 << 24) // (n * n))
    for i in range(0, m, step):
        d = defocus[i:i + step]
        ctf[i:i + step] = torch.sin(0.5 + 30.0 * d * s2)
        X[i:i + step] = torch.fft.fft2(torch.randn(d.shape[0], n, n, generator=g, device="cuda")) * fall
    pw = 0.2 + 0.8 * torch.rand(m, generator=g, device="cuda") if c["posterior"] else None
    return rot, X, ctf, pw


def _fsc_inputs(c, seed):
    g = _gen(seed)
    shape = (c["n"],) * 3
    ph = _phantom(shape, g)
    return [(ph + 0.3 * torch.randn(shape, generator=g, device="cuda")).contiguous() for _ in range(2)]


# ---------------------------------------------------------------- what is measured

def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind == "solve":
        b, w, x0 = _solve_inputs(c, seed)
        s = spg.SPG(dict(shape=_shape(c), **HYPER), data_dtype=c.get("dtype", "f32"),
                    storage=c.get("storage", "delta"), restart=c.get("restart", False))
        return dict(case=c, solver=s, b=b, w=w, x0=x0)
    if kind == "batch":
        vols, lam = _batch_inputs(c, seed)
        s = spg.SPG([dict(HYPER, shape=v[0].shape, lambda_tv=t) for v, t in zip(vols, lam)])
        return dict(case=c, solver=s, vols=vols)
    if kind == "unrolled":
        b, w, _, ph = _volume(_shape(c), seed)
        return dict(case=c, b=b.requires_grad_(), w=w.requires_grad_(), target=ph,
                    l1=torch.tensor(HYPER["lambda_l1"], requires_grad=True),
                    tv=torch.tensor(HYPER["lambda_tv"], requires_grad=True))
    if kind == "fourier":
        y, N, x0 = _fourier_inputs(c, seed)
        return dict(case=c, solver=spg.SPG(dict(shape=_shape(c), **HYPER)), y=y, N=N, x0=x0)
    if kind == "grid":
        return dict(case=c, grid=spg.Grid(c["n"], kernel=c["kernel"]), inputs=_grid_inputs(c, seed))
    return dict(case=c, maps=_fsc_inputs(c, seed))


def run(state):
    c, kind = state["case"], state["case"]["kind"]
    if kind == "solve":
        s = state["solver"]
        bf16 = c.get("dtype") == "bf16"
        s.set_data(0, state["b"], state["w"], spg.SPG_BF16 if bf16 else spg.SPG_F32)
        if c.get("gamma"):
            s.set_anchor(0, c["gamma"], state["x0"])
        s.set_x(0, state["x0"])
        s.solve(c["rounds"], c["iters"])
        out = dict(x=s.get_x(0), objective=s.objective(0))
        # the gap bound after the last round, as a stopping test reads it
        out["certificate"] = s.certificate(0)
        return out
    if kind == "batch":
        s = state["solver"]
        for j, (b, w, x0) in enumerate(state["vols"]):
            s.set_data(j, b, w)
            s.set_x(j, x0)
        s.solve(c["rounds"], c["iters"])
        return dict(x=[s.get_x(j) for j in range(s.nvol)])
    if kind == "unrolled":
        x = spg.UnrolledSPG.apply(state["b"], state["w"], state["l1"], state["tv"], c["K"], ckpt_every=c["ckpt"],
                                  **{k: HYPER[k] for k in ("mu", "eps", "eps_tv")})
        loss = ((x - state["target"]) ** 2).sum()
        g = torch.autograd.grad(loss, [state["b"], state["w"], state["l1"], state["tv"]])
        return dict(x=x.detach(), gb=g[0], gw=g[1], gl1=g[2], gtv=g[3])
    if kind == "fourier":
        s = state["solver"]
        s.set_data_fourier(0, state["y"], state["N"])
        s.set_x(0, state["x0"])
        s.solve(1, c["iters"])
        return dict(x=s.get_x(0), objective=s.objective(0))
    if kind == "grid":
        g = state["grid"]
        g.reset()
        g.add(*state["inputs"])
        y, N = g.finish()
        return dict(y=y, N=N)
    fsc, counts = spg.spg_fsc(*state["maps"], stream=torch.cuda.current_stream().cuda_stream)
    return dict(fsc=fsc, counts=counts)


def _solve_bytes(vox, per_iter, iters, rounds, once):
    """`iters` passes over the volume's arrays, or one where they stay in the L2 cache between iterations."""
    if vox * per_iter <= L2_BYTES:
        return vox * once
    return vox * (once + rounds * (iters * per_iter + 12))  # 12: x read, om1 and omtv written by the re-weighting


def work(case):
    c, kind = case, case["kind"]
    if kind == "solve":
        vox = c["nz"] * c["ny"] * c["nx"]
        es = 2 if c.get("dtype") == "bf16" else 4
        # x_k, x_{k-1}, om1, omtv, b, w read, x_{k+1} written; once: b, w, the start in, x out
        return dict(bytes=_solve_bytes(vox, 20 + 2 * es, c["iters"], c["rounds"], 8 + 2 * es),
                    flops=STEP_FLOPS * vox * c["iters"] * c["rounds"])
    if kind == "batch":
        vox = sum(s[0] * s[1] * s[2] for s in _batch_shapes(c))
        return dict(bytes=_solve_bytes(vox, 28, c["iters"], c["rounds"], 16),
                    flops=STEP_FLOPS * vox * c["iters"] * c["rounds"])
    if kind == "unrolled":
        vox = c["nz"] * c["ny"] * c["nx"]
        # forward 28 each; backward a forward sweep, a recomputation, and an adjoint step that reads x_k, x_{k-1},
        # b, w, om1, omtv, the cotangents of x_{k+1} and x_k, and accumulates b's and w's and writes x_{k-1}'s
        K = c["K"]
        return dict(bytes=vox * K * (28 + 28 + 28 * (1 - 1.0 / c["ckpt"]) + 56), flops=vox * K * (3 * 40 + 120))
    if kind == "fourier":
        vox = c["nz"] * c["ny"] * c["nx"]
        half = c["nz"] * c["ny"] * (c["nx"] // 2 + 1)
        # forward and inverse real transform (each in and out once), N and the data spectrum, the step on the gradient
        per = vox * (4 + 4 + 4 + 4) + half * 12 + vox * 24
        fl = c["iters"] * (vox * 5 * math.log2(vox) + STEP_FLOPS * vox)
        return dict(bytes=(half * 12 + vox * 8) + (c["iters"] * per if per > L2_BYTES else 0), flops=fl)
    if kind == "grid":
        n, m = c["n"], c["images"]
        r = n / 2 - 2
        kept = m * math.pi * r * r / 2  # coefficients of a half disc
        half = n * n * (n // 2 + 1)
        return dict(bytes=kept * 12 + half * 12, flops=kept * (27 if c["kernel"] == "gauss" else 8) * 6)
    n = c["n"]
    vox = n ** 3
    return dict(bytes=2 * 4 * vox, flops=2 * 2.5 * vox * math.log2(vox) + 14 * vox / 2)


# ---------------------------------------------------------------- the same in 64 bits

def _diff(u, a):
    """Backward difference along axis a, zero on the first plane (Eq. 12)."""
    d = torch.zeros_like(u)
    d.narrow(a, 1, u.shape[a] - 1).copy_(u.narrow(a, 1, u.shape[a] - 1) - u.narrow(a, 0, u.shape[a] - 1))
    return d


def _div(p):
    """D^T p (Eq. 17): p_a(v) - p_a(v + e_a); p_a vanishes on its first plane."""
    out = 0.0
    for a, q in enumerate(p):
        n = q.shape[a]
        q = torch.cat([torch.zeros_like(q.narrow(a, 0, 1)), q.narrow(a, 1, n - 1)], a)
        out = out + q - torch.cat([q.narrow(a, 1, n - 1), torch.zeros_like(q.narrow(a, 0, 1))], a)
    return out


def _p(u, omtv, mu):
    g = [_diff(u, a) for a in range(3)]
    s = omtv / torch.clamp(g[0] ** 2 + g[1] ** 2 + g[2] ** 2, min=mu * mu).sqrt()
    return [v * s for v in g]


def _betas(n):
    t, out = 1.0, []
    for _ in range(n):
        tn = 0.5 * (1 + math.sqrt(1 + 4 * t * t))
        out.append((t - 1) / tn)
        t = tn
    return out


def _solve64(b, w, x, lam_l1, lam_tv, rounds, iters, restart=False, data=None, max_w=None):
    """The reweighted solve in float64: (x, objective terms, certificate). `data`: (gradient, value) of another data
    term than 1/2 w (x - b)^2."""
    mu, eps, eps_tv = HYPER["mu"], HYPER["eps"], HYPER["eps_tv"]
    grad = data[0] if data else lambda u: w * (u - b)
    value = data[1] if data else lambda u: float((0.5 * w * (u - b) ** 2).sum())
    max_w = float(w.max()) if max_w is None else max_w
    beta = _betas(iters + 1)
    for _ in range(rounds):
        gn = sum(_diff(x, a) ** 2 for a in range(3)).sqrt()
        om1, omtv = eps / (x.abs() + eps), eps_tv / (gn + eps_tv)
        tau = 1.0 / (max_w + 12.0 * lam_tv * float(omtv.max()) / mu)
        d, k = torch.zeros_like(x), 0
        for _ in range(iters):
            y = x + beta[k] * d
            gy = grad(y) + lam_tv * _div(_p(y, omtv, mu))
            z = y - tau * gy
            d = torch.sign(z) * torch.clamp(z.abs() - tau * lam_l1 * om1, min=0.0) - x
            k = 0 if restart and float(((y - x - d) * d).sum()) > 0 else k + 1
            x = x + d
    g2 = sum(_diff(x, a) ** 2 for a in range(3))
    h = torch.where(g2 <= mu * mu, g2 / (2 * mu), g2.sqrt() - mu / 2)
    f = [value(x), lam_l1 * float((om1 * x.abs()).sum()), lam_tv * float((omtv * h).sum())]
    cert = None
    if not data:
        r = (y - x) * (1.0 / tau - w) + lam_tv * (_div(_p(x, omtv, mu)) - _div(_p(y, omtv, mu)))
        cert = float((r * r).sum())
    return x, torch.tensor(f + [sum(f)], dtype=torch.float64), cert


def _unrolled64(c, seed):
    b, w, _, ph = _volume(_shape(c), seed)
    b, w = b.double().requires_grad_(), w.double().requires_grad_()
    l1 = torch.tensor(float(torch.tensor(HYPER["lambda_l1"])), dtype=torch.float64, device="cuda", requires_grad=True)
    tv = torch.tensor(float(torch.tensor(HYPER["lambda_tv"])), dtype=torch.float64, device="cuda", requires_grad=True)
    tau = 1.0 / (float(w.detach().max()) + 12.0 * float(tv) / HYPER["mu"])
    one = torch.ones_like(ph, dtype=torch.float64)
    x = xp = torch.zeros_like(one)
    for bk in _betas(c["K"]):
        y = x + bk * (x - xp)
        z = y - tau * (w * (y - b) + tv * _div(_p(y, one, HYPER["mu"])))
        xp, x = x, torch.where(z.abs() > tau * l1, z - tau * l1 * torch.sign(z), torch.zeros_like(z))
    g = torch.autograd.grad(((x - ph.double()) ** 2).sum(), [b, w, l1, tv])
    return dict(x=x.detach(), gb=g[0], gw=g[1], gl1=g[2], gtv=g[3])


def _fourier64(c, seed):
    y, N, x0 = _fourier_inputs(c, seed)
    shape = _shape(c)
    y, N = y.to(torch.complex128), N.double()
    root = N.sqrt()
    wgt = torch.full((shape[2] // 2 + 1,), 2.0, dtype=torch.float64, device="cuda")
    wgt[0] = 1.0
    if shape[2] % 2 == 0:
        wgt[-1] = 1.0

    def grad(u):
        return torch.fft.irfftn(N * torch.fft.rfftn(u, norm="ortho") - root * y, s=shape, norm="ortho")

    def value(u):
        return float(0.5 * (wgt * (y - root * torch.fft.rfftn(u, norm="ortho")).abs() ** 2).sum())

    x, f, _ = _solve64(None, None, x0.double(), HYPER["lambda_l1"], HYPER["lambda_tv"], 1, c["iters"],
                       data=(grad, value), max_w=float(N.max()))
    return dict(x=x, objective=f)


def _grid64(c, seed):
    rot, X, ctf, pw = _grid_inputs(c, seed)
    n, m = c["n"], c["images"]
    dev = rot.device
    k = torch.arange(-(n // 2), n // 2, device=dev)
    ky, kx = torch.meshgrid(k[n // 2:], k, indexing="ij")
    keep = ((ky > 0) | (kx >= 0)) & ((kx * kx + ky * ky).float() <= (n * 0.5 - 2.0) ** 2)
    kx, ky = kx[keep], ky[keep]
    src = ky * n + kx % n
    wgt = torch.where((kx == 0) & (ky == 0), 0.5, 1.0).double()  # k = 0 is its own mate: half here, half mirrored
    acc = torch.zeros(n ** 3, 3, dtype=torch.float64, device=dev)
    gauss = c["kernel"] == "gauss"
    offs = (-1, 0, 1) if gauss else (0, 1)
    for i in range(0, m, max(1, (1 << 21) // kx.numel())):
        sl = slice(i, i + max(1, (1 << 21) // kx.numel()))
        R = rot[sl].double()
        p = torch.stack([R[:, 3 * a, None] * kx + R[:, 3 * a + 1, None] * ky for a in range(3)])  # x, y, z
        cell = torch.round(p) if gauss else torch.floor(p)
        f, cell = p - cell, cell.long()
        Xs = X[sl].reshape(f.shape[1], -1)[:, src].to(torch.complex128)
        cs = ctf[sl].reshape(f.shape[1], -1)[:, src].double()
        pc = cs * wgt * (pw[sl, None].double() if pw is not None else 1.0)
        val = torch.stack([pc * Xs.real, pc * Xs.imag, pc * cs], -1)
        for oz in offs:
            for oy in offs:
                for ox in offs:
                    e = [f[0] - ox, f[1] - oy, f[2] - oz]
                    K = torch.exp(-(e[0] ** 2 + e[1] ** 2 + e[2] ** 2) / 2.0) if gauss else \
                        (1 - e[0].abs()) * (1 - e[1].abs()) * (1 - e[2].abs())
                    at = ((cell[2] + oz) % n * n + (cell[1] + oy) % n) * n + (cell[0] + ox) % n
                    acc.index_add_(0, at.reshape(-1), (K[..., None] * val).reshape(-1, 3))
    acc = acc.reshape(n, n, n, 3)
    mirror = torch.roll(torch.flip(acc, (0, 1, 2)), (1, 1, 1), (0, 1, 2))
    num = torch.complex(acc[..., 0] + mirror[..., 0], acc[..., 1] - mirror[..., 1])[..., :n // 2 + 1]
    N = (acc[..., 2] + mirror[..., 2])[..., :n // 2 + 1]
    i = torch.arange(n, device=dev)
    sgn = 1.0 - 2.0 * ((i[:, None, None] + i[None, :, None] + i[None, None, :n // 2 + 1]) % 2)
    y = torch.where(N > 0, sgn * num / torch.where(N > 0, N, torch.ones_like(N)).sqrt(), torch.zeros_like(num))
    return dict(y=y, N=N * float(n) ** 3)


def _fsc64(c, seed):
    n = c["n"]
    F, G = (torch.fft.rfftn(a.double()) for a in _fsc_inputs(c, seed))
    f = torch.round(torch.fft.fftfreq(n, device="cuda", dtype=torch.float64) * n)
    h = torch.arange(n // 2 + 1, device="cuda", dtype=torch.float64)
    s = torch.round((f[:, None, None] ** 2 + f[None, :, None] ** 2 + h[None, None, :] ** 2).sqrt()).long().reshape(-1)
    wgt = torch.full((n // 2 + 1,), 2.0, dtype=torch.float64, device="cuda")
    wgt[0] = 1.0
    if n % 2 == 0:
        wgt[-1] = 1.0

    def shells(v):
        v = (v * wgt).reshape(-1)
        return torch.zeros(int(s.max()) + 1, dtype=torch.float64, device="cuda").index_add_(0, s, v)[:n // 2 + 1]

    ab, aa, bb = shells((F * G.conj()).real), shells(F.abs() ** 2), shells(G.abs() ** 2)
    return dict(fsc=ab / (aa * bb).sqrt(), counts=shells(torch.ones_like(F.real)))


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "solve":
        b, w, x0 = (t.double() for t in _solve_inputs(c, seed))
        g = c.get("gamma") or 0.0
        if g:
            b, w = (w * b + 2 * g * x0) / (w + 2 * g), w + 2 * g
            if c.get("dtype") == "bf16":
                return None  # the library rounds the anchored b and w to bfloat16 again
        x, f, cert = _solve64(b, w, x0, HYPER["lambda_l1"], HYPER["lambda_tv"], c["rounds"], c["iters"],
                              c.get("restart", False))
        return dict(x=x, objective=f, certificate=cert)
    if kind == "batch":
        vols, lam = _batch_inputs(c, seed)
        return dict(x=[_solve64(b.double(), w.double(), x0.double(), HYPER["lambda_l1"], t, c["rounds"], c["iters"])[0]
                       for (b, w, x0), t in zip(vols, lam)])
    return dict(unrolled=_unrolled64, fourier=_fourier64, grid=_grid64, fsc=_fsc64)[kind](c, seed)
