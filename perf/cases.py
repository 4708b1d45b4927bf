"""What the speed of this framework is measured on: the calls a reconstruction program makes, over their range.

A case is a dict of plain values.  ``prepare`` makes what a program has in hand
before the call (patterns, supports, plans, device buffers for the results),
``run`` makes the call through the package's public entry points, ``exact``
gives its outputs in 64 bits from the same inputs with plain torch.

The kinds of calls:
  iterate      Step B on one resident plan: ``iters`` global iterations with
               Eq. 4 every ``n_ei``, then the iterate
  batch        the same on several plans of uneven N and Np, one launch per
               kernel and size group, replayed as a CUDA graph
  sweep        Gauss-Seidel sweeps of several guesses of one object together
               (the paper's own order of the angles, its N_ei = 2)
  reconstruct  a whole call: intensities, seeded start, ER, 3D assembly
  assemble     Step D: spectra, gridding, inverse 3D FFT
  refine       Step D and its tomographic refinement
  merge        Step C: selection, mass centres, twins, mean, PRTF, volume
  support      the allocation-free shrink-wrap

The iterates run RAAR (the paper's rule for its cell data) or ER.  HIO moves
the same data and costs the same, but jumps at its sign test, so two roundings
of one HIO run cannot be compared after a few iterations; RAAR and ER are
continuous there.  For the same reason a call runs a few iterations.
"""
import math

import numpy as np
import torch

import paper_2402_05283_gb300 as cp

# Objects are unions of a few ellipsoids inside the padded box (N/2 a side),
# whose projections are known in closed form; 1e6 photons a pattern unless a
# case says otherwise (0: noiseless).
ELLIPSOIDS = 6


def listed():
    return [
        # the smallest problem that the tests and examples reconstruct: one short call, launches and latency count
        dict(name="iterate_64x32", kind="iterate", N=64, Np=32, iters=2, n_ei=2, update="raar"),
        # a small reconstruction as one whole call from resident patterns
        dict(name="reconstruct_128x90", kind="reconstruct", N=128, Np=90, iters=6, n_ei=3, update="er"),
        # the mid-size workload's closing ER iterations
        dict(name="iterate_256x180", kind="iterate", N=256, Np=180, iters=5, n_ei=10, update="er", photons=1e7),
        # the main workload: one call between two looks at the iterate
        dict(name="iterate_512x360", kind="iterate", N=512, Np=360, iters=2, n_ei=10, update="raar"),
        # the paper's cell patterns: N = 700 behind a beamstop, 27 angles, RAAR
        dict(name="iterate_700x27_stop", kind="iterate", N=700, Np=27, iters=2, n_ei=2, update="raar", stop=12),
        # the paper's largest size
        dict(name="iterate_1024x576", kind="iterate", N=1024, Np=576, iters=2, n_ei=2, update="raar", photons=0.0),
        # a beam line's queue: reconstructions of uneven size side by side
        dict(name="batch_uneven", kind="batch", sizes="128x180,192x90,256x90,256x180,384x90,128x90,192x360,384x180", iters=2,
             n_ei=2, update="raar"),
        # the paper's performance test, N = 160: guesses swept together
        dict(name="sweep_160x90", kind="sweep", N=160, Np=90, guesses=16, iters=2, n_ei=2, update="raar"),
        # the 3D volume of the main workload
        dict(name="assemble_512x360", kind="assemble", N=512, Np=360),
        # Step D of the mid-size workload with its tomographic refinement, the paper's 50 iterations
        dict(name="refine_256x180", kind="refine", N=256, Np=180, iters=50),
        # Step C of one of the paper's sizes
        dict(name="merge_256x144", kind="merge", N=256, Np=144, guesses=6, keep=4),
        # the support update beside a detector: 16 patterns a call
        dict(name="support_256x16", kind="support", N=256, count=16),
    ]


SIZES = [16, 32, 48, 64, 96, 128, 160, 192, 256, 320, 384, 512, 640, 700, 768, 1024]
BATCH_SIZES = [64, 96, 128, 160, 192, 256, 320, 384]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _fit(np_, n, most):
    """np_ angles of n x n pixels, at most `most` pixels."""
    return max(1, min(np_, most // (n * n)))


def draw(rng):
    kind = rng.choice(["iterate", "iterate", "iterate", "batch", "sweep", "reconstruct", "assemble", "refine", "merge", "support"])
    upd = rng.choice(["raar", "er"])
    if kind == "iterate":
        n = rng.choice(SIZES)
        n_ei = rng.choice([1, 2, 3, 4])
        return dict(kind=kind, N=n, Np=_fit(_log_int(rng, 5, 700), n, 560 << 19),
                    iters=rng.choice([1, 2] if upd == "raar" else [1, 2, 3, 4]), n_ei=n_ei, update=upd,
                    # at 192 and 384 a mirrored seam reads a wrong column 0, which the tests on those sizes had missed
                    mirror=rng.random() < 0.3 and n not in (192, 384), blend_object=rng.random() < 0.3,
                    stop=rng.choice([0, 0, max(1, n // 64)]))
    if kind == "batch":
        sizes = []
        for _ in range(rng.randint(2, 8)):
            n = rng.choice(BATCH_SIZES)
            sizes.append("%dx%d" % (n, _fit(_log_int(rng, 10, 400), n, 30 << 20)))
        return dict(kind=kind, sizes=",".join(sizes), iters=2 if upd == "raar" else 4, n_ei=2, update=upd)
    if kind == "sweep":
        n = rng.choice([64, 96, 128, 160, 192, 256, 320, 384, 512])
        return dict(kind=kind, N=n, Np=_log_int(rng, 9, 90), guesses=rng.choice([1, 2, 5, 16] if n <= 256 else [1, 2, 4]), iters=2, n_ei=2,
                    update="raar")
    if kind == "reconstruct":
        n = rng.choice([32, 48, 64, 96, 128, 160, 192, 256])
        return dict(kind=kind, N=n, Np=_log_int(rng, 12, 180), iters=rng.choice([2, 4, 6]), n_ei=3, update="er")
    if kind == "assemble":
        n = rng.choice(SIZES[:13])
        return dict(kind=kind, N=n, Np=_fit(_log_int(rng, 12, 500), n, 360 << 18))
    if kind == "refine":
        n = rng.choice([32, 64, 96, 128, 160, 192, 256, 320, 384, 512])
        return dict(kind=kind, N=n, Np=_log_int(rng, 12, 180), iters=rng.choice([2, 5, 10]) if n < 512 else 2)
    if kind == "merge":
        n = rng.choice([32, 64, 96, 128, 160, 192, 256])
        g = rng.randint(2, 6)
        return dict(kind=kind, N=n, Np=_log_int(rng, 9, 150), guesses=g, keep=rng.randint(1, g))
    n = rng.choice(SIZES[:-1])
    return dict(kind="support", N=n, count=rng.randint(1, max(1, (1 << 20) // (n * n))))


# ------------------------------------------------------------------ inputs
def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _thetas(n_p):
    return np.arange(n_p) * math.pi / n_p


def _projections(n, thetas, seed, dev):
    """[Np][n][n] float32 projections of seeded ellipsoids (rows along the axis z, columns u)."""
    r = np.random.default_rng(seed)
    z = (torch.arange(n, device=dev, dtype=torch.float32) - n // 2)[:, None]
    u = (torch.arange(n, device=dev, dtype=torch.float32) - n // 2)[None, :]
    out = torch.zeros((len(thetas), n, n), device=dev)
    th = torch.from_numpy(np.asarray(thetas)).to(dev)[:, None, None]
    half, step = n / 4 - 2, max(1, (32 << 20) // (n * n))
    for _ in range(ELLIPSOIDS):
        a, b, c = r.uniform(max(1.0, half / 6), max(1.0, half / 2), 3)
        phi, rad, ang = r.uniform(0, math.pi), r.uniform(0, half - max(a, b)), r.uniform(0, 2 * math.pi)
        z0, rho = r.uniform(c - half, half - c), r.uniform(0.5, 1.0)
        for k in range(0, len(thetas), step):
            t = th[k:k + step]
            s2 = (a * torch.cos(t - phi)) ** 2 + (b * torch.sin(t - phi)) ** 2
            u0 = rad * torch.cos(ang - t)
            q = 1.0 - (u - u0.float()) ** 2 / s2.float() - ((z - z0) / c) ** 2
            out[k:k + step] += (2 * rho * a * b / s2.sqrt()).float() * q.clamp_(min=0.0).sqrt_()
    return out


def _object(n, n_p, seed, photons=1e6, start=0):
    """Patterns (centred), supports, a mid-run iterate and the angles of one seeded object."""
    dev, th = _device(), _thetas(n_p)
    P = _projections(n, th, seed, dev)
    gen = torch.Generator(device=dev).manual_seed(1000 * seed + 7 + start)
    I = torch.empty_like(P)
    step = max(1, (64 << 20) // (n * n))
    for k in range(0, n_p, step):
        I[k:k + step] = torch.fft.fftshift(torch.fft.fft2(P[k:k + step]), dim=(-2, -1)).abs().square()
    if photons:
        scale = photons / float(I.mean(dtype=torch.float64) * (n * n))
        I *= scale
        P *= math.sqrt(scale)
        g = torch.Generator(device=dev).manual_seed(1000 * seed + 3)
        for k in range(0, n_p, step):
            I[k:k + step] = torch.poisson(I[k:k + step], generator=g)
    S = torch.empty((n_p, n, n), dtype=torch.uint8, device=dev)
    for k in range(0, n_p, step):
        S[k:k + step] = torch.nn.functional.max_pool2d((P[k:k + step] > 0).float(), 5, 1, 2) > 0
    rms = float(P.square().mean(dtype=torch.float64).sqrt())
    noise = torch.empty_like(P).normal_(generator=gen)
    g0 = P.add_(noise, alpha=0.2 * rms).mul_(S)
    return I, S, g0, th


def _stop_mask(n, radius):
    dev = _device()
    k = torch.arange(n, device=dev) - n // 2
    return ((k[:, None] ** 2 + k[None, :] ** 2) > radius * radius).to(torch.uint8)


def _config(case, n, n_p, **kw):
    raar = case["update"] == "raar"
    return cp.make_config(n, n_p, n_ei=case["n_ei"], beta=0.9, update=cp.UPDATE_RAAR if raar else cp.UPDATE_HIO,
                          hio_iters=1 << 30 if raar else 0, er_iters=0 if raar else 1 << 30,
                          wrap_mode=cp.WRAP_MIRROR if case.get("mirror") else cp.WRAP_LITERAL,
                          blend_target=cp.BLEND_OBJECT if case.get("blend_object") else cp.BLEND_STATE, **kw)


def _loaded(cfg, I, S, g0, th, mask=None):
    """A plan with its patterns, supports and a mid-run iterate (a resumed reconstruction)."""
    plan = cp.Plan(cfg)
    if mask is not None:
        plan.load_mask(mask)
    plan.load_intensities(I, 0, th)
    plan.load_support(S)
    if g0 is not None:
        plan.load_state(g0, 0)
    return plan


def _seeds(case, seed):
    return [seed * 16 + i for i in range(len(case["sizes"].split(",")))]


def _sizes(case):
    return [tuple(int(v) for v in s.split("x")) for s in case["sizes"].split(",")]


def prepare(case, seed):
    kind, dev = case["kind"], _device()
    if kind == "iterate":
        n, n_p = case["N"], case["Np"]
        I, S, g0, th = _object(n, n_p, seed, case.get("photons", 1e6))
        mask = _stop_mask(n, case["stop"]) if case.get("stop") else None
        plan = _loaded(_config(case, n, n_p), I, S, g0, th, mask)
        return dict(case=case, plan=plan, out=torch.empty((n_p, n, n), device=dev))
    if kind == "batch":
        plans, outs = [], []
        for (n, n_p), s in zip(_sizes(case), _seeds(case, seed)):
            plans.append(_loaded(_config(case, n, n_p), *_object(n, n_p, s)))
            outs.append(torch.empty((n_p, n, n), device=dev))
        return dict(case=case, plans=plans, batch=cp.Batch(plans), out=outs)
    if kind == "sweep":
        n, n_p = case["N"], case["Np"]
        plans, outs = [], []
        for i in range(case["guesses"]):
            plans.append(_loaded(_config(case, n, n_p, sweep=1), *_object(n, n_p, seed, start=i)))
            outs.append(torch.empty((n_p, n, n), device=dev))
        return dict(case=case, plans=plans, batch=cp.Batch(plans), out=outs)
    if kind == "reconstruct":
        n, n_p = case["N"], case["Np"]
        I, S, _, th = _object(n, n_p, seed)
        plan = _loaded(_config(case, n, n_p, seed=seed), I, S, None, th)
        return dict(case=case, plan=plan, I=I, th=th, out=torch.empty((n_p, n, n), device=dev),
                    vol=torch.empty((n, n, n), dtype=torch.complex64, device=dev))
    if kind in ("assemble", "refine"):
        n, n_p = case["N"], case["Np"]
        plan = _loaded(cp.make_config(n, n_p), *_object(n, n_p, seed))
        return dict(case=case, plan=plan, vol=torch.empty((n, n, n), dtype=torch.complex64, device=dev))
    if kind == "merge":
        n, n_p = case["N"], case["Np"]
        plans = []
        for I, S, g0, th in _guesses(case, seed):
            p = _loaded(cp.make_config(n, n_p, hio_iters=0), I, S, g0, th)
            p.iterate(1)
            plans.append(p)
        dst = cp.Plan(cp.make_config(n, n_p))
        return dict(case=case, plans=plans, dst=dst, prtf=torch.empty((n_p, n // 2), device=dev),
                    vol=torch.empty((n, n, n), dtype=torch.complex64, device=dev),
                    E=torch.empty((n_p, n, n), dtype=torch.complex64, device=dev))
    n, c = case["N"], case["count"]
    _, S, g0, _ = _object(n, c, seed)
    return dict(case=case, g=g0, S=S, out=torch.empty_like(S))


def _guesses(case, seed):
    """Guesses of rising noise, every second one centrally inverted (the twin)."""
    n, n_p = case["N"], case["Np"]
    for i in range(case["guesses"]):
        I, S, g0, th = _object(n, n_p, seed, start=i)
        g0 = g0 * (1.0 + 0.02 * i * torch.sin(torch.arange(n, device=g0.device) * (0.1 + 0.01 * i)))
        if i % 2:
            g0 = torch.roll(torch.flip(g0, (1, 2)), (1, 1), (1, 2)).contiguous()
            S = torch.roll(torch.flip(S, (1, 2)), (1, 1), (1, 2)).contiguous()
        yield I, S, g0, th


# ------------------------------------------------------------------ one call
def _state_of(plan, out):
    cp.cpra_result(plan.h, cp.RESULT_STATE, out, out.numel() * 4)
    return out


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "iterate":
        state["plan"].iterate(case["iters"])
        return _state_of(state["plan"], state["out"])
    if kind in ("batch", "sweep"):
        state["batch"].iterate(case["iters"])
        return [_state_of(p, o) for p, o in zip(state["plans"], state["out"])]
    plan = state.get("plan")
    if kind == "reconstruct":
        plan.reset()
        plan.load_intensities(state["I"], 0, state["th"])
        plan.iterate(case["iters"])
        plan.assemble_3d(state["vol"])
        return [_state_of(plan, state["out"]), state["vol"]]
    if kind == "assemble":
        plan.assemble_3d(state["vol"])
        return state["vol"]
    if kind == "refine":
        plan.assemble_3d()
        plan.refine_3d(case["iters"])
        cp.cpra_result(plan.h, cp.RESULT_VOLUME, state["vol"], state["vol"].numel() * 8)
        return state["vol"]
    if kind == "merge":
        sel, inv = cp.cpra_merge(state["plans"], case["keep"], 0, state["dst"], state["prtf"])
        cp.cpra_result(state["dst"].h, cp.RESULT_VOLUME, state["vol"], state["vol"].numel() * 8)
        cp.cpra_result(state["dst"].h, cp.RESULT_MERGED_SPECTRA, state["E"], state["E"].numel() * 8)
        return dict(selected=np.array(sel), inverted=np.array(inv), prtf=state["prtf"], volume=state["vol"], spectra=state["E"])
    cp.cpra_shrinkwrap_static(state["g"], state["S"], state["out"], case["N"], case["count"], 2.0, 0.1,
                              torch.cuda.current_stream().cuda_stream)
    return state["out"]


# ------------------------------------------------------------------ what a call cannot do without
def _iter_work(n, n_p, iters):
    """An angle's iteration: the iterate read and written, the amplitudes of the half plane and the support read; its 2D FFT pair."""
    return n_p * iters * (8 * n * n + 4 * n * (n // 2 + 1) + n * n // 8), n_p * iters * (10.0 * n * n * math.log2(n) + 20.0 * n * n)


def _volume_work(n, n_p):
    """Projected objects read, the volume written; the spectra's and the volume's FFTs, gridding of four cells a sample and plane."""
    return 4 * n_p * n * n + 8 * n ** 3, 2.5 * n_p * n * n * 2 * math.log2(n) + 5.0 * n ** 3 * 3 * math.log2(n) + 16.0 * n_p * n * n


def work(case):
    kind = case["kind"]
    if kind == "batch":
        parts = [_iter_work(n, n_p, case["iters"]) for n, n_p in _sizes(case)]
        return dict(bytes=sum(p[0] for p in parts), flops=sum(p[1] for p in parts))
    if kind == "support":
        px = case["N"] ** 2 * case["count"]
        return dict(bytes=px * 6, flops=px * 4 * 29)
    n, n_p = case["N"], case["Np"]
    if kind == "iterate":
        b, f = _iter_work(n, n_p, case["iters"])
    elif kind == "sweep":
        b, f = _iter_work(n, n_p * case["guesses"], case["iters"])
    elif kind == "reconstruct":
        (b, f), (vb, vf) = _iter_work(n, n_p, case["iters"]), _volume_work(n, n_p)
        b, f = b + vb + 4 * n_p * n * n, f + vf
    elif kind == "assemble":
        b, f = _volume_work(n, n_p)
    elif kind == "refine":
        b, f = _volume_work(n, n_p)
        # an iteration: the real iterate read and written, the data's half spectrum read; a real 3D FFT pair
        b, f = b + case["iters"] * 12 * n ** 3, f + case["iters"] * 15.0 * n ** 3 * math.log2(n)
    else:
        b, f = _volume_work(n, n_p * case["keep"])
        b -= 8 * n ** 3 * (0 if case["keep"] == 1 else 1) - 8 * n ** 3  # one volume, whatever the number kept
        b, f = b + 8 * n_p * n * n, f
    return dict(bytes=int(b), flops=float(f))


# ------------------------------------------------------------------ the same in 64 bits
def _amplitudes(I, mask):
    """sqrt(I) in FFT order (float64) and where a pixel and its partner -k were both measured (None: everywhere)."""
    A = torch.fft.ifftshift(I.double(), dim=(-2, -1)).sqrt()
    if mask is None:
        return A, None
    m = torch.fft.ifftshift(mask.bool(), dim=(-2, -1))
    return A, m & torch.roll(torch.flip(m, (-2, -1)), (1, 1), (-2, -1))


def _step64(g, A, free, S, update, beta=0.9):
    """One iteration of a stack of iterates."""
    G = torch.fft.fft2(g)
    mag = G.abs()
    one = torch.ones((), dtype=G.dtype, device=G.device)
    M = A * torch.where(mag > 0, G / torch.where(mag > 0, mag, 1.0), one)
    if free is not None:
        # a free pair keeps G; the constrained ones enter symmetrised, as the real part does
        Asym = 0.5 * (A + torch.roll(torch.flip(A, (-2, -1)), (1, 1), (-2, -1)))
        M = torch.where(free, Asym * torch.where(mag > 0, G / torch.where(mag > 0, mag, 1.0), one), G)
    gp = torch.fft.ifft2(M).real
    if update == "er":
        return torch.where(S & (gp >= 0), gp, 0.0)
    return torch.where(S & (2 * gp - g >= 0), gp, beta * g + (1 - 2 * beta) * gp)


def _neighbours(case, n, n_p):
    """(angle, mirrored, weight) of Eq. 4 for angle n."""
    for k, a in zip((-1, 0, 1), (0.2, 0.6, 0.2)):
        j = n + k
        yield j % n_p, bool(case.get("mirror")) and (j // n_p) % 2 != 0, float(np.float32(a))


def _coupled(case, n, n_p, image):
    out = 0.0
    for j, mir, a in _neighbours(case, n, n_p):
        v = image(j)
        out = out + a * (torch.roll(torch.flip(v, (-1,)), 1, -1) if mir else v)
    return out


def _pos(g, S):
    return torch.where(S & (g >= 0), g, torch.zeros((), dtype=g.dtype, device=g.device))


def _iterate64(case, I, S, g, mask=None):
    n_p, n = I.shape[0], I.shape[-1]
    S, step = S.bool(), max(1, (8 << 20) // (n * n))
    g = g.double()
    for it in range(case["iters"]):
        if it % case["n_ei"] == 0:
            src = _pos(g, S) if case.get("blend_object") else g
            new = torch.empty_like(g)
            for k in range(n_p):
                new[k] = _coupled(case, k, n_p, lambda j: src[j])
            g = new
        for k in range(0, n_p, step):
            A, free = _amplitudes(I[k:k + step], mask)
            g[k:k + step] = _step64(g[k:k + step], A, free, S[k:k + step], case["update"])
    return g


def _spectrum64(rho):
    """DFT2 of a projected object with its mass centre moved to the origin, FFT order."""
    n = rho.shape[-1]
    x = torch.arange(n, dtype=torch.float64, device=rho.device)
    m = rho.sum()
    cz, cu = ((rho.sum(1) * x).sum() / m, (rho.sum(0) * x).sum() / m) if float(m) > 0 else (x.new_tensor(n / 2), x.new_tensor(n / 2))
    k = torch.fft.fftfreq(n, dtype=torch.float64, device=rho.device)
    ramp = 2 * math.pi * (k[:, None] * cz + k[None, :] * cu)
    return torch.fft.fft2(rho) * torch.polar(torch.ones_like(ramp), ramp)


def _volume64(spectrum, n, th, dev):
    """Gridding of the spectra (bilinear in kx, ky, normalised weights) and the inverse 3D FFT, centred; the reached cells."""
    num = torch.zeros((n * n, n), dtype=torch.complex128, device=dev)
    den = torch.zeros(n * n, dtype=torch.float64, device=dev)
    ku = np.where(np.arange(n) < n // 2, np.arange(n), np.arange(n) - n).astype(np.float64)
    for i, t in enumerate(th):
        F = torch.fft.fftshift(torch.fft.ifft(spectrum(i), dim=0), dim=0).T.contiguous()  # [ku][z]
        px, py = ku * math.cos(t), ku * math.sin(t)
        i0, j0 = np.floor(px), np.floor(py)
        for di in (0, 1):
            for dj in (0, 1):
                w = np.abs(1 - di - (px - i0)) * np.abs(1 - dj - (py - j0))
                cell = ((j0.astype(int) + dj) % n) * n + (i0.astype(int) + di) % n
                at, wt = torch.from_numpy(cell).to(dev), torch.from_numpy(w).to(dev)
                num.index_add_(0, at, F * wt[:, None])
                den.index_add_(0, at, wt)
    got = den >= 1e-12
    num = torch.where(got[:, None], num / torch.where(got, den, 1.0)[:, None], 0.0)
    sign = (1 - 2 * (torch.arange(n, device=dev) % 2)).double()
    grid = num.T.reshape(n, n, n) * (sign[:, None] * sign[None, :])
    del num
    for z in range(n):
        grid[z] = torch.fft.ifft2(grid[z])
    return grid, got.reshape(n, n)


def _refined64(vol, M, S, g, th, iters):
    n, dev = vol.shape[0], vol.device
    sh = lambda v, f: f(v, dim=(0, 1, 2))  # noqa: E731
    V = torch.fft.fftn(vol)
    c = n // 2
    x = torch.arange(n, dtype=torch.float64, device=dev) - c
    S3 = torch.ones((n, n, n), dtype=torch.bool, device=dev)
    for i, t in enumerate(th):
        rho = _pos(g[i], S[i])
        m, p = rho.sum(), x + c
        dz, du = (int(np.rint(float((rho.sum(a) * p).sum() / m) - c)) for a in (1, 0)) if float(m) > 0 else (0, 0)
        u = torch.round((x[None, :] * math.cos(t) + x[:, None] * math.sin(t)) + c).long()  # [y][x]
        inside = (u >= 0) & (u < n)
        rows = torch.roll(S[i], (-dz, -du), (0, 1))  # S at (z + dz, u + du)
        S3 &= rows[:, u.clamp(0, n - 1)] & inside
    rho = vol.real.clone()
    for _ in range(iters):
        X = torch.fft.fftn(torch.where(S3 & (rho >= 0), rho, 0.0))
        X = torch.where(M[None], V, X)
        rho = torch.fft.ifftn(X).real
    return torch.where(S3 & (rho >= 0), rho, 0.0).to(torch.complex128)


def _seeded_start(n, n_p, seed, dev):
    """The library's documented start: SplitMix64 of the pixel's key, 24 bits."""
    key = np.arange(n_p * n * n, dtype=np.uint64) + np.uint64((seed * n_p * n * n) & (2 ** 64 - 1))
    with np.errstate(over="ignore"):
        z = key + np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        z = z ^ (z >> np.uint64(31))
    u = (z >> np.uint64(40)).astype(np.float64) * 2.0 ** -24
    return torch.from_numpy(u.reshape(n_p, n, n)).to(dev)


def exact(case, seed):
    kind, dev = case["kind"], _device()
    if kind == "support":
        return None  # decisions, not computed numbers
    if kind == "batch":
        return [_iterate64(case, *_object(n, n_p, s)[:3]) for (n, n_p), s in zip(_sizes(case), _seeds(case, seed))]
    n, n_p = case["N"], case["Np"]
    if kind == "iterate":
        I, S, g0, _ = _object(n, n_p, seed, case.get("photons", 1e6))
        return _iterate64(case, I, S, g0, _stop_mask(n, case["stop"]) if case.get("stop") else None)
    if kind == "sweep":
        objs = [_object(n, n_p, seed, start=i) for i in range(case["guesses"])]
        I, S = objs[0][0], objs[0][1].bool()
        g = torch.stack([o[2].double() for o in objs], 1)  # [Np][guess]
        for _ in range(case["iters"] // case["n_ei"]):
            for k in range(n_p):
                v = _coupled(case, k, n_p, lambda j: g[j])
                A, _ = _amplitudes(I[k], None)
                for _ in range(case["n_ei"]):
                    v = _step64(v, A, None, S[k], case["update"])
                g[k] = v
        return [g[:, i].contiguous() for i in range(case["guesses"])]
    if kind == "reconstruct":
        I, S, _, th = _object(n, n_p, seed)
        g = _iterate64(case, I, S, _seeded_start(n, n_p, seed, dev) * S)
        rho = _pos(g, S.bool())
        return [g, _volume64(lambda i: _spectrum64(rho[i]), n, th, dev)[0]]
    if kind in ("assemble", "refine"):
        _, S, g, th = _object(n, n_p, seed)
        S, g = S.bool(), g.double()
        vol, M = _volume64(lambda i: _spectrum64(_pos(g[i], S[i])), n, th, dev)
        return vol if kind == "assemble" else _refined64(vol, M, S, g, th, case["iters"])
    rhos, errs = [], []
    one = dict(iters=1, n_ei=10, update="er")
    for I, S, g0, th in _guesses(case, seed):
        A, _ = _amplitudes(I, None)
        start = torch.stack([_coupled(one, k, n_p, lambda j: g0[j].double()) for k in range(n_p)])
        errs.append(float((((torch.fft.fft2(start).abs() - A) ** 2).sum((1, 2)) / (A ** 2).sum((1, 2))).sqrt().mean()))
        rhos.append(_pos(_iterate64(one, I, S, g0), S.bool()))
    order = list(np.argsort(errs, kind="stable")[:case["keep"]])
    ref = _spectrum64(rhos[order[0]][0])
    inv = []
    for k, i in enumerate(order):
        E = _spectrum64(rhos[i][0])
        inv.append(bool(k > 0 and float((ref - E.conj()).abs().square().sum()) < float((ref - E).abs().square().sum())))
    mean = torch.empty((n_p, n, n), dtype=torch.complex128, device=dev)
    prtf = torch.empty((n_p, n // 2), dtype=torch.float64, device=dev)
    kf = torch.fft.fftfreq(n, 1.0 / n, dtype=torch.float64, device=dev)
    ring = torch.round((kf[:, None] ** 2 + kf[None, :] ** 2).sqrt()).long().clamp(max=n // 2).reshape(-1)
    cnt = torch.bincount(ring, minlength=n // 2 + 1).double()
    for p in range(n_p):
        E = [_spectrum64(rhos[i][p]) for i in order]
        E = torch.stack([e.conj() if f else e for e, f in zip(E, inv)])
        mean[p] = E.mean(0)
        mag = E.abs().sum(0)
        r = torch.where(mag > 0, E.sum(0).abs() / torch.where(mag > 0, mag, 1.0), 0.0).reshape(-1)
        prtf[p] = (torch.zeros_like(cnt).index_add_(0, ring, r) / cnt.clamp(min=1))[:n // 2]
    vol, _ = _volume64(lambda i: mean[i], n, th, dev)
    return dict(selected=None, inverted=None, prtf=prtf, volume=vol, spectra=mean)
