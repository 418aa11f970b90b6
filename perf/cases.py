"""The work that users have this library do, as cases that can be timed and checked.

listed() gives the cases, draw() further ones of the same ranges, prepare() what a
program has in hand before the call, run() one pass through the public entry points of
paper_1702_08852_gb300.wf, work() what the pass cannot do without, and exact() the same
outputs in 64 bits from plain torch.

Every case is one of six kinds ("op"):
  sht    alm2map of one set of coefficients and map2alm of one map, the transform pair of
         an iteration, in the precision "prec" (f64, f32 or df64);
  group  the same pair for several maps of one geometry through the grouped calls;
  solve  a Wiener-filter solve to the default tolerance, plain FP64 or mixed;
  batch  several independent mixed solves in one wf_solve_batch call;
  flat   the solver on an n x n flat grid;
  train  one loss-and-gradient call of the warm-start network.
The transforms f32 and group and the mixed solves work in single precision (their error is
that of FP32, or of a solve to 1e-6), so a program keeps their maps and coefficients in
single precision, the type in which HEALPix maps are written to disk; run() does so too.
"""
import math

import numpy as np
import torch

from paper_1702_08852_gb300 import inputs, wf

DEV = "cuda"


# ------------------------------------------------------------------------- the cases
def listed():
    return [
        # the README's smallest workload as single calls: latency and launches
        dict(name="sht_f64_n32", op="sht", prec="f64", nside=32, lmax=64),
        # a ragged geometry: Nside not a power of two, odd lmax above 2 Nside
        dict(name="sht_f64_n150", op="sht", prec="f64", nside=150, lmax=311),
        # the flagship geometry (the benchmark's Nside 1024, lmax 2048) in plain FP64
        dict(name="sht_f64_n1024", op="sht", prec="f64", nside=1024, lmax=2048),
        # the FP32 transforms of the mixed solver, at its Nside 256 workload's geometry
        dict(name="sht_f32_n256", op="sht", prec="f32", nside=256, lmax=512),
        # and at a small ragged one
        dict(name="sht_f32_n90", op="sht", prec="f32", nside=90, lmax=199),
        # the double-float transforms of the mixed solver's anchors
        dict(name="sht_df64_n512", op="sht", prec="df64", nside=512, lmax=1024),
        # a simulation campaign: 64 maps of one geometry (the benchmark's grouped workload)
        dict(name="group_n256_x64", op="group", nside=256, lmax=512, nmaps=64),
        # the plain FP64 solver at Nside 32: thousands of short iterations
        dict(name="solve_f64_n32", op="solve", prec="f64", nside=32, lmax=64, noise="lognormal"),
        # the mixed solver on the Nside 256 scan workload, launch variants autotuned
        dict(name="solve_mixed_n256", op="solve", prec="mixed", nside=256, lmax=512, noise="scan"),
        # uneven maps solved together, as the benchmark's batch workload does with 64
        dict(name="batch_x6", op="batch", nsides="64,64,128,64,128,64"),
        # the paper's own flat-sky set-up
        dict(name="flat_n256", op="flat", n=256),
        # a training step of the warm-start network at Nside 256 (default sizes)
        dict(name="train_n256", op="train", nside=256, lmax=512, channels=16, kernel=9, hidden=32),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["sht", "sht", "sht", "sht", "group", "solve", "solve", "batch", "flat", "train"])
    if op == "sht":
        prec = rng.choice(["f64", "f32", "df64"])
        nside = _log_int(rng, 8, {"f64": 800, "f32": 256, "df64": 512}[prec])
        lmax = max(2, min(3 * nside - 1, int(nside * rng.uniform(1.5, 2.2))))
        return dict(op=op, prec=prec, nside=nside, lmax=lmax)
    if op == "group":
        nside = _log_int(rng, 16, 200)
        return dict(op=op, nside=nside, lmax=int(nside * rng.uniform(1.5, 2.2)), nmaps=_log_int(rng, 3, 64))
    if op == "solve":
        prec = rng.choice(["f64", "mixed"])
        nside = _log_int(rng, 12, 40) if prec == "f64" else _log_int(rng, 24, 200)
        return dict(op=op, prec=prec, nside=nside, lmax=2 * nside, noise=rng.choice(["lognormal", "scan"]))
    if op == "batch":
        return dict(op=op, nsides=",".join(str(rng.choice([32, 48, 64, 96])) for _ in range(rng.randint(2, 6))))
    if op == "flat":
        return dict(op=op, n=rng.choice([64, 128, 256]))
    nside = _log_int(rng, 32, 256)
    return dict(op=op, nside=nside, lmax=2 * nside, channels=rng.choice([8, 12, 16]), kernel=rng.choice([5, 7, 9]), hidden=rng.choice([16, 32]))


# ------------------------------------------------------------------------- the inputs
def _rng(case, seed):
    return np.random.default_rng([int(seed)] + [int(v) for v in case.values() if isinstance(v, int)])


def _noise_map(gen, nside, count):
    """Maps of scan-modulated white noise with the galactic band masked to 0."""
    z, phi = inputs.pixel_centres(nside)
    sig = np.where(np.abs(z) < 0.2, 0.0, 1.0 + 0.5 * np.abs(z) * np.cos(phi))
    m = torch.randn(count, 12 * nside * nside, dtype=torch.float64, device=DEV, generator=gen)
    return m * torch.from_numpy(sig).to(DEV)


def _alms(gen, nside, lmax, count):
    """Gaussian coefficients of the workloads' spectrum, m-major."""
    cl = torch.from_numpy(inputs.cl_spectrum(lmax, nside)).to(DEV)
    ls, ms = (torch.from_numpy(v).to(DEV) for v in inputs.lm_of_slots(lmax))
    a = torch.randn(count, len(ls), 2, dtype=torch.float64, device=DEV, generator=gen)
    scale = torch.sqrt(cl[ls] / torch.where(ms == 0, 1.0, 2.0))
    a[:, ms == 0, 1] = 0.0
    return torch.view_as_complex(a * scale[:, None]).contiguous()


def _sht_inputs(case, seed):
    gen = torch.Generator(DEV).manual_seed(1000003 * int(seed) + case["nside"])
    n = case.get("nmaps", 1)
    return _alms(gen, case["nside"], case["lmax"], n), _noise_map(gen, case["nside"], n)


def _problem(nside, lmax, noise, seed, **kw):
    """The workloads' problems: scan noise with a quarter of the sky masked, or lognormal."""
    if noise == "scan":
        p = inputs.scan_problem(nside, lmax, seed=seed, discs=kw.pop("discs", min(500, 2 * nside)), **kw)
    else:
        p = inputs.lognormal_problem(nside, lmax, seed=seed, **kw)
    a = torch.from_numpy(p.alm_true).to(DEV)[None]
    signal = _synthesis(a, nside, lmax)[0].cpu().numpy()
    return p, torch.from_numpy(p.data(signal)).to(DEV)


def _plan_of(p, **opts):
    nv = torch.from_numpy(p.noise_var).to(DEV)
    mk = torch.from_numpy(p.mask.astype(np.uint8)).to(DEV)
    return wf.wf_plan(p.nside, p.lmax, p.cl, nv, mk, **opts)


def _batch_problems(case, seed):
    rng = _rng(case, seed)
    out = []
    for i, ns in enumerate(int(v) for v in case["nsides"].split(",")):
        out.append(_problem(ns, 2 * ns, "scan", 100 * int(seed) + i, mask_fraction=float(rng.uniform(0.1, 0.4)),
                            discs=int(rng.integers(0, 60)), amplitude=float(rng.uniform(0.5, 2.0))))
    return out


def _flat_inputs(case, seed):
    n, side = case["n"], math.radians(10.0)
    rng = _rng(case, seed)
    ck = inputs.flat_cl(inputs.flat_mode_ell(n, side))
    area = (side / n) ** 2
    nv, mask = inputs.flat_paper_noise(n)
    d = inputs.flat_gaussian_field(rng, ck, area) + np.sqrt(nv) * rng.standard_normal((n, n))
    return ck, area, torch.from_numpy(nv).to(DEV), torch.from_numpy(np.where(mask, 0.0, d)).to(DEV)


def _train_inputs(case, seed):
    """A problem, a target (its true coefficients, damped) and the weights of a net in mid-training."""
    p, d = _problem(case["nside"], case["lmax"], "scan", int(seed))
    rng = _rng(case, seed)
    H, K, M = case["channels"], case["kernel"], case["hidden"]
    sizes = [(H * 3 * K, 3 * K), (H, 0), (H * H * K, H * K), (H, 0), (H * K, H * K), (1, 0),
             (M * 4, 4), (M, 0), (M * M, M), (M, 0), (M, M), (1, 0)]
    theta = np.concatenate([math.sqrt(1.0 / f) * rng.standard_normal(n) if f else 0.1 * rng.standard_normal(n)
                            for n, f in sizes]).astype(np.float32)
    return p, d, torch.from_numpy(0.8 * p.alm_true).to(DEV), theta


def prepare(case, seed):
    op = case["op"]
    s = {"case": case}
    if op in ("sht", "group"):
        alm, maps = _sht_inputs(case, seed)
        s["plan"] = wf.wf_plan(case["nside"], case["lmax"], inputs.cl_spectrum(case["lmax"], case["nside"]))
        s["alm"], s["map"] = (alm, maps) if op == "group" else (alm[0], maps[0])
    elif op == "solve":
        p, s["d"] = _problem(case["nside"], case["lmax"], case["noise"], int(seed))
        mixed = case["prec"] == "mixed"
        s["plan"] = _plan_of(p, precision=wf.WF_PREC_MIXED, autotune=1) if mixed else _plan_of(p)
    elif op == "batch":
        probs = _batch_problems(case, seed)
        s["plans"] = [_plan_of(p, precision=wf.WF_PREC_MIXED, autotune=1) for p, _ in probs]
        s["ds"] = [d for _, d in probs]
    elif op == "flat":
        ck, area, nv, s["d"] = _flat_inputs(case, seed)
        s["plan"] = wf.FlatPlan(case["n"], area, ck, nv)
    else:
        p, s["d"], s["target"], theta = _train_inputs(case, seed)
        s["plan"] = _plan_of(p)
        s["net"] = wf.Net(s["plan"], case["channels"], case["kernel"], case["hidden"])
        s["net"].set_params(theta)
    return s


def run(s):
    op = s["case"]["op"]
    if op == "sht":
        prec = s["case"]["prec"]
        if prec == "f64":
            return {"map": wf.wf_alm2map(s["plan"], s["alm"]), "alm": wf.wf_map2alm(s["plan"], s["map"])}
        if prec == "df64":
            return {"map": wf.wf_alm2map_df64(s["plan"], s["alm"]), "alm": wf.wf_map2alm_df64(s["plan"], s["map"])}
        m, a = wf.wf_alm2map_f32(s["plan"], s["alm"]), wf.wf_map2alm_f32(s["plan"], s["map"])
        return {"map": m.to(torch.float32), "alm": a.to(torch.complex64)}
    if op == "group":
        m, a = wf.wf_alm2map_group(s["plan"], s["alm"]), wf.wf_map2alm_group(s["plan"], s["map"])
        return {"map": m.to(torch.float32), "alm": a.to(torch.complex64)}
    if op == "solve":
        alm, m, _ = wf.wf_solve(s["plan"], s["d"])
        if s["case"]["prec"] == "f64":
            return {"alm": alm, "map": m}
        return {"alm": alm.to(torch.complex64), "map": m.to(torch.float32)}
    if op == "batch":
        alms, _, _, _ = wf.wf_solve_batch(s["plans"], s["ds"])
        return [a.to(torch.complex64) for a in alms]
    if op == "flat":
        return s["plan"].solve(s["d"])[0]
    loss, grad = s["net"].loss_grad(s["d"], s["target"], want_grad=True)
    return {"loss": loss, "grad": grad}


# ------------------------------------------------------------------------- the work
#: Iterations that a solve to the default tolerance takes, about (it depends on the data).
ITERATIONS = {"f64": 6500, "mixed": 4200, "batch": 4200, "flat": 12000}


def _pair_flops(nside, lmax):
    """One synthesis and one analysis: a complex multiply-add with each of the ~3/4 of the
    Legendre values that are not negligible and one multiply-add to make it, and a real FFT
    of every ring."""
    npix, nalm = 12 * nside * nside, (lmax + 1) * (lmax + 2) // 2
    return 2 * (0.75 * 6.0 * nalm * 2 * nside + 2.5 * npix * math.log2(4 * nside + 1))


def work(case):
    op = case["op"]
    if op == "flat":
        n2 = case["n"] ** 2
        return {"bytes": 8.0 * 2 * n2, "flops": ITERATIONS["flat"] * (2 * 2.5 * n2 * math.log2(n2) + 12.0 * n2)}
    if op == "batch":
        nsides = [int(v) for v in case["nsides"].split(",")]
        return {"bytes": sum(8.0 * 12 * n * n + 16.0 * (2 * n + 1) * (n + 1) for n in nsides),
                "flops": ITERATIONS["batch"] * sum(_pair_flops(n, 2 * n) for n in nsides)}
    nside, lmax = case["nside"], case["lmax"]
    npix, nalm = 12.0 * nside * nside, (lmax + 1) * (lmax + 2) / 2.0
    if op in ("sht", "group"):
        count = case.get("nmaps", 1)
        # in FP64 (8 and 16 bytes), out in the precision that is kept
        kept = 1.0 if op == "sht" and case["prec"] != "f32" else 0.5
        return {"bytes": count * (16 * nalm + 8 * npix) * (1.0 + kept), "flops": count * _pair_flops(nside, lmax)}
    if op == "solve":
        kept = 1.0 if case["prec"] == "f64" else 0.5
        return {"bytes": 8 * npix + kept * (16 * nalm + 8 * npix), "flops": ITERATIONS[case["prec"]] * _pair_flops(nside, lmax)}
    H, K = case["channels"], case["kernel"]
    conv = 2.0 * K * (3 * H + H * H + H) * npix
    return {"bytes": 8 * npix + 16 * nalm, "flops": 3 * conv + 1.5 * _pair_flops(nside, lmax)}


# ------------------------------------------------------------------------- 64-bit values
def _pairs(nside):
    """z, sin theta, pixels, phi0 of the north ring of every pair, and the first pixels of
    its north and south ring (-1: the equator has none)."""
    out = []
    npix, ofs = 12 * nside * nside, 0
    for r in range(1, 2 * nside + 1):
        if r < nside:
            omz, n = r * r / (3.0 * nside * nside), 4 * r
            z, p0 = 1.0 - omz, math.pi / n
            st = math.sqrt(omz * (2.0 - omz))
        else:
            z, n = 2.0 * (2 * nside - r) / (3.0 * nside), 4 * nside
            st = math.sqrt((1.0 - z) * (1.0 + z))
            p0 = 0.0 if (r + nside) % 2 else math.pi / n
        out.append((z, st, n, p0, ofs, npix - ofs - n if r < 2 * nside else -1))
        ofs += n
    return out


def _legendre(nside, lmax):
    """Yields l and lam_lm(z) of the north rings, [l + 1, pairs], for l = 0 .. lmax: the
    three-term recurrence with a power-of-two scale for each value (0 where below 2^-150)."""
    pr = _pairs(nside)
    z = torch.tensor([p[0] for p in pr], dtype=torch.float64, device=DEV)
    st = torch.tensor([p[1] for p in pr], dtype=torch.float64, device=DEV)
    K, m = len(pr), torch.arange(lmax + 1, dtype=torch.float64, device=DEV)
    start, scale = [], []
    v, e = torch.full_like(z, 1.0 / math.sqrt(4.0 * math.pi)), torch.zeros_like(z)
    for k in range(lmax + 1):
        if k:
            v = -v * st * math.sqrt((2.0 * k + 1.0) / (2.0 * k))
            low = v.abs() < 2.0 ** -300
            v, e = torch.where(low, v * 2.0 ** 300, v), torch.where(low, e - 1, e)
        start.append(v)
        scale.append(e)
    cur, prev = torch.stack(start), torch.zeros(lmax + 1, K, dtype=torch.float64, device=DEV)
    exp = torch.stack(scale)
    one = torch.ones((), dtype=torch.float64, device=DEV)
    down = one * 2.0 ** -300
    for l in range(lmax + 1):
        if l:
            mm = m[:l]
            a = torch.sqrt((4.0 * l * l - 1.0) / (l * l - mm * mm))
            b = torch.where(mm == l - 1, torch.zeros_like(mm), torch.sqrt(((l - 1.0) ** 2 - mm * mm).clamp(min=0) / (4.0 * (l - 1.0) ** 2 - 1.0)))
            new = (z * cur[:l] - b[:, None] * prev[:l]) * a[:, None]
            prev[:l] = cur[:l]
            cur[:l] = new
            if l % 4 == 0:
                grown = (cur[:l].abs() > 2.0 ** 100) & (exp[:l] < 0)
                f = torch.where(grown, down, one)
                cur[:l] *= f
                prev[:l] *= f
                exp[:l] += grown
        yield l, torch.where(exp[:l + 1] == 0, cur[:l + 1], 0.0 * one)


def _slot(lmax, l):
    m = torch.arange(l + 1, device=DEV)
    return m * (2 * lmax + 1 - m) // 2 + l


def _ring_groups(nside):
    """Rings with the same number of pixels: (n, [(ring rows: pair, north?, phi0, first pixel)])."""
    by = {}
    for k, (_, _, n, p0, on, os_) in enumerate(_pairs(nside)):
        by.setdefault(n, []).append((k, 0, p0, on))
        if os_ >= 0:
            by[n].append((k, 1, p0, os_))
    return by


def _phase(rows, lmax):
    p0 = torch.tensor([r[2] for r in rows], dtype=torch.float64, device=DEV)
    ang = p0[:, None] * torch.arange(lmax + 1, dtype=torch.float64, device=DEV)
    return torch.polar(torch.ones_like(ang), ang)


def _synthesis(alm, nside, lmax):
    """Maps [B, npix] of coefficients [B, nalm] (m-major), all in FP64."""
    B, K = alm.shape[0], 2 * nside
    par = torch.zeros(2, B, lmax + 1, K, dtype=torch.complex128, device=DEV)
    for l, lam in _legendre(nside, lmax):
        a = alm[:, _slot(lmax, l)]
        for q in (0, 1):  # rows with (l - m) even, odd
            m0 = (l - q) % 2
            if m0 <= l:
                par[q, :, m0:l + 1:2] += a[:, m0::2, None] * lam[m0::2]
    F = torch.stack([par[0] + par[1], par[0] - par[1]])
    out = torch.empty(B, 12 * nside * nside, dtype=torch.float64, device=DEV)
    for n, rows in _ring_groups(nside).items():
        f = F[[r[1] for r in rows], :, :, [r[0] for r in rows]]  # [rows, B, m]
        f = f * _phase(rows, lmax)[:, None]
        f[..., 1:] *= 2.0
        pad = -(lmax + 1) % n
        f = torch.nn.functional.pad(f, (0, pad)).reshape(len(rows), B, -1, n).sum(2)
        s = torch.fft.ifft(f, dim=-1).real * n
        at = torch.tensor([r[3] for r in rows], device=DEV)[:, None] + torch.arange(n, device=DEV)
        out[:, at] = s.transpose(0, 1)
    return out


def _analysis(maps, nside, lmax):
    """Omega Y^T of maps [B, npix]: coefficients [B, nalm] (m-major), all in FP64."""
    B, K = maps.shape[0], 2 * nside
    G = torch.zeros(2, B, lmax + 1, K, dtype=torch.complex128, device=DEV)
    for n, rows in _ring_groups(nside).items():
        at = torch.tensor([r[3] for r in rows], device=DEV)[:, None] + torch.arange(n, device=DEV)
        x = torch.fft.fft(maps[:, at], dim=-1)  # [B, rows, n]
        g = x[..., torch.arange(lmax + 1, device=DEV) % n] * _phase(rows, lmax).conj()
        G[[r[1] for r in rows], :, :, [r[0] for r in rows]] = g.transpose(0, 1)
    par = torch.stack([G[0] + G[1], G[0] - G[1]])
    alm = torch.zeros(B, (lmax + 1) * (lmax + 2) // 2, dtype=torch.complex128, device=DEV)
    omega = 4.0 * math.pi / (12 * nside * nside)
    for l, lam in _legendre(nside, lmax):
        at = _slot(lmax, l)
        for q in (0, 1):
            m0 = (l - q) % 2
            if m0 <= l:
                alm[:, at[m0::2]] = omega * (par[q, :, m0:l + 1:2] * lam[m0::2]).sum(-1)
    return alm


def _messenger(step, update, cl_max_mu, alpha, eps=1e-6, cap=1e-2, beta=0.75):
    """Algorithm 2's loop: step(xi, mu) -> (||x_new - x||^2, ||x_new||^2) of the signal step,
    update(xi, mu) the messenger step; cooling and tolerances as documented in wf.h."""
    mu = cl_max_mu
    xi = alpha + mu
    for _ in range(200000):
        num, den = step(xi, mu)
        c = math.sqrt(num / den) if den > 0 else 0.0
        update(xi, mu)
        tol = eps if mu == 0.0 else min(cap, eps * max(1.0, mu / alpha))
        if c < tol:
            if mu == 0.0:
                return
            xi = max(alpha, beta * xi)
            mu = xi - alpha if xi > alpha else 0.0
    raise RuntimeError("not converged")


def _exact_solve(case, seed):
    """The FP64 solve with a dense matrix of the real basis functions (small Nside only)."""
    nside, lmax = case["nside"], case["lmax"]
    p, d = _problem(nside, lmax, case["noise"], int(seed))
    npix, pr = 12 * nside * nside, _pairs(nside)
    z_of, sign, phi = (torch.empty(npix, dtype=t, device=DEV) for t in (torch.int64, torch.float64, torch.float64))
    for k, (_, _, n, p0, on, os_) in enumerate(pr):
        for o, s in ((on, 1.0), (os_, -1.0)):
            if o >= 0:
                z_of[o:o + n], sign[o:o + n] = k, s
                phi[o:o + n] = p0 + 2.0 * math.pi * torch.arange(n, dtype=torch.float64, device=DEV) / n
    nalm = (lmax + 1) * (lmax + 2) // 2
    Y = torch.empty(2, nalm, npix, dtype=torch.float64, device=DEV)
    m = torch.arange(lmax + 1, dtype=torch.float64, device=DEV)
    r2 = math.sqrt(2.0)
    for l, lam in _legendre(nside, lmax):
        par = torch.where(((l - torch.arange(l + 1, device=DEV)) % 2 == 1)[:, None], sign, 1.0)
        v = lam[:, z_of] * par
        ang = m[:l + 1, None] * phi
        w = (1.0 + (r2 - 1.0) * (m[:l + 1] > 0).to(torch.float64))[:, None]
        Y[0, _slot(lmax, l)] = v * w * torch.cos(ang)
        Y[1, _slot(lmax, l)] = v * w * torch.sin(ang)  # m = 0: zero rows
    Y = Y.reshape(2 * nalm, npix)
    omega = 4.0 * math.pi / npix
    ls, ms = inputs.lm_of_slots(lmax)
    cl = torch.from_numpy(p.cl[ls]).to(DEV).repeat(2)
    mask = torch.from_numpy(p.mask).to(DEV)
    nv = torch.from_numpy(p.noise_var).to(DEV)
    alpha = float(nv[~mask].min())
    st = {"x": torch.zeros(2 * nalm, dtype=torch.float64, device=DEV), "t": torch.where(mask, 0.0, d)}

    def step(xi, mu):
        sb = (cl - mu * omega).clamp(min=0.0)
        x = sb / (sb + xi * omega) * (omega * (Y @ st["t"]))
        num, den = torch.stack([((x - st["x"]) ** 2).sum(), (x * x).sum()]).tolist()
        st["x"] = x
        return num, den

    def update(xi, mu):
        s = Y.T @ st["x"]
        st["t"] = s + torch.where(mask, 0.0, xi / (nv + mu)) * (torch.where(mask, 0.0, d) - s)

    _messenger(step, update, 0.75 * float(p.cl.max()) / omega, alpha)
    x = st["x"].reshape(2, nalm) / torch.from_numpy(np.where(ms == 0, 1.0, r2)).to(DEV)
    return {"alm": torch.complex(x[0], -x[1]), "map": Y.T @ st["x"]}


def _exact_flat(case, seed):
    ck, area, nv, d = _flat_inputs(case, seed)
    ck = torch.from_numpy(ck).to(DEV)
    st = {"x": torch.zeros_like(d, dtype=torch.complex128), "t": d}

    def step(xi, mu):
        sb = (ck - mu * area).clamp(min=0.0)
        x = torch.where(sb > 0, sb / (sb + xi * area), 0.0) * torch.fft.fft2(st["t"])
        e = torch.view_as_real(x - st["x"])
        num, den = torch.stack([(e * e).sum(), (torch.view_as_real(x) ** 2).sum()]).tolist()
        st["x"] = x
        return num, den

    def update(xi, mu):
        s = torch.fft.ifft2(st["x"]).real
        st["t"] = s + xi / (nv + mu) * (d - s)

    _messenger(step, update, 0.75 * float(ck.max()) / area, float(nv.min()))
    return torch.fft.ifft2(st["x"]).real


def _conv(x, W, b, rings):
    """Circular convolutions along every ring: x [C, npix], W [O, C, K] -> [O, npix]."""
    h = W.shape[2] // 2
    out = []
    for n, at in rings:
        j = (torch.arange(n, device=DEV)[:, None] + torch.arange(W.shape[2], device=DEV) - h) % n
        out.append(torch.einsum("crnk,ock->orn", x[:, at][:, :, j], W).reshape(W.shape[0], -1))
    y = torch.cat(out, 1) + b[:, None]
    back = torch.empty(y.shape[1], dtype=torch.int64, device=DEV)
    back[torch.cat([at.reshape(-1) for _, at in rings])] = torch.arange(y.shape[1], device=DEV)
    return y[:, back]


def _exact_train(case, seed):
    nside, lmax, H, K, M = (case[k] for k in ("nside", "lmax", "channels", "kernel", "hidden"))
    p, d, target, theta = _train_inputs(case, seed)
    t = torch.from_numpy(theta).to(torch.bfloat16).to(torch.float64).to(DEV)
    shapes = [(H, 3, K), (H,), (H, H, K), (H,), (1, H, K), (1,), (M, 4), (M,), (M, M), (M,), (1, M), (1,)]
    par, o = [], 0
    for s in shapes:
        n = math.prod(s)
        par.append(t[o:o + n].reshape(s).clone().requires_grad_())
        o += n
    W1, b1, W2, b2, W3, b3, V1, c1, V2, c2, V3, c3 = par
    mask = torch.from_numpy(p.mask).to(DEV)
    lg = torch.from_numpy(np.log(p.noise_var)).to(DEV)
    seen = ~mask
    sig = float(d[seen].square().mean().sqrt())
    mean, std = float(lg[seen].mean()), float(lg[seen].var(unbiased=False).sqrt())
    dm = torch.where(mask, 0.0, d)
    x = torch.stack([dm / sig, torch.where(mask, 0.0, (lg - mean) / std), mask.to(torch.float64)])
    rings = [(n, torch.tensor([r[3] for r in rows], device=DEV)[:, None] + torch.arange(n, device=DEV))
             for n, rows in _ring_groups(nside).items()]
    r = _conv(torch.relu(_conv(torch.relu(_conv(x, W1, b1, rings)), W2, b2, rings)), W3, b3, rings)[0]
    with torch.no_grad():
        a, ad = _analysis(torch.stack([dm + sig * r, dm]), nside, lmax)
    ls, ms = (torch.from_numpy(v).to(DEV) for v in inputs.lm_of_slots(lmax))
    w = torch.where(ms == 0, 1.0, 2.0).to(torch.float64)
    zero = torch.zeros(lmax + 1, dtype=torch.float64, device=DEV)
    cl = torch.from_numpy(p.cl).to(DEV) + 1e-30
    l = torch.arange(lmax + 1, dtype=torch.float64, device=DEV)
    pd = zero.index_add(0, ls, w * ad.abs() ** 2) / (2 * l + 1)
    aom = float(torch.from_numpy(p.noise_var).to(DEV)[seen].min()) * 4.0 * math.pi / (12 * nside * nside)
    feat = torch.stack([l / lmax, (torch.log10(cl) / 10).clamp(-4, 4), (torch.log10((pd + 1e-30) / cl) / 5).clamp(-4, 4),
                        (torch.log10(aom / cl) / 5).clamp(-4, 4)], 1)
    q = torch.sigmoid(torch.relu(torch.relu(feat @ V1.T + c1) @ V2.T + c2) @ V3.T + c3)[:, 0]
    norm = (w * target.abs() ** 2).sum()
    err = q[ls] * a - target
    loss = (w * err.abs() ** 2).sum() / norm
    loss.backward()
    with torch.no_grad():
        up = _synthesis((2.0 * q[ls] * err / norm)[None], nside, lmax)[0] * (4.0 * math.pi / (12 * nside * nside)) * sig
    r.backward(up)
    return {"loss": float(loss), "grad": torch.cat([v.grad.reshape(-1) for v in par])}


def exact(case, seed):
    op = case["op"]
    if op in ("sht", "group"):
        alm, maps = _sht_inputs(case, seed)
        m, a = _synthesis(alm, case["nside"], case["lmax"]), _analysis(maps, case["nside"], case["lmax"])
        return {"map": m, "alm": a} if op == "group" else {"map": m[0], "alm": a[0]}
    if op == "solve":
        # a mixed solve's workload is too large for a dense matrix
        return _exact_solve(case, seed) if case["prec"] == "f64" else None
    if op == "batch":
        return None
    return _exact_flat(case, seed) if op == "flat" else _exact_train(case, seed)
