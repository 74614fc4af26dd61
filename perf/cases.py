"""What the framework's speed is measured on.

Each case is one call, or one short sequence of calls, that a program using the
framework makes: the photon transport, a whole projection, a ray-traced view,
the scatter denoiser, the reconstruction of a scan, the learned scatter
estimator and its matrix product.  ``prepare`` builds what such a program holds
before the call (phantom, context, images, weights) from the seed, ``run`` makes
the call, ``work`` says what the call cannot do without, and ``exact`` gives the
floating-point results in 64 bits with plain torch.
"""
import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_1204_6367_gb300 import gdrr, inputs, scan

DETECTOR_MM = (397.3, 298.0)      # extent of the flat panel: 512 x 384 pixels of 0.776 mm
PHANTOM_MM = (512.0, 512.0, 256.0)
# free flights of a history in the torso and in the small cylinder (global
# majorant), and FP32 operations of one flight (Philox apart): about 40
FLIGHTS = {"torso": 46.0, "cylinder": 5.1}
FLIGHT_FLOPS = 40.0


def listed():
    return [
        # 20000 histories of the 64 x 64 cylinder: the package's smoke test, and
        # the tuning and sanity runs that users make first; launch latency
        {"name": "mc-cylinder-2e4", "kind": "mc", "phantom": "cylinder", "vox": 4.0, "nu": 64, "nv": 64,
         "n": 20_000, "option": "default"},
        # one high-photon projection of the 2 mm torso, the usual operating
        # point (about 36 counts per coarse scatter pixel)
        {"name": "mc-torso-1e8", "kind": "mc", "phantom": "torso", "vox": 2.0, "nu": 512, "nv": 384,
         "n": 100_000_000, "option": "default"},
        # the transport with tabulated Rayleigh form factors, on the 4 mm torso
        # and the coarse scatter grid
        {"name": "mc-torso-ff-1e7", "kind": "mc", "phantom": "torso", "vox": 4.0, "nu": 128, "nv": 96,
         "n": 10_000_000, "option": "form-factor"},
        # the transport with local majorants, the option for speed
        {"name": "mc-torso-local-2e7", "kind": "mc", "phantom": "torso", "vox": 2.0, "nu": 512, "nv": 384,
         "n": 20_000_000, "option": "local"},
        # a multi-angle scan replayed from its graph
        {"name": "scan-16-angles", "kind": "scan", "phantom": "torso", "vox": 4.0, "nu": 128, "nv": 96,
         "angles": 16, "n": 16_000_000},
        # one low-photon projection on the coarse grid: what the learned
        # estimator's input and training pairs are made of
        {"name": "project-coarse-1e6", "kind": "project", "phantom": "torso", "vox": 4.0, "nu": 128, "nv": 96,
         "n": 1_000_000, "bin": 1, "smoothing": 12.0, "iters": 800},
        # one ray-traced view of the 2 mm torso, the step of a primary-only scan
        {"name": "raytrace-torso", "kind": "raytrace", "vox": 2.0, "nu": 512, "nv": 384},
        # reconstruction of a 360-view scan onto the 2 mm grid
        {"name": "reconstruct-360", "kind": "fdk", "views": 360, "nu": 512, "nv": 384, "nx": 256, "ny": 256,
         "nz": 128},
        # the scatter denoiser alone on the coarse grid of a full detector
        {"name": "denoise-128x96", "kind": "denoise", "nu": 128, "nv": 96, "iters": 300, "beta": 0.05},
        # the learned estimator on 64 projections at once
        {"name": "estimator-forward-64", "kind": "forward", "batch": 64, "height": 96, "width": 128, "channels": 32},
        # eight training steps of the estimator on batches of 16
        {"name": "estimator-train-8x16", "kind": "train", "batch": 16, "height": 96, "width": 128, "channels": 32,
         "steps": 8},
        # the estimator's matrix product at the size its rate is quoted on
        {"name": "gemm-8192", "kind": "gemm", "m": 8192, "n": 8192, "k": 8192},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _detector(rng, lo, hi):
    nu = _log(rng, lo, hi)
    return {"nu": nu, "nv": int(nu * rng.uniform(0.6, 0.75))}


def draw(rng):
    kind = rng.choice(["mc", "mc", "mc", "scan", "project", "raytrace", "fdk", "denoise", "forward", "train", "gemm"])
    if kind == "mc":
        phantom = rng.choice(["torso", "torso", "cylinder"])
        option = rng.choice(["default", "default", "local", "form-factor", "nearest", "hardened"])
        if phantom == "cylinder" and option == "hardened":
            option = "default"
        return {"kind": kind, "phantom": phantom, "vox": round(rng.uniform(2.0, 6.0), 2) if phantom == "torso" else 4.0,
                **_detector(rng, 64, 512),
                "n": _log(rng, 10_000, 50_000_000 if option == "default" else 20_000_000), "option": option}
    if kind == "scan":
        return {"kind": kind, "phantom": "torso", "vox": round(rng.uniform(2.5, 6.0), 2), **_detector(rng, 64, 256),
                "angles": rng.randint(2, 32), "n": _log(rng, 200_000, 30_000_000)}
    if kind == "project":
        f = rng.choice([1, 2, 4])
        return {"kind": kind, "phantom": "torso", "vox": round(rng.uniform(2.0, 5.0), 2),
                "nu": f * rng.randint(48, 128), "nv": f * rng.randint(36, 96), "n": _log(rng, 300_000, 20_000_000),
                "bin": f, "smoothing": float(rng.randint(4, 12)), "iters": rng.randint(200, 800)}
    if kind == "raytrace":
        return {"kind": kind, "vox": round(rng.uniform(2.0, 6.0), 2), **_detector(rng, 64, 512)}
    if kind == "fdk":
        return {"kind": kind, "views": rng.randint(60, 360), **_detector(rng, 128, 512),
                "nx": rng.randint(64, 256), "ny": rng.randint(64, 256), "nz": rng.randint(32, 128)}
    if kind == "denoise":
        return {"kind": kind, "nu": _log(rng, 48, 512), "nv": _log(rng, 32, 384), "iters": _log(rng, 100, 600),
                "beta": round(rng.uniform(0.05, 0.5), 3)}
    if kind in ("forward", "train"):
        c = {"kind": kind, "batch": _log(rng, 1, 64 if kind == "forward" else 24), "height": 8 * rng.randint(4, 12),
             "width": 8 * rng.randint(4, 16), "channels": rng.choice([16, 32, 32])}
        if kind == "train":
            c["steps"] = rng.randint(2, 8)
        return c
    return {"kind": kind, "m": _log(rng, 256, 8192), "n": 8 * _log(rng, 16, 1024), "k": 64 * _log(rng, 1, 128)}


# ---- inputs ---------------------------------------------------------------

def _rng(seed):
    return np.random.default_rng([77, int(seed)])


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(1_000_003 * (int(seed) + 1))
    return g


def _problem(case, seed):
    """The torso (anatomy by the seed) or the cylinder (rod and water by the seed)."""
    nu, nv = case["nu"], case["nv"]
    if case.get("phantom", "torso") == "torso":
        px = max(DETECTOR_MM[0] / nu, DETECTOR_MM[1] / nv)
        return inputs.torso_problem(vox=case["vox"], seed=int(seed), nu=nu, nv=nv, det_px=px,
                                    hardened_bowtie=case.get("option") == "hardened")
    r = _rng(seed)
    p = inputs.small_problem(energy=float(r.integers(50, 71)))
    if (nu, nv) != (p.nu, p.nv):
        px = 256.0 / max(nu, nv)
        p.nu, p.nv, p.du, p.dv = nu, nv, px, px
        p.fluence = inputs.fluence_map(nu, nv, px, px, p.sdd)
    p.material, p.density = inputs.cylinder_phantom(32, 4.0, float(r.uniform(45, 55)), float(r.uniform(8, 12)))
    return p


def _angle(seed):
    return float(_rng(seed).uniform(0.0, 2.0 * math.pi))


def _specs(c):
    """(input channels, output channels, kernel) of the estimator's convolutions in parameter order."""
    return [(2, c, 3), (c, 2 * c, 3), (2 * c, 4 * c, 3), (4 * c, 8 * c, 3), (12 * c, 4 * c, 3), (6 * c, 2 * c, 3),
            (3 * c, c, 3), (c, 1, 1)]


def _weights(c, seed):
    r = _rng(seed)
    parts = []
    for ci, co, k in _specs(c):
        parts += [r.normal(0.0, math.sqrt(2.0 / (ci * k * k)), co * ci * k * k), r.normal(0.0, 0.01, co)]
    return np.concatenate(parts).astype(np.float32)


def _smooth(n, ch, h, w, g, lo, hi):
    """Smooth positive images, as scatter and primary images are."""
    z = torch.rand((n, ch, 5, 6), device="cuda", generator=g)
    z = F.interpolate(z, size=(h, w), mode="bicubic", align_corners=True)
    return (lo + (hi - lo) * z).clamp_min(lo).float().contiguous()


def _pairs(case, seed, n):
    g = _gen(seed)
    y = _smooth(n, 1, case["height"], case["width"], g, 0.3, 1.2)
    x = torch.cat([y * (1.0 + 0.05 * torch.randn(y.shape, device="cuda", generator=g)),
                   _smooth(n, 1, case["height"], case["width"], g, 0.2, 3.0)], 1).contiguous()
    return x, y


def _ellipsoids(seed):
    """(centre, radii, attenuation per mm) of a torso-like object in mm."""
    r = _rng(seed)
    e = [((0.0, 0.0, 0.0), (170.0, 110.0, 200.0), 0.019)]
    for side in (-1.0, 1.0):
        e.append(((side * r.uniform(60, 80), r.uniform(-5, 15), r.uniform(-20, 20)),
                  (r.uniform(45, 60), r.uniform(50, 65), r.uniform(90, 120)), -0.013))
    for _ in range(3):
        a = r.uniform(0, 2 * math.pi)
        e.append(((60 * math.cos(a), 60 * math.sin(a), r.uniform(-60, 60)), tuple(r.uniform(8, 25, 3)), 0.02))
    return e


def _fdk_problem(case, seed):
    px = max(DETECTOR_MM[0] / case["nu"], DETECTOR_MM[1] / case["nv"])
    return inputs.torso_problem(vox=8.0, seed=int(seed), nu=case["nu"], nv=case["nv"], det_px=px)


def _air(prob):
    """Unattenuated signal of every pixel in 64 bits: w(u) sum phi r(E)."""
    phi = prob.spec_w / prob.spec_w.sum()
    r = np.interp(prob.spec_e, prob.r0 + prob.dr * np.arange(prob.response.size), prob.response.astype(np.float64))
    w = torch.from_numpy(prob.fluence / prob.fluence.sum()).cuda()
    return w * float((phi * r).sum())


def _frame(prob, angle):
    """Source, detector centre and detector axes (imager opposite the source)."""
    c, s = math.cos(angle), math.sin(angle)
    t = angle + prob.theta
    n = (math.cos(t), math.sin(t))
    aid = prob.sdd - prob.sad
    return (-prob.sad * c, -prob.sad * s, 0.0), (aid * n[0], aid * n[1], 0.0), (n[1], -n[0], 0.0), n


def _rays(prob, angle):
    """Unit directions [3][nv, nu] and lengths of the rays to the pixel centres, and the source."""
    S, P, eu, _ = _frame(prob, angle)
    u = (torch.arange(prob.nu, device="cuda", dtype=torch.float64) + 0.5 - 0.5 * prob.nu) * prob.du
    v = (torch.arange(prob.nv, device="cuda", dtype=torch.float64) + 0.5 - 0.5 * prob.nv) * prob.dv
    d = [(P[0] - S[0] + u * eu[0])[None, :].expand(prob.nv, -1), (P[1] - S[1] + u * eu[1])[None, :].expand(prob.nv, -1),
         v[:, None].expand(-1, prob.nu)]
    length = torch.sqrt(d[0] ** 2 + d[1] ** 2 + d[2] ** 2)
    return S, [x / length for x in d], length


def _scan_signal(case, prob, seed):
    """Noisy signals of a full orbit around the ellipsoids, FP64 [views, nv, nu]."""
    I0, g = _air(prob), _gen(seed)
    out = torch.empty((case["views"], prob.nv, prob.nu), dtype=torch.float64, device="cuda")
    for i, a in enumerate(scan.full_orbit(case["views"])):
        S, d, _ = _rays(prob, float(a))
        path = torch.zeros_like(d[0])
        for c, r, mu in _ellipsoids(seed):
            p = [(S[k] - c[k]) / r[k] for k in range(3)]
            q = [d[k] / r[k] for k in range(3)]
            aa = q[0] ** 2 + q[1] ** 2 + q[2] ** 2
            bb = p[0] * q[0] + p[1] * q[1] + p[2] * q[2]
            disc = bb * bb - aa * (p[0] ** 2 + p[1] ** 2 + p[2] ** 2 - 1.0)
            path += mu * 2.0 * torch.sqrt(disc.clamp_min(0.0)) / aa
        path.clamp_(min=0.0)
        noise = torch.randn(path.shape, device="cuda", generator=g)
        out[i] = I0 * torch.exp(-path) * (1.0 + 0.002 * torch.exp(0.5 * path) * noise)
    return out


def _counts(case, seed):
    """A Poisson-noisy scatter image on the signal scale and the signal of one count."""
    g = _gen(seed)
    scale = 1.0e-9 * (1.0 + float(_rng(seed).random()))
    mean = _smooth(1, 1, case["nv"], case["nu"], g, 15.0, 60.0)[0, 0]
    return torch.poisson(mean, generator=g).double().mul_(scale).contiguous(), scale


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("mc", "scan", "project", "raytrace"):
        prob = _problem(case, seed)
        ctx = gdrr.Context(prob)
        state = {"case": case, "ctx": ctx, "seed": 1 + int(seed), "angle": _angle(seed)}
        opt = case.get("option", "default")
        if opt == "local":
            gdrr.gdrr_set_options(ctx, local_majorant=1)
        elif opt == "form-factor":
            gdrr.gdrr_set_options(ctx, rayleigh_form_factor=1)
        elif opt == "nearest":
            gdrr.gdrr_set_options(ctx, nearest_voxel=1)
        if kind == "scan":
            share = _rng(seed).uniform(1.0, 5.0, case["angles"])
            budgets = np.maximum(1, share / share.sum() * case["n"]).astype(np.uint64)
            angles = np.arange(case["angles"]) * (2.0 * math.pi / case["angles"])
            state["scan"] = gdrr.gdrr_scan_create(ctx, angles, budgets, 1 + int(seed))
        return state
    if kind == "fdk":
        prob = _fdk_problem(case, seed)
        return {"case": case, "ctx": gdrr.Context(prob), "signal": _scan_signal(case, prob, seed),
                "angles": scan.full_orbit(case["views"])}
    if kind == "denoise":
        s_hat, scale = _counts(case, seed)
        return {"case": case, "ctx": gdrr.Context(inputs.small_problem()), "s_hat": s_hat, "scale": scale}
    if kind in ("forward", "train"):
        net = gdrr.Cnn(case["batch"], case["height"], case["width"], case["channels"])
        net.set_params(_weights(case["channels"], seed))
        x, y = _pairs(case, seed, case["batch"] * case.get("steps", 1))
        return {"case": case, "net": net, "x": x, "y": y}
    g = _gen(seed)
    return {"case": case, "a": torch.randn((case["m"], case["k"]), device="cuda", generator=g).bfloat16(),
            "b": torch.randn((case["n"], case["k"]), device="cuda", generator=g).bfloat16()}


# ---- one pass ---------------------------------------------------------------

LEARNING_RATE = 1e-5     # a fine-tuning step


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "mc":
        stats = torch.zeros(gdrr.GDRR_NSTATS, dtype=torch.int64, device="cuda")
        prim, scat = gdrr.gdrr_mc_project(state["ctx"], case["n"], state["seed"], state["angle"], stats=stats)
        return {"prim": prim, "scat": scat, "stats": stats}
    if kind == "scan":
        prim, scat = gdrr.gdrr_scan_launch(state["scan"])
        return {"prim": prim, "scat": scat}
    if kind == "project":
        r = gdrr.project(state["ctx"], case["n"], state["seed"], state["angle"], bin_factor=case["bin"],
                         smoothing_px=case["smoothing"], iters=case["iters"])
        return {k: r[k] for k in ("P", "P_hat", "S_hat", "S", "N", "S_hat_coarse", "S_coarse", "prim", "scat", "stats",
                                  "count_scale", "beta", "mean_count")}
    if kind == "raytrace":
        return {"P": gdrr.gdrr_raytrace_primary(state["ctx"], state["angle"])}
    if kind == "fdk":
        return {"volume": scan.reconstruct(state["ctx"], state["angles"], state["signal"],
                                           (case["nz"], case["ny"], case["nx"]), _grid(case))}
    if kind == "denoise":
        return {"S": gdrr.gdrr_denoise_scatter(state["ctx"], state["s_hat"], state["scale"], case["beta"],
                                               iters=case["iters"])}
    if kind == "forward":
        return {"out": state["net"].forward(state["x"])}
    if kind == "train":
        net, b, losses = state["net"], case["batch"], []
        for i in range(case["steps"]):
            net.forward(state["x"][i * b:(i + 1) * b])
            losses.append(net.backward(state["y"][i * b:(i + 1) * b]))
            net.adam_step(LEARNING_RATE)
        return {"losses": losses, "grads": net.get_grads(), "params": net.get_params()}
    return {"c": gdrr.gdrr_gemm_bf16(state["a"], state["b"])}


def _grid(case):
    """Voxel size of the reconstruction grid: the torso's extent, whatever the counts."""
    return (PHANTOM_MM[0] / case["nx"], PHANTOM_MM[1] / case["ny"], PHANTOM_MM[2] / case["nz"])


# ---- what a pass cannot do without -------------------------------------------

def _voxels(case):
    if case.get("phantom", "torso") == "cylinder":
        return 32 ** 3
    return math.prod(int(round(e / case["vox"])) for e in PHANTOM_MM)


def work(case):
    kind = case["kind"]
    if kind in ("mc", "scan", "project", "raytrace"):
        pixels = case["nu"] * case["nv"]
        phantom = 5.0 * _voxels(case)                       # density and material, once
        steps = 600.0 * 2.0 / case["vox"]                   # midpoints of a ray's chord
        ray = pixels * (steps * 40.0 + 110.0 * 10.0)
        flights = case.get("n", 0) * FLIGHTS[case.get("phantom", "torso")]
        if kind == "raytrace":
            return {"bytes": phantom + 8.0 * pixels, "flops": ray}
        if kind == "project":
            return {"bytes": phantom + 64.0 * pixels,
                    "flops": flights * FLIGHT_FLOPS + ray + 10.0 * case["iters"] * pixels / case["bin"] ** 2}
        return {"bytes": phantom + 16.0 * pixels * case.get("angles", 1), "flops": flights * FLIGHT_FLOPS}
    if kind == "fdk":
        rays = case["views"] * case["nu"] * case["nv"]
        voxels = case["nx"] * case["ny"] * case["nz"]
        return {"bytes": 8.0 * rays + 4.0 * voxels,
                "flops": rays * (20.0 + case["nu"]) + 12.0 * voxels * case["views"]}
    if kind == "denoise":
        pixels = case["nu"] * case["nv"]
        return {"bytes": 16.0 * pixels, "flops": 10.0 * pixels * case["iters"]}
    if kind in ("forward", "train"):
        c, px = case["channels"], case["height"] * case["width"]
        level = [0, 1, 2, 3, 2, 1, 0, 0]
        macs = sum(px / 4 ** l * ci * co * k * k for l, (ci, co, k) in zip(level, _specs(c)))
        n = sum(co * ci * k * k + co for ci, co, k in _specs(c))
        images = case["batch"] * case.get("steps", 1)
        if kind == "forward":
            return {"bytes": 12.0 * px * images + 2.0 * n, "flops": 2.0 * macs * images}
        return {"bytes": 12.0 * px * images + 24.0 * n * case["steps"], "flops": 6.0 * macs * images}
    m, n, k = case["m"], case["n"], case["k"]
    return {"bytes": 2.0 * (m + n) * k + 4.0 * m * n, "flops": 2.0 * m * n * k}


# ---- the results in 64 bits ---------------------------------------------------

def _exact_primary(prob, angle):
    """Eq. 1 with trilinear interpolation at the midpoints of equal intervals
    of at most half the smallest voxel edge, FP64 [nv, nu]."""
    dev, f64 = "cuda", torch.float64
    S, d, length = _rays(prob, angle)
    d = [x.reshape(-1) for x in d]
    nz, ny, nx = prob.material.shape
    dims, vox = (nx, ny, nz), prob.voxel
    lo = [-0.5 * n * e for n, e in zip(dims, vox)]
    tmin, tmax = torch.zeros_like(d[0]), length.reshape(-1).clone()
    for a in range(3):
        inv = 1.0 / torch.where(d[a] == 0.0, torch.full_like(d[a], 1e-300), d[a])
        t1, t2 = (lo[a] - S[a]) * inv, (-lo[a] - S[a]) * inv
        tmin = torch.maximum(tmin, torch.minimum(t1, t2))
        tmax = torch.minimum(tmax, torch.maximum(t1, t2))
    chord = (tmax - tmin).clamp_min(0.0)
    n = torch.ceil(chord / (0.5 * min(vox))).clamp_min(1.0)
    dl = chord / n
    n_mat = prob.mu_hat.shape[0]
    mat = torch.from_numpy(np.ascontiguousarray(prob.material)).to(dev).reshape(-1).long()
    rho = torch.from_numpy(np.ascontiguousarray(prob.density)).to(dev).reshape(-1).double()
    ell = torch.zeros((n_mat, d[0].numel()), dtype=f64, device=dev)
    rows = 8192
    for r0 in range(0, d[0].numel(), rows):
        sl = slice(r0, min(d[0].numel(), r0 + rows))
        m = int(n[sl].max())
        j = torch.arange(m, device=dev, dtype=f64)[None, :]
        t = tmin[sl, None] + (j + 0.5) * dl[sl, None]
        inside = (j < n[sl, None]) & (chord[sl, None] > 0.0)
        i0, i1, w = [], [], []
        for a in range(3):
            f = (S[a] + t * d[a][sl, None] - lo[a]) / vox[a] - 0.5
            g = torch.floor(f)
            w.append(f - g)
            i0.append(g.long().clamp(0, dims[a] - 1))
            i1.append((g.long() + 1).clamp(0, dims[a] - 1))
        part = torch.zeros((n_mat,) + t.shape, dtype=f64, device=dev)
        for c in range(8):
            k = [(i1 if (c >> a) & 1 else i0)[a] for a in range(3)]
            ww = [w[a] if (c >> a) & 1 else 1.0 - w[a] for a in range(3)]
            v = (k[2] * ny + k[1]) * nx + k[0]
            val = ww[0] * ww[1] * ww[2] * rho[v] * inside
            part.scatter_add_(0, mat[v][None], val[None])
        ell[:, sl] = part.sum(-1) * dl[None, sl]
    grid = prob.e0 + prob.de * np.arange(prob.mu_hat.shape[2])
    total = prob.mu_hat.astype(np.float64).sum(1)
    mu = torch.from_numpy(np.stack([np.interp(prob.spec_e, grid, total[q]) for q in range(n_mat)]) * 0.1).to(dev)
    phi = prob.spec_w / prob.spec_w.sum()
    r = np.interp(prob.spec_e, prob.r0 + prob.dr * np.arange(prob.response.size), prob.response.astype(np.float64))
    sig = torch.zeros_like(d[0])
    for b in range(prob.spec_e.size):
        sig += float(phi[b] * r[b]) * torch.exp(-(mu[:, b, None] * ell).sum(0))
    w = torch.from_numpy(prob.fluence / prob.fluence.sum()).to(dev)
    return w * sig.reshape(prob.nv, prob.nu)


def _exact_volume(case, seed):
    prob = _fdk_problem(case, seed)
    signal, I0, dev, f64 = _scan_signal(case, prob, seed), _air(prob), "cuda", torch.float64
    nu, nv, mag = prob.nu, prob.nv, prob.sad / prob.sdd
    tu, tv = prob.du * mag, prob.dv * mag
    a = (torch.arange(nu, device=dev, dtype=f64) + 0.5 - 0.5 * nu) * tu
    b = (torch.arange(nv, device=dev, dtype=f64) + 0.5 - 0.5 * nv) * tv
    cosine = prob.sad / torch.sqrt(prob.sad ** 2 + a[None, :] ** 2 + b[:, None] ** 2)
    off = torch.arange(nu, device=dev)[:, None] - torch.arange(nu, device=dev)[None, :]
    odd = off.abs() % 2 == 1
    ramp = torch.where(odd, -1.0 / (math.pi * torch.where(odd, off, 1).double()) ** 2, torch.zeros((), dtype=f64, device=dev))
    ramp = torch.where(off == 0, torch.full((), 0.25, dtype=f64, device=dev), ramp) / (2.0 * tu)
    vx, vy, vz = _grid(case)
    x = ((torch.arange(case["nx"], device=dev, dtype=f64) + 0.5 - 0.5 * case["nx"]) * vx)[None, :]
    y = ((torch.arange(case["ny"], device=dev, dtype=f64) + 0.5 - 0.5 * case["ny"]) * vy)[:, None]
    z = ((torch.arange(case["nz"], device=dev, dtype=f64) + 0.5 - 0.5 * case["nz"]) * vz)[:, None, None]
    vol = torch.zeros((case["nz"], case["ny"], case["nx"]), dtype=f64, device=dev)
    d_beta = 2.0 * math.pi / case["views"]
    for i, phi in enumerate(scan.full_orbit(case["views"])):
        g = -torch.log(torch.maximum(signal[i], 1e-6 * I0) / I0)
        q = F.pad((g * cosine) @ ramp, (2, 2, 2, 2))
        c, s = math.cos(float(phi)), math.sin(float(phi))
        depth = prob.sad + x * c + y * s
        fu = (prob.sad * (x * s - y * c) / depth / tu + 0.5 * nu - 0.5).clamp(-2.0, nu + 0.5)
        fv = (prob.sad / depth / tv * z + 0.5 * nv - 0.5).clamp(-2.0, nv + 0.5)
        iu, iv = torch.floor(fu), torch.floor(fv)
        wu, wv = (fu - iu)[None], fv - iv
        k = (iv.long() + 2) * (nu + 4) + (iu.long() + 2)[None]
        q = q.reshape(-1)
        lo = q[k] * (1.0 - wu) + q[k + 1] * wu
        hi = q[k + nu + 4] * (1.0 - wu) + q[k + nu + 5] * wu
        vol += d_beta * (prob.sad / depth)[None] ** 2 * (lo * (1.0 - wv) + hi * wv)
    return vol


def _exact_denoise(case, seed):
    s_hat, scale = _counts(case, seed)
    sc = s_hat / scale
    s, omega, beta = sc.clamp_min(1e-3), 0.8, case["beta"]
    for _ in range(case["iters"]):
        p = F.pad(s[None, None], (1, 1, 1, 1), mode="replicate")[0, 0]
        sigma = p[1:-1, 2:] + p[2:, 1:-1] + p[1:-1, :-2] + p[:-2, 1:-1]
        s = ((1.0 - omega) * s + omega / 4.0 * (sigma - (1.0 - sc / s) / beta)).clamp_min(1e-3)
    return s * scale


def _network(p, x, c):
    """The encoder-decoder on flat 64-bit parameters."""
    w, off = [], 0
    for ci, co, k in _specs(c):
        n = co * ci * k * k
        w.append((p[off:off + n].reshape(co, ci, k, k), p[off + n:off + n + co]))
        off += n + co

    def conv(i, v):
        return F.relu(F.conv2d(v, w[i][0], w[i][1], padding=1))

    def up(v):
        return v.repeat_interleave(2, 2).repeat_interleave(2, 3)

    e1 = conv(0, x)
    e2 = conv(1, F.avg_pool2d(e1, 2))
    e3 = conv(2, F.avg_pool2d(e2, 2))
    e4 = conv(3, F.avg_pool2d(e3, 2))
    d3 = conv(4, torch.cat([up(e4), e3], 1))
    d2 = conv(5, torch.cat([up(d3), e2], 1))
    d1 = conv(6, torch.cat([up(d2), e1], 1))
    return F.conv2d(d1, w[7][0], w[7][1]) + x[:, :1]


def exact(case, seed):
    kind = case["kind"]
    if kind in ("mc", "scan"):
        return None                       # counts and fixed-point tallies: whole numbers
    if kind in ("raytrace", "project"):
        P = _exact_primary(_problem(case, seed), _angle(seed))
        return {"P": P}                   # the rest of a projection follows from its random histories
    if kind == "fdk":
        return {"volume": _exact_volume(case, seed)}
    if kind == "denoise":
        return {"S": _exact_denoise(case, seed)}
    if kind == "gemm":
        s = prepare(case, seed)
        return {"c": s["a"].double() @ s["b"].double().T}
    p = torch.from_numpy(_weights(case["channels"], seed)).cuda().double()
    b = case["batch"]
    x, y = _pairs(case, seed, b * case.get("steps", 1))
    if kind == "forward":
        with torch.no_grad():
            return {"out": torch.cat([_network(p, v.double(), case["channels"]) for v in x.split(8)])}
    m, v, losses, grad = torch.zeros_like(p), torch.zeros_like(p), [], None
    for i in range(case["steps"]):
        p = p.detach().requires_grad_()
        loss = F.mse_loss(_network(p, x[i * b:(i + 1) * b].double(), case["channels"]), y[i * b:(i + 1) * b].double())
        grad, = torch.autograd.grad(loss, p)
        losses.append(float(loss))
        m, v = 0.9 * m + 0.1 * grad, 0.999 * v + 0.001 * grad * grad
        p = p.detach() - LEARNING_RATE * (m / (1 - 0.9 ** (i + 1))) / (torch.sqrt(v / (1 - 0.999 ** (i + 1))) + 1e-8)
    return {"losses": losses, "grads": grad, "params": p}
