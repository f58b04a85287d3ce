"""Workloads of the library, each one pass through its public entry points.

A case is a dict of plain values; ``prepare`` makes its inputs on the GPU from a seed,
``run`` makes one pass, ``work`` gives the bytes and flops the pass cannot do without and
``exact`` its outputs in 64 bits by plain torch (all pairs, no tree).

Particle sets are those of the benchmark: uniform in the periodic unit cube, or
clustered (half uniform, half in 256 Plummer spheres); equal masses 1/N, Gaussian
velocities, log-normal internal energies.  Smoothing lengths come from particle counts
on a hierarchy of grids, so that a sphere of radius h holds about 64 particles with a
scatter of some 10% in h (the spread of h before a timestep's iteration); density and f,
where a case takes them as inputs, are 64 m / (4 pi h^3 / 3) and 1 with a scatter.
Active subsets are runs along the curve of mean length 32.
"""

import math

import numpy as np
import torch

import paper_1810_09898_gb300 as sg

NNGB = 64.0
GAMMA, ALPHA, BETA, EPS = 5.0 / 3.0, 1.0, 2.0, 0.01
KERNEL = 8.0 / math.pi
# the iteration's tolerance where a gradient is to follow (h has to satisfy the relation
# between h and the density); it also makes the accepted h a smooth function of the inputs
TIGHT = 1e-3
EXACT_MAX_N = 140_000


def listed():
    return [
        # keys and order of a small set by the allocation-free call: a plug-in's per-step sort
        {"name": "order_static_20k", "kind": "order_static", "set": "uniform", "n": 20_000},
        # keys, order and octree of a mid-size set, ragged count: what every step starts with
        {"name": "order_4M", "kind": "order", "set": "clustered", "n": 4_000_037},
        # the small standard box, every particle active, h iterated from the uniform guess
        {"name": "density_iterated_32k", "kind": "density", "set": "uniform", "n": 32_768, "g": 16, "frac": 1.0,
         "iterate": True},
        # density of a sparse step: 20% active in runs, groups of 8
        {"name": "density_runs_2M", "kind": "density", "set": "clustered", "n": 2_097_152, "g": 8, "frac": 0.2,
         "iterate": False},
        # hydro forces of every particle at converged h
        {"name": "hydro_4M", "kind": "hydro", "set": "clustered", "n": 4_194_304, "g": 16, "frac": 1.0,
         "balsara": False},
        # hydro forces with the viscosity limiter, 30% active, ragged count
        {"name": "hydro_balsara_131k", "kind": "hydro", "set": "clustered", "n": 131_071, "g": 32, "frac": 0.3,
         "balsara": True},
        # density with velocity divergence and curl in the same loop (the limiter's inputs)
        {"name": "derivs_100k", "kind": "derivs", "set": "clustered", "n": 100_003, "g": 16, "frac": 1.0},
        # differentiable forces of a small set: autograd forward and backward
        {"name": "gradient_30k", "kind": "gradient", "set": "clustered", "n": 30_011, "g": 16},
        # the adjoint alone at the size of the gradient workload
        {"name": "backward_2M", "kind": "backward", "set": "clustered", "n": 2_097_152, "g": 16},
        # the standard method: one walk per particle, density and hydro
        {"name": "individual_1M", "kind": "individual", "set": "clustered", "n": 1_048_576, "frac": 1.0},
        # a whole timestep of the large box: order, octree, iterated density, hydro
        {"name": "step_16M", "kind": "step", "set": "clustered", "n": 16_777_216, "g": 16, "frac": 1.0},
        # many independent boxes of uneven sizes in one captured call, forward and backward
        {"name": "batch_16", "kind": "batch", "boxes": 16, "n_min": 10_000, "n_max": 400_000, "layout": 5,
         "backward": True},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["order_static", "order", "density", "density", "hydro", "hydro", "derivs", "velocity",
                       "gradient", "backward", "individual", "step", "batch"])
    c = {"kind": kind}
    if kind == "batch":
        c.update(boxes=rng.randint(2, 24), n_min=10_000, n_max=_log_int(rng, 40_000, 600_000),
                 layout=rng.randint(0, 1 << 20), backward=rng.random() < 0.5)
        return c
    top = {"order_static": 1 << 19, "gradient": 1 << 20, "individual": 1 << 21, "backward": 1 << 21}
    c["set"] = rng.choice(["uniform", "clustered"])
    c["n"] = _log_int(rng, 3_000, top.get(kind, 1 << 24))
    if kind in ("order_static", "order"):
        return c
    if kind != "individual":
        c["g"] = rng.choice([4, 8, 16, 16, 32, 64, 128])
        if c["g"] > 32:
            c["n"] = min(c["n"], _log_int(rng, 3_000, 1 << 21))
    if kind not in ("gradient", "backward"):
        c["frac"] = rng.choice([1.0, 1.0, round(rng.uniform(0.05, 0.9), 3)])
    if kind == "density":
        c["iterate"] = rng.random() < 0.4
    if kind == "hydro":
        c["balsara"] = rng.random() < 0.3
    return c


# ---------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------

def _particles(kind, n, gen, rng, dev):
    """Positions (n, 3) FP64 and the analytic number density (n,) FP64 of one set."""
    if kind == "uniform":
        pos = torch.rand((n, 3), generator=gen, device=dev, dtype=torch.float64)
        return pos, torch.full((n,), float(n), device=dev, dtype=torch.float64)
    centre = rng.random((256, 3))
    scale = np.exp(rng.uniform(math.log(0.002), math.log(0.02), 256))
    weight = rng.pareto(1.5, 256) + 1.0
    weight /= weight.sum()
    m = n - n // 2
    cen_t, a_t, cum = (torch.as_tensor(v, device=dev) for v in (centre, scale, np.cumsum(weight)))
    k = torch.searchsorted(cum, torch.rand(m, generator=gen, device=dev, dtype=torch.float64)).clamp_(max=255)
    a = a_t[k]
    # radii of a Plummer sphere cut at r = 0.25
    u = torch.rand(m, generator=gen, device=dev, dtype=torch.float64).clamp_(min=1e-9)
    u *= (1.0 + (a / 0.25) ** 2) ** -1.5
    r = a / torch.sqrt(u ** (-2.0 / 3.0) - 1.0)
    d = torch.randn((m, 3), generator=gen, device=dev, dtype=torch.float64)
    d *= (r / torch.linalg.vector_norm(d, dim=1))[:, None]
    pos = torch.empty((n, 3), device=dev, dtype=torch.float64)
    pos[:n // 2] = torch.rand((n // 2, 3), generator=gen, device=dev, dtype=torch.float64)
    pos[n // 2:] = torch.remainder(cen_t[k] + d, 1.0)
    pos[pos >= 1.0] = 0.0
    del d, r, u, a, k
    pos = pos[torch.randperm(n, generator=gen, device=dev)].contiguous()
    x, y, z = (pos[:, q].float() for q in range(3))
    dens = torch.full((n,), float(n // 2), device=dev)
    for q in range(256):
        cx, cy, cz = (float(v) for v in centre[q])
        a2 = float(scale[q]) ** 2
        r2 = sum((v - c - torch.round(v - c)).square_() for v, c in ((x, cx), (y, cy), (z, cz)))
        t = r2.div_(a2).add_(1.0).rsqrt_()
        dens += t.pow_(5).mul_(m * float(weight[q]) * 3.0 / (4.0 * math.pi * a2 ** 1.5))
    return pos, dens.double()


def _inputs(case, seed, dev):
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    rng = np.random.default_rng(seed)
    n = case["n"]
    pos, dens = _particles(case["set"], n, gen, rng, dev)
    s = _fields(n, pos, dens, gen, dev)
    s["pos"] = pos
    return s, gen


def _smoothing(pos, dens):
    """h with about 64 particles in its sphere: the counts of ever finer grids, taken at the
    particle by trilinear interpolation, give the number expected within one cell size;
    h lies where that crosses 64.  Cores too dense for the grids take the analytic density."""
    n = pos.shape[0]
    h = (3.0 * NNGB / (4.0 * math.pi * dens)) ** (1.0 / 3.0)
    found = torch.zeros(n, dtype=torch.bool, device=pos.device)
    last = torch.full_like(h, n * 4.0 * math.pi / 3.0 / 8.0)   # within half the box
    for level in range(2, 10):
        size = 1 << level
        x = pos * size - 0.5
        cell = torch.floor(x)
        w = (x - cell).float()
        i0 = torch.remainder(cell.long(), size)
        i1 = torch.remainder(i0 + 1, size)
        own = torch.floor(pos * size).long().clamp_(max=size - 1)
        count = torch.bincount((own[:, 0] * size + own[:, 1]) * size + own[:, 2], minlength=size ** 3)
        c = torch.zeros(n, device=pos.device)
        for a in range(8):
            ix, iy, iz = ((i1 if a >> q & 1 else i0)[:, q] for q in range(3))
            f = torch.ones(n, device=pos.device)
            for q in range(3):
                f *= w[:, q] if a >> q & 1 else 1.0 - w[:, q]
            c += f * count[(ix * size + iy) * size + iz]
        c = (c.double() * (4.0 * math.pi / 3.0)).clamp_(min=1e-3)
        cross = ~found & (c < NNGB)
        t = (torch.log(last) - math.log(NNGB)) / (torch.log(last) - torch.log(c)).clamp(min=1e-9)
        h = torch.where(cross, 2.0 ** (1.0 - level) * 0.5 ** t.clamp(0.0, 1.0), h)
        found |= cross
        last = c
        if 8 ** (level + 1) > 64 * n:
            break
    h = torch.where(found, h, torch.clamp(h, max=0.5 ** level))
    return h.clamp_(max=0.45)


def _fields(n, pos, dens, gen, dev):
    m = torch.full((n,), 1.0 / n, device=dev)
    h = _smoothing(pos, dens)
    vel = torch.randn((n, 3), generator=gen, device=dev) * 0.1
    u = torch.exp(torch.randn(n, generator=gen, device=dev))
    rho = (3.0 * NNGB / (4.0 * math.pi * n) / h ** 3).float() * torch.exp(0.1 * torch.randn(n, generator=gen, device=dev))
    fgrad = 1.0 + 0.1 * torch.randn(n, generator=gen, device=dev).clamp_(-3, 3)
    return {"m": m, "h": h, "vel": vel, "u": u, "rho": rho, "fgrad": fgrad}


def _active(case, s, gen, dev):
    """Active indices, ascending: every particle, or runs along the curve (mean length 32)."""
    n, frac = case["n"], case.get("frac", 1.0)
    if frac >= 1.0:
        return torch.arange(n, dtype=torch.int32, device=dev)
    perm = torch.empty(n, dtype=torch.int32, device=dev)
    s["ctx"].sfc_keys_sort(s["pos"], None, perm)
    # alternating gaps and runs with geometric lengths
    k = int(n / 32 * frac * 1.5) + 64
    u = torch.rand((2, k), generator=gen, device=dev, dtype=torch.float64).clamp_(min=1e-12)
    run = (torch.log(u[0]) / math.log(1.0 - 1.0 / 32.0)).floor_().long() + 1
    gap = (torch.log(u[1]) / math.log(1.0 - 1.0 / max(2.0, 32.0 * (1.0 - frac) / frac))).floor_().long() + 1
    end = torch.cumsum(run + gap, 0)
    at = torch.arange(n, device=dev)
    j = torch.searchsorted(end, at, right=True).clamp_(max=k - 1)
    mask = (at >= (end - run)[j]) & (at < end[j])
    mask[0] = True
    return torch.sort(perm[mask]).values.to(torch.int32).contiguous()


def _sizes(case):
    rng = np.random.default_rng(case["layout"])
    return np.exp(rng.uniform(math.log(case["n_min"]), math.log(case["n_max"]), case["boxes"])).astype(np.int64), rng


def _prepare_batch(case, seed, dev):
    sizes, rng = _sizes(case)
    kinds = ["clustered" if rng.random() < 0.5 else "uniform" for _ in sizes]
    fracs = rng.uniform(0.01, 1.0, len(sizes))
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    srng = np.random.default_rng(seed)
    parts = []
    for n, kind, frac in zip(sizes, kinds, fracs):
        pos, dens = _particles(kind, int(n), gen, srng, dev)
        f = _fields(int(n), pos, dens, gen, dev)
        f["pos"] = pos
        act = torch.rand(int(n), generator=gen, device=dev) < frac
        act[0] = True
        f["active"] = act.to(torch.uint8)
        parts.append(f)
    s = {k: torch.cat([p[k] for p in parts]).contiguous() for k in parts[0]}
    n = int(sizes.sum())
    off = np.zeros(len(sizes) + 1, dtype=np.int64)
    off[1:] = np.cumsum(sizes)
    s["batch"] = sg.Batch(off, np.array([k == "clustered" for k in kinds], dtype=np.int32), nngb_tol=TIGHT)
    s["h_guess"] = s["h"].clone()
    s["drhodh"] = torch.zeros(n, device=dev)
    s["nngb"] = torch.zeros(n, dtype=torch.int32, device=dev)
    s["acc"] = torch.zeros((n, 3), device=dev)
    s["dudt"] = torch.zeros(n, device=dev)
    if case["backward"]:
        s["g_acc"] = torch.randn((n, 3), generator=gen, device=dev)
        s["g_rho"] = torch.randn(n, generator=gen, device=dev)
        s["g_pos"] = torch.zeros((n, 3), device=dev)
        s["g_vel"] = torch.zeros((n, 3), device=dev)
        s["g_m"] = torch.zeros(n, device=dev)
    return s


def prepare(case, seed):
    dev = torch.device("cuda", torch.cuda.current_device())
    kind = case["kind"]
    if kind == "batch":
        return {"case": case, **_prepare_batch(case, seed, dev)}
    n = case["n"]
    s, gen = _inputs(case, seed, dev)
    s["case"] = case
    if kind in ("order_static", "order"):
        s["keys"] = torch.empty(n, dtype=torch.int64, device=dev)
        s["perm"] = torch.empty(n, dtype=torch.int32, device=dev)
        if kind == "order":
            s["ctx"] = sg.Context(n)
        return s
    iterate = kind == "step" or case.get("iterate", False)
    s["ctx"] = sg.Context(n, **({"nngb_tol": TIGHT} if iterate else {}))
    s["active"] = _active(case, s, gen, dev)
    if kind == "density" and iterate:
        s["h"].fill_((3.0 * NNGB / (4.0 * math.pi * n)) ** (1.0 / 3.0))
    if kind in ("gradient", "backward"):
        s["w"] = torch.randn((n, 3), generator=gen, device=dev)
        s["v"] = torch.randn(n, generator=gen, device=dev)
    if case.get("balsara"):
        s["divv"] = torch.randn(n, generator=gen, device=dev)
        s["curlv"] = torch.randn((n, 3), generator=gen, device=dev)
    if kind in ("derivs", "velocity"):
        s["o_divv"], s["o_curlv"] = torch.zeros(n, device=dev), torch.zeros((n, 3), device=dev)
    if iterate:
        s["h_work"] = s["h"].clone()
    if kind in ("density", "derivs", "step", "individual"):
        s["o_rho"], s["o_drhodh"], s["o_fgrad"] = (torch.zeros(n, device=dev) for _ in range(3))
        s["o_nngb"] = torch.zeros(n, dtype=torch.int32, device=dev)
        if kind == "step":   # particles that are not active keep their density and f
            s["o_rho"].copy_(s["rho"])
            s["o_fgrad"].copy_(s["fgrad"])
    if kind in ("hydro", "step", "individual"):
        s["o_acc"], s["o_dudt"] = torch.zeros((n, 3), device=dev), torch.zeros(n, device=dev)
        s["o_nh"] = torch.zeros(n, dtype=torch.int32, device=dev)
    if kind == "backward":
        s["o_gx"], s["o_gv"] = torch.zeros((n, 3), device=dev), torch.zeros((n, 3), device=dev)
        s["o_gm"] = torch.zeros(n, device=dev)
    if kind == "gradient":
        for k in ("pos", "vel", "m"):
            s[k].requires_grad_(True)
    elif kind != "step":
        s["ctx"].sfc_keys_sort(s["pos"])
        s["ctx"].tree_build(s["pos"], s["m"])
    return s


# ---------------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------------

def run(s):
    """Outputs of one pass.  An iterated h comes back in FP32: the iteration takes its
    Newton step on FP32 sums, its last bits carry nothing.  The neighbour count at an
    iterated h is not returned: a neighbour closer to the sphere than those bits is in
    or out by them (cases that are given h return their counts)."""
    case = s["case"]
    kind = case["kind"]
    if kind == "order_static":
        sg.sfc_keys_sort_static(s["pos"], s["keys"], s["perm"])
        return {"keys": s["keys"], "perm": s["perm"]}
    if kind == "order":
        s["ctx"].sfc_keys_sort(s["pos"], s["keys"], s["perm"])
        s["ctx"].tree_build(s["pos"], s["m"])
        return {"keys": s["keys"], "perm": s["perm"]}
    if kind == "batch":
        s["h"].copy_(s["h_guess"])
        names = ("pos", "m", "vel", "u", "h", "active", "rho", "drhodh", "fgrad", "nngb", "acc", "dudt",
                 "g_acc", "g_rho", "g_pos", "g_vel", "g_m")
        s["batch"].run({k: s[k] for k in names if k in s}, backward=case["backward"], graph=True)
        out = {k: s[k] for k in ("rho", "drhodh", "fgrad", "acc", "dudt", "g_pos", "g_vel", "g_m") if k in s}
        out["h"] = s["h"].float()
        return out
    ctx = s["ctx"]
    if kind == "density":
        if case["iterate"]:
            s["h_work"].copy_(s["h"])
            ctx.density(s["active"], s["h_work"], 1, sg.GROUPED, case["g"], s["o_rho"], s["o_drhodh"], s["o_fgrad"],
                        s["o_nngb"])
            return {"rho": s["o_rho"], "drhodh": s["o_drhodh"], "fgrad": s["o_fgrad"], "h": s["h_work"].float()}
        ctx.density(s["active"], s["h"], 0, sg.GROUPED, case["g"], s["o_rho"], s["o_drhodh"], s["o_fgrad"],
                    s["o_nngb"])
        return {"rho": s["o_rho"], "drhodh": s["o_drhodh"], "fgrad": s["o_fgrad"], "nngb": s["o_nngb"]}
    if kind == "hydro":
        ctx.hydro_force(s["active"], s["h"], s["rho"], s["fgrad"], s["vel"], s["u"], sg.GROUPED, case["g"],
                        s["o_acc"], s["o_dudt"], s["o_nh"], s.get("divv"), s.get("curlv"))
        return {"acc": s["o_acc"], "dudt": s["o_dudt"], "nngb": s["o_nh"]}
    if kind == "derivs":
        ctx.density_derivs(s["active"], s["h"], 0, case["g"], s["vel"], s["o_rho"], s["o_drhodh"], s["o_fgrad"],
                           s["o_nngb"], s["o_divv"], s["o_curlv"])
        return {"rho": s["o_rho"], "drhodh": s["o_drhodh"], "fgrad": s["o_fgrad"], "nngb": s["o_nngb"],
                "divv": s["o_divv"], "curlv": s["o_curlv"]}
    if kind == "velocity":
        ctx.velocity_derivs(s["active"], s["h"], s["rho"], s["vel"], case["g"], s["o_divv"], s["o_curlv"])
        return {"divv": s["o_divv"], "curlv": s["o_curlv"]}
    if kind == "gradient":
        acc, rho = sg.sph_forces(ctx, s["pos"], s["vel"], s["m"], s["u"], s["h"], case["g"])
        gx, gv, gm = torch.autograd.grad([acc, rho], [s["pos"], s["vel"], s["m"]], [s["w"], s["v"]])
        # the gradient is computed in FP32 and returned in the type of the positions
        return {"acc": acc.detach(), "rho": rho.detach(), "g_pos": gx.float(), "g_vel": gv, "g_m": gm}
    if kind == "backward":
        ctx.backward(s["h"], s["vel"], s["u"], s["w"], s["v"], case["g"], s["o_gx"], s["o_gv"], s["o_gm"])
        return {"g_pos": s["o_gx"], "g_vel": s["o_gv"], "g_m": s["o_gm"]}
    if kind == "individual":
        ctx.density(s["active"], s["h"], 0, sg.INDIVIDUAL, 1, s["o_rho"], s["o_drhodh"], s["o_fgrad"], s["o_nngb"])
        ctx.hydro_force(s["active"], s["h"], s["rho"], s["fgrad"], s["vel"], s["u"], sg.INDIVIDUAL, 1, s["o_acc"],
                        s["o_dudt"], s["o_nh"])
        return {"rho": s["o_rho"], "drhodh": s["o_drhodh"], "fgrad": s["o_fgrad"], "nngb": s["o_nngb"],
                "acc": s["o_acc"], "dudt": s["o_dudt"], "nngb_hydro": s["o_nh"]}
    # a timestep
    s["h_work"].copy_(s["h"])
    ctx.sfc_keys_sort(s["pos"])
    ctx.tree_build(s["pos"], s["m"])
    ctx.density(s["active"], s["h_work"], 1, sg.GROUPED, case["g"], s["o_rho"], s["o_drhodh"], s["o_fgrad"],
                s["o_nngb"])
    ctx.hydro_force(s["active"], s["h_work"], s["o_rho"], s["o_fgrad"], s["vel"], s["u"], sg.GROUPED, case["g"],
                    s["o_acc"], s["o_dudt"], s["o_nh"])
    return {"h": s["h_work"].float(), "rho": s["o_rho"], "drhodh": s["o_drhodh"], "fgrad": s["o_fgrad"],
            "acc": s["o_acc"], "dudt": s["o_dudt"]}


# ---------------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------------

# flops per neighbour pair: distance 8, kernel and sums
_PAIR = {"density": 25, "velocity": 40, "derivs": 55, "hydro": 70, "adjoint": 200}


def work(case):
    """Bytes: each input read and each output written once.  Flops: 64 neighbours per
    active particle and evaluation (about 80 under the symmetric criterion)."""
    kind = case["kind"]
    if kind == "batch":
        sizes, rng = _sizes(case)
        for _ in sizes:
            rng.random()
        n = float(sizes.sum())
        na = float((rng.uniform(0.01, 1.0, len(sizes)) * sizes).sum())
        b = n * (24 + 4 + 12 + 4 + 8 + 1 + 8) + na * (8 + 12 + 16)
        f = na * (2 * 64 * _PAIR["density"] + 80 * _PAIR["hydro"])
        if case["backward"]:
            b += n * (16 + 28)
            f += n * (64 * _PAIR["density"] + 80 * _PAIR["adjoint"] + 80 * 60)
        return {"bytes": b, "flops": f}
    n = float(case["n"])
    na = n * case.get("frac", 1.0)
    if kind in ("order_static", "order"):
        return {"bytes": n * (24 + 12 + (4 if kind == "order" else 0)), "flops": 0.0}
    if kind == "density":
        it = 3 if case["iterate"] else 1
        return {"bytes": n * (28 + 8) + na * (4 + 16 + (8 if case["iterate"] else 0)),
                "flops": na * it * 64 * _PAIR["density"]}
    if kind == "hydro":
        return {"bytes": n * (28 + 8 + 24 + (16 if case["balsara"] else 0)) + na * (4 + 20),
                "flops": na * 80 * _PAIR["hydro"]}
    if kind == "derivs":
        return {"bytes": n * (28 + 8 + 12) + na * (4 + 32), "flops": na * 64 * _PAIR["derivs"]}
    if kind == "velocity":
        return {"bytes": n * (28 + 8 + 16) + na * (4 + 16), "flops": na * 64 * _PAIR["velocity"]}
    adj = n * (64 * _PAIR["density"] + 80 * _PAIR["adjoint"] + 80 * 60)
    if kind == "backward":
        return {"bytes": n * (28 + 8 + 16 + 16 + 28), "flops": adj}
    if kind == "gradient":
        return {"bytes": n * (28 + 8 + 16 + 16 + 16 + 40), "flops": adj + n * 64 * _PAIR["density"] +
                n * 80 * _PAIR["hydro"]}
    b = n * (28 + 8 + 24) + na * (4 + 16 + 20)
    f = na * (64 * _PAIR["density"] + 80 * _PAIR["hydro"])
    if kind == "step":
        b += na * 8
        f += na * 2 * 64 * _PAIR["density"]
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------------------------
# 64-bit outputs by plain torch
# ---------------------------------------------------------------------------------

def _pairs(pos, h, rows, symmetric):
    """(i, j) of every pair with |x_i - x_j| < h_i (or max(h_i, h_j)) for i in rows."""
    x, y, z = pos.t().contiguous()
    h2 = h * h
    n = pos.shape[0]
    step = max(1, (1 << 28) // n)
    ii, jj = [], []
    for a in range(0, rows.shape[0], step):
        r = rows[a:a + step]
        d2 = None
        for v in (x, y, z):
            d = v[None, :] - v[r][:, None]
            d -= torch.round(d)
            d.mul_(d)
            d2 = d if d2 is None else d2.add_(d)
        lim = h2[r][:, None]
        i, j = torch.nonzero(d2 < (torch.maximum(lim, h2[None, :]) if symmetric else lim), as_tuple=True)
        ii.append(r[i])
        jj.append(j)
    return torch.cat(ii), torch.cat(jj)


def _shape(q):
    """w(q) of the M4 spline and dw/dq."""
    u = (1.0 - q).clamp(min=0.0)
    inner = q <= 0.5
    return (torch.where(inner, 1.0 + q * q * (6.0 * q - 6.0), 2.0 * u ** 3),
            torch.where(inner, q * (18.0 * q - 12.0), -6.0 * u * u))


def _separation(pos, i, j):
    d = pos[i] - pos[j]
    return d - torch.round(d.detach())


def _sum(n, i, v):
    out = torch.zeros((n,) + tuple(v.shape[1:]), dtype=torch.float64, device=v.device)
    return out.index_add(0, i, v)


def _radius(d):
    """|d|, with r = 0 pairs kept out of the square root's derivative."""
    r2 = (d * d).sum(1)
    zero = r2 == 0.0
    return torch.where(zero, torch.zeros_like(r2), torch.sqrt(torch.where(zero, torch.ones_like(r2), r2))), zero


def _density64(pos, m, h, i, j):
    """rho and drho/dh of the particles i occurs for (others 0)."""
    n = pos.shape[0]
    r, _ = _radius(_separation(pos, i, j))
    w, dw = _shape(r / h[i])
    s0 = _sum(n, i, m[j] * w)
    s1 = _sum(n, i, m[j] * (3.0 * w + r / h[i] * dw))
    return KERNEL / h ** 3 * s0, -KERNEL / h ** 4 * s1


def _velocity64(pos, m, h, vel, rho, i, j):
    n = pos.shape[0]
    d = _separation(pos, i, j)
    r, zero = _radius(d)
    _, dw = _shape(r / h[i])
    g = torch.where(zero, torch.zeros_like(r), KERNEL / h[i] ** 4 * dw / torch.where(zero, torch.ones_like(r), r))
    grad = g[:, None] * d
    v = vel[i] - vel[j]
    div = _sum(n, i, -m[j] * (v * grad).sum(1))
    curl = _sum(n, i, m[j][:, None] * torch.linalg.cross(v, grad))
    return div / rho, curl / rho[:, None]


def _hydro64(pos, m, h, vel, u, rho, f, limiter, i, j):
    n = pos.shape[0]
    A = f * (GAMMA - 1.0) * u / rho
    c = torch.sqrt(GAMMA * (GAMMA - 1.0) * u)
    d = _separation(pos, i, j)
    r, zero = _radius(d)
    one = torch.where(zero, torch.ones_like(r), r)
    gi = KERNEL / h[i] ** 4 * _shape(r / h[i])[1]
    gj = KERNEL / h[j] ** 4 * _shape(r / h[j])[1]
    v = vel[i] - vel[j]
    vr = (v * d).sum(1)
    hb = 0.5 * (h[i] + h[j])
    mu = hb * vr / (r * r + EPS * hb * hb)
    pi = (-ALPHA * 0.5 * (c[i] + c[j]) * mu + BETA * mu * mu) / (0.5 * (rho[i] + rho[j]))
    pi = torch.where(vr < 0.0, pi, torch.zeros_like(pi))
    if limiter is not None:
        pi = pi * 0.5 * (limiter[i] + limiter[j])
    gb = 0.5 * (gi + gj)
    zeros = torch.zeros_like(r)
    k = torch.where(zero, zeros, -m[j] * (A[i] * gi + A[j] * gj + pi * gb) / one)
    e = torch.where(zero, zeros, m[j] * (A[i] * gi + 0.5 * pi * gb) * vr / one)
    return _sum(n, i, k[:, None] * d), _sum(n, i, e)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("batch", "step", "order", "order_static") or case.get("iterate") or case["n"] > EXACT_MAX_N:
        return None
    s = prepare(case, seed)
    dev, n = s["pos"].device, case["n"]
    pos, vel, m = (s[k].detach().double() for k in ("pos", "vel", "m"))
    h, u = s["h"], s["u"].double()
    rows = s["active"].long()
    on = torch.zeros(n, dtype=torch.float64, device=dev)
    on[rows] = 1.0
    out = {}
    if kind in ("density", "derivs", "individual"):
        i, j = _pairs(pos, h, rows, False)
        rho, rh = _density64(pos, m, h, i, j)
        safe = torch.where(on > 0, rho, torch.ones_like(rho))
        out.update(rho=rho, drhodh=rh, fgrad=on / (1.0 + h * rh / (3.0 * safe)), nngb=None)
        if kind == "derivs":
            out["divv"], out["curlv"] = _velocity64(pos, m, h, vel, safe, i, j)
    if kind == "velocity":
        i, j = _pairs(pos, h, rows, False)
        out["divv"], out["curlv"] = _velocity64(pos, m, h, vel, s["rho"].double(), i, j)
    if kind in ("hydro", "individual"):
        i, j = _pairs(pos, h, rows, True)
        limiter = None
        if case.get("balsara"):
            dv, cv = s["divv"].double().abs(), torch.linalg.vector_norm(s["curlv"].double(), dim=1)
            limiter = dv / (dv + cv + 1e-4 * torch.sqrt(GAMMA * (GAMMA - 1.0) * u) / h)
        out["acc"], out["dudt"] = _hydro64(pos, m, h, vel, u, s["rho"].double(), s["fgrad"].double(), limiter, i, j)
        out["nngb" if kind == "hydro" else "nngb_hydro"] = None
    if kind in ("gradient", "backward"):
        i, j = _pairs(pos, h, rows, True)
        x, v, mm, hh = (t.clone().requires_grad_(True) for t in (pos, vel, m, h))
        close = _radius(_separation(pos, i, j))[0] < h[i]
        rho, rh = _density64(x, mm, hh, i[close], j[close])
        f = 1.0 / (1.0 + hh * rh / (3.0 * rho))
        acc, _ = _hydro64(x, mm, hh, v, u, rho, f, None, i, j)
        loss = (s["w"].double() * acc).sum() + (s["v"].double() * rho).sum()
        # h follows the relation (4 pi / 3) h^3 rho = 64 m: dh = -(dG/dh)^-1 dG
        gx, gv, gm, gh = torch.autograd.grad(loss, [x, v, mm, hh], retain_graph=True)
        rel = 4.0 * math.pi / 3.0 * hh ** 3 * rho - NNGB * mm
        lam = -gh * f.detach() / (4.0 * math.pi * h * h * rho.detach())
        ix, im = torch.autograd.grad((lam * rel).sum(), [x, mm])
        if kind == "gradient":
            out.update(acc=acc.detach(), rho=rho.detach())
        out.update(g_pos=gx + ix, g_vel=gv, g_m=gm + im)
    return out
