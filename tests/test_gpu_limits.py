"""Inputs at the limits of what the calls take: pairs closer than FP32 squares reach,
densities near the top of the FP32 range, smoothing lengths beyond half the box or not a
number, forests that outgrow their arrays, box counts around the digits of the box sort,
lists on either side of the in-group iteration's size rule, several octrees of one context,
and groups above 32 members in every grouping mode.  References are the FP64 oracle's."""

import numpy as np
import pytest

import oracle
import sphgen
from gpu_common import NEFF_TOL, RHO_TOL, Gpu, dataset

pytestmark = pytest.mark.gpu

ACC_TOL = 1e-4
GRAD_TOL = 1e-3


def _rel(a, b):
    return np.linalg.norm(np.asarray(a, np.float64) - b) / np.linalg.norm(b)


# ---------------------------------------------------------------- pairs of subnormal r^2

def _close_pairs():
    """400 particles; three pairs 1e-20 to 9e-20 apart: r^2 is a subnormal FP32 number, the
    forces of such a pair are those of the limit r -> 0."""
    rng = np.random.default_rng(sphgen.SEED_BASE + 71)
    n = 400
    pos = rng.random((n, 3))
    pos[:6] = [[0.0, 0.5, 0.5], [1e-20, 0.5, 0.5], [0.25, 0.0, 0.25], [0.25, 3e-20, 0.25], [0.0, 0.0, 0.0],
               [4e-20, 5e-20, 6e-20]]
    m = np.full(n, 1.0 / n, np.float32)
    h = oracle.h_exact(pos, m.astype(np.float64), oracle.density_iterate(pos, m, np.full(n, 0.25))[0])
    vel = (0.1 * rng.standard_normal((n, 3))).astype(np.float32)
    return pos, m, h, vel, np.ones(n, np.float32), rng


@pytest.mark.parametrize("mode,g", [(0, 1), (1, 1), (1, 16)])
def test_close_pairs_forces(cuda_device, mode, g):
    pos, m, h, vel, u, _ = _close_pairs()
    n = len(h)
    m64, v64 = m.astype(np.float64), vel.astype(np.float64)
    d = oracle.density(pos, m64, h)
    rho, f = d["rho"].astype(np.float32), d["f"].astype(np.float32)
    G = Gpu(pos, m)
    act = np.arange(n, dtype=np.int32)
    got = G.hydro(act, h, rho, f, vel, u, mode, g)
    ref = oracle.hydro(pos, v64, m64, h, rho.astype(np.float64), f.astype(np.float64), u.astype(np.float64))
    assert np.array_equal(got["nngb"], ref["nngb"])
    assert _rel(got["acc"], ref["acc"]) <= ACC_TOL and _rel(got["dudt"], ref["dudt"]) <= ACC_TOL
    if mode == 1:
        torch = G.torch
        z = lambda *s: torch.zeros(s, device=G.dev)  # noqa: E731
        rdiv, rcurl = oracle.velocity_derivs(pos, v64, m64, h, d["rho"])
        div, curl, r, dr, ff = z(n), z(n, 3), z(n), z(n), z(n)
        nn = torch.zeros(n, dtype=torch.int32, device=G.dev)
        G.ctx.velocity_derivs(G.t(act), G.t(h), G.t(rho), G.t(vel), g, div, curl)
        assert _rel(div.cpu(), rdiv) <= ACC_TOL and _rel(curl.cpu(), rcurl) <= ACC_TOL
        G.ctx.density_derivs(G.t(act), G.t(h), 0, g, G.t(vel), r, dr, ff, nn, div, curl)
        assert _rel(div.cpu(), rdiv) <= ACC_TOL and _rel(curl.cpu(), rcurl) <= ACC_TOL
    G.ctx.close()


def test_close_pairs_gradient(cuda_device):
    """Groups of one member, whose centre is the member: larger groups place such a pair at
    r = 0, where the pair's own second derivative is left out."""
    pos, m, h, vel, u, rng = _close_pairs()
    n = len(h)
    w, s = rng.standard_normal((n, 3)).astype(np.float32), rng.standard_normal(n).astype(np.float32)
    _, *ref = oracle.loss_grad(pos, vel.astype(np.float64), m.astype(np.float64), u.astype(np.float64), h,
                               w.astype(np.float64), s.astype(np.float64))
    G = Gpu(pos, m)
    for g in (1, 16):
        out = [G.torch.zeros(sh, device=G.dev) for sh in ((n, 3), (n, 3), (n,))]
        G.ctx.backward(G.t(h), G.t(vel), G.t(u), G.t(w), G.t(s), g, *out)
        for got, want, what in zip(out, ref, ("x", "v", "m")):
            got = got.cpu().numpy()
            assert np.all(np.isfinite(got)), (g, what)
            if g == 1 or what != "x":
                assert _rel(got, want) <= GRAD_TOL, (g, what)
    G.ctx.close()


# ---------------------------------------------------------------- smoothing lengths

@pytest.mark.parametrize("mode,g", [(0, 1), (1, 1), (1, 16), (1, 64)])
@pytest.mark.parametrize("n", [104, 116])
def test_iterated_h_beyond_half_the_box(cuda_device, n, mode, g):
    """So few particles that the relation holds at h between 0.4 and 0.6: the default
    iteration follows the oracle's there (an iterate accepted at the edge of the band by one
    of them and not by the other may differ: two particles are let off)."""
    rng = np.random.default_rng(sphgen.SEED_BASE + n)
    pos = rng.random((n, 3))
    m = np.full(n, 1.0 / n, np.float32)
    href, ref = oracle.density_iterate(pos, m.astype(np.float64), np.full(n, 0.3))
    assert ref["failed"] == 0 and (href > 0.5).any() and ((href > 0.49) & (href < 0.5)).any()
    G = Gpu(pos, m)
    out = G.density(np.arange(n, dtype=np.int32), np.full(n, 0.3), 1, mode, g)
    same = np.abs(out["h"] / href - 1.0) <= 1e-5
    assert same.sum() >= n - 2
    assert np.max(np.abs(out["rho"][same] / ref["rho"][same] - 1.0)) <= 5 * RHO_TOL   # rho goes as h^-3
    G.ctx.close()


@pytest.mark.parametrize("iteration", [0, 1])
def test_h_not_a_number_searches_nothing(cuda_device, iteration):
    """A NaN h is EINVAL, and no pair is found for it on the way there."""
    import paper_1810_09898_gb300 as sg

    n = 3000
    d = dataset("uniform", n, 1)
    G = Gpu(d["pos"], d["m32"], iteration=iteration)
    with pytest.raises(sg.SphgrpError, match="EINVAL"):
        G.density(np.arange(n, dtype=np.int32), np.full(n, np.nan), 1, 1, 16)
    assert G.ctx.stats()["pairs"] == 0
    out = G.density(np.arange(n, dtype=np.int32), np.full(n, d["h0"]), 0, 1, 16)   # still usable
    assert np.array_equal(out["nngb"], oracle.density(d["pos"], d["m32"].astype(np.float64), np.full(n, d["h0"]))["nngb"])
    G.ctx.close()


def test_iteration_on_both_sides_of_the_size_rule(cuda_device):
    """Lists of 4096 particles per SM iterate inside their groups, longer ones by passes:
    the same iterates, both converged under the oracle's arithmetic."""
    import torch

    edge = 4096 * torch.cuda.get_device_properties(0).multi_processor_count
    n = edge + 1000
    d = dataset("clustered", n, 2)
    G = Gpu(d["pos"], d["m32"])
    # from h around the converged ones, so that a pass or two settles most of them
    rng = np.random.default_rng(sphgen.SEED_BASE + 73)
    order = G.perm.cpu().numpy()
    h0 = np.full(n, d["h0"])
    h0 = G.density(np.arange(n, dtype=np.int32), h0, 1, 1, 16)["h"] * np.exp(0.05 * rng.standard_normal(n))
    h0 = np.minimum(h0, 0.49)
    out = [G.density(np.sort(order[:nu]).astype(np.int32), h0, 1, 1, 16) for nu in (edge, edge + 1)]
    assert out[0]["stats"]["search_launches"] == 1 and out[1]["stats"]["search_launches"] > 1
    both = order[:edge]
    a, b = (o["h"][both] for o in out)
    assert np.mean(np.abs(a / b - 1.0) <= 1e-5) > 0.999
    t = np.sort(order[rng.integers(0, edge, 2048)]).astype(np.int32)
    for o in out:
        chk = oracle.density(d["pos"], d["m32"].astype(np.float64), o["h"], targets=t)
        neff = 4.0 * np.pi / 3.0 * o["h"][t] ** 3 * chk["rho"] / d["m32"][t].astype(np.float64)
        assert np.all(np.abs(neff - 64.0) <= NEFF_TOL)
        assert np.array_equal(o["nngb"][t], chk["nngb"])
        assert np.max(np.abs(o["rho"][t] / chk["rho"] - 1.0)) <= RHO_TOL
    G.ctx.close()


# ---------------------------------------------------------------- batches

def _batch_io(pos, h):
    import torch

    n = len(pos)
    z = lambda *s: torch.zeros(s, device="cuda")  # noqa: E731
    return {"pos": torch.as_tensor(pos, device="cuda"), "m": z(n) + 1 / n, "vel": z(n, 3), "u": z(n) + 1,
            "h": torch.as_tensor(h, device="cuda"), "rho": z(n) + 1, "drhodh": z(n), "fgrad": z(n) + 1,
            "nngb": torch.zeros(n, dtype=torch.int32, device="cuda"), "acc": z(n, 3), "dudt": z(n),
            "g_acc": z(n, 3) + 1, "g_rho": z(n), "g_pos": z(n, 3), "g_vel": z(n, 3), "g_m": z(n)}


@pytest.mark.parametrize("graph", [False, True])
def test_forest_overflow_does_no_search(cuda_device, graph):
    """Chains that outgrow the forest's arrays in one of two boxes: EOVERFLOW without a
    search, whose walks would start at leaves as large as the boxes; the next call with
    positions that fit gives the oracle's counts."""
    import torch

    import paper_1810_09898_gb300 as sg

    rng = np.random.default_rng(sphgen.SEED_BASE + 74)
    k = 4000
    a = rng.random((k, 3)) * 0.99
    good = rng.random((2 * k, 3))
    pos = np.concatenate([a, a + 2.0 ** -20, good])
    n = len(pos)
    B = sg.Batch([0, 2 * k, n], leaf_size=1)
    io = _batch_io(pos, np.full(n, 0.05))
    with pytest.raises(sg.SphgrpError, match="EOVERFLOW"):
        B.run(io, backward=True, graph=graph)
    st = B.stats()
    assert st["pair_tests"] == 0 and st["walks"] == 0
    B.close()
    B = sg.Batch([0, 2 * k, n])
    io["h"].fill_(0.12)
    B.run(io, backward=True, graph=graph)
    h = io["h"].cpu().numpy()
    for s in (slice(0, 2 * k), slice(2 * k, n)):
        ref = oracle.density(pos[s], np.full(2 * k, 1 / n), h[s])
        assert np.array_equal(io["nngb"].cpu().numpy()[s], ref["nngb"])
    assert torch.isfinite(io["g_pos"]).all()
    B.close()


@pytest.mark.parametrize("nbox", [512, 513, 600, 1100])
def test_box_counts_around_the_sort_digit(cuda_device, nbox):
    """The box sort takes 9 bits of the box index a pass: one pass up to 512 boxes, two above
    (the result then ends in the other pair of buffers); every box's counts and densities
    are the oracle's on that box alone."""
    import paper_1810_09898_gb300 as sg

    rng = np.random.default_rng(sphgen.SEED_BASE + nbox)
    sizes = rng.integers(300, 500, nbox)
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    n = int(off[-1])
    pos = rng.random((n, 3))
    io = _batch_io(pos, np.full(n, 0.3))
    B = sg.Batch(off)
    B.run({k: v for k, v in io.items() if not k.startswith("g_")})
    h, rho, nn = (io[k].cpu().numpy() for k in ("h", "rho", "nngb"))
    B.close()
    for k in [*rng.integers(0, nbox, 20), 0, 255, 256, 511, nbox - 1]:
        s = slice(int(off[k]), int(off[k + 1]))
        ref = oracle.density(pos[s], np.full(sizes[k], np.float32(1 / n), np.float64), h[s])
        assert np.all(np.abs(ref["neff"] - 64.0) <= NEFF_TOL), k
        assert np.array_equal(nn[s], ref["nngb"]), k
        assert np.max(np.abs(rho[s] / ref["rho"] - 1.0)) <= RHO_TOL, k


# ---------------------------------------------------------------- octree storage

def test_rebuilds_of_one_context(cuda_device):
    """A context for 20k particles builds octrees of a few particles, of chains that outgrow
    the node arrays, and of more and fewer particles after that, on two streams."""
    import torch

    import paper_1810_09898_gb300 as sg

    rng = np.random.default_rng(sphgen.SEED_BASE + 75)
    a = rng.random((3000, 3)) * 0.99
    sets = [rng.random((300, 3)), np.concatenate([a, a + 2.0 ** -20]), rng.random((20000, 3)), rng.random((5, 3)),
            np.concatenate([a, a + 2.0 ** -20])]
    ctx = sg.Context(20000, leaf_size=1)
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    for k, pos in enumerate(sets):
        n = len(pos)
        h = np.full(n, min(0.3, (20.0 / n) ** (1 / 3)))
        with torch.cuda.stream(streams[k % 2]):
            p, m = torch.as_tensor(pos, device="cuda"), torch.full((n,), 1.0 / n, device="cuda")
            f = [torch.zeros(n, device="cuda") for _ in range(3)]
            nn = torch.zeros(n, dtype=torch.int32, device="cuda")
            act = torch.arange(n, dtype=torch.int32, device="cuda")
            ctx.sfc_keys_sort(p)
            ctx.tree_build(p, m)
            ctx.density(act, torch.as_tensor(h, device="cuda"), 0, 1, 16, *f, nn)
            got = nn.cpu().numpy()
        assert np.array_equal(got, oracle.density(pos, np.full(n, 1.0 / n), h)["nngb"]), k
    ctx.close()


# ---------------------------------------------------------------- the top of the FP32 range

@pytest.mark.parametrize("mode,g", [(0, 1), (1, 16)])
def test_viscosity_at_large_densities(cuda_device, mode, g):
    """rho_i + rho_j above 2^126, whose reciprocal is subnormal: the viscosity of cold gas."""
    rng = np.random.default_rng(sphgen.SEED_BASE + 72)
    n = 500
    pos = rng.random((n, 3))
    m = np.full(n, 1.0 / n, np.float32)
    h = np.full(n, 0.2)
    vel = (1e3 * rng.standard_normal((n, 3))).astype(np.float32)
    rho = (6e37 * (1.0 + rng.random(n))).astype(np.float32)
    zero, one = np.zeros(n, np.float32), np.ones(n, np.float32)
    ref = oracle.hydro(pos, vel.astype(np.float64), m.astype(np.float64), h, rho.astype(np.float64), one, zero)
    G = Gpu(pos, m)
    got = G.hydro(np.arange(n, dtype=np.int32), h, rho, one, vel, zero, mode, g)
    scale = 1e30   # the forces themselves are about 1e-30
    assert _rel(scale * got["acc"].astype(np.float64), scale * ref["acc"]) <= ACC_TOL
    assert _rel(scale * got["dudt"].astype(np.float64), scale * ref["dudt"]) <= ACC_TOL
    G.ctx.close()


# ---------------------------------------------------------------- groups above 32 members

@pytest.mark.parametrize("params", [{"group_mode": 1, "group_f": 2.0}, {"group_mode": 2, "group_level": 3},
                                    {"group_split": 0.0}], ids=["radius", "tree", "chunks"])
@pytest.mark.parametrize("g", [33, 64, 100, 128])
def test_large_groups_in_every_mode(cuda_device, params, g):
    """Groups of more than 32 members are searched in parts of 32."""
    d = dataset("clustered", 9001, 2)
    n = 9001
    G = Gpu(d["pos"], d["m32"], **params)
    h = np.full(n, 0.8 * d["h0"])
    act = np.sort(G.perm.cpu().numpy()[np.arange(n) % 11 < 9]).astype(np.int32)
    m64 = d["m32"].astype(np.float64)
    out = G.density(act, h, 0, 1, g)
    ref = oracle.density(d["pos"], m64, h, targets=act)
    assert np.array_equal(out["nngb"][act], ref["nngb"])
    assert np.max(np.abs(out["rho"][act] / ref["rho"] - 1.0)) <= RHO_TOL
    one = np.ones(n, np.float32)
    hy = G.hydro(act, h, one, one, d["vel32"], d["u32"], 1, g)
    href = oracle.hydro(d["pos"], d["vel32"].astype(np.float64), m64, h, one, one, d["u32"].astype(np.float64),
                        targets=act)
    assert np.array_equal(hy["nngb"][act], href["nngb"])
    assert _rel(hy["acc"][act], href["acc"]) <= ACC_TOL
    off, idx = G.ngb_sets(act, h, 1, 1, g)
    roff, ridx = oracle.ngb_sets(d["pos"], h, act, 1)
    assert np.array_equal(off, roff)
    for k in range(len(act)):
        assert np.array_equal(np.sort(idx[off[k]:off[k + 1]]), np.sort(ridx[roff[k]:roff[k + 1]]))
    G.ctx.close()
