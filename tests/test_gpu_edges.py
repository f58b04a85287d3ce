"""Sizes at which the search's parts meet: group parts of 32 members, slices of every member
count, whole nodes and leaf sizes, tiles that fill, pieces beside a dense clump, sort tiles,
octree chains and capacity.  Keys, order, counts and neighbour sets are compared bit for bit
with the oracle, the density within the usual 1e-5."""

import numpy as np
import pytest

import oracle
import sphgen
from gpu_common import RHO_TOL, Gpu

pytestmark = pytest.mark.gpu


def _clump(n, seed=1):
    """Nine tenths of the particles in a ball of radius 0.004, the rest spread over the box,
    some of them at the ball's edge; h that of 50 neighbours in the ball, and outside it from
short of the ball to half way through it."""
    rng = np.random.default_rng(sphgen.SEED_BASE + seed)
    d = rng.standard_normal((n, 3))
    d /= np.linalg.norm(d, axis=1)[:, None]
    nd = 9 * n // 10
    r = np.where(np.arange(n) < nd, 0.004 * rng.random(n) ** (1 / 3), 0.004 + 0.3 * rng.random(n) ** 2)
    pos = np.mod(np.array([0.5, 0.497, 0.01]) + d * r[:, None], 1.0)
    h = np.where(np.arange(n) < nd, 0.004 * (50.0 / nd) ** (1 / 3), np.maximum(r + 0.008 * (rng.random(n) - 0.75), 0.001))
    m = np.full(n, 1.0 / n, dtype=np.float32)
    return pos, m, np.minimum(h, 0.2)


def _check(pos, m32, h, act, g, **params):
    G = Gpu(pos, m32, **params)
    ref = oracle.density(pos, m32.astype(np.float64), h, targets=act)
    out = G.density(act, h, 0, 1, g)
    assert np.array_equal(out["nngb"][act], ref["nngb"])
    assert np.max(np.abs(out["rho"][act] / ref["rho"] - 1.0)) <= RHO_TOL
    off, idx = G.ngb_sets(act, h, 1, 1, g)
    roff, ridx = oracle.ngb_sets(pos, h, act, 1)
    assert np.array_equal(off, roff)
    for k in range(len(act)):
        assert np.array_equal(np.sort(idx[off[k]:off[k + 1]]), np.sort(ridx[roff[k]:roff[k + 1]]))
    hy = oracle.hydro(pos, np.zeros_like(pos), m32.astype(np.float64), h, np.ones(len(h)), np.ones(len(h)),
                      np.ones(len(h)), targets=act)
    got = G.hydro(act, h, np.ones(len(h), np.float32), np.ones(len(h), np.float32),
                  np.zeros((len(h), 3), np.float32), np.ones(len(h), np.float32), 1, g)
    assert np.linalg.norm(got["acc"][act] - hy["acc"]) <= 1e-4 * np.linalg.norm(hy["acc"])
    G.ctx.close()


@pytest.mark.parametrize("g", [1, 2, 3, 5, 7, 11, 16, 31, 32, 33, 100, 128])
def test_group_sizes_beside_a_clump(cuda_device, g):
    """Outer particles whose dilated box covers the clump (the walk's member test), groups of
    every slice count, parts of 32, and a ragged active list."""
    pos, m32, h = _clump(12_007)
    act = np.sort(np.concatenate([np.arange(0, 10_806, 37), np.arange(10_806, 12_007)])).astype(np.int32)
    _check(pos, m32, h, act, g)


@pytest.mark.parametrize("leaf", [1, 2, 7, 16, 33, 300, 1024])
def test_leaf_sizes(cuda_device, leaf):
    """Leaves of one particle (more than 32 ranges pending), beyond the whole-node size, and
    larger than most cells; with coincident particles."""
    d = sphgen.make("clustered", 5003, config=2)
    pos = d["pos"].copy()
    pos[100:160] = pos[100]
    h = np.full(5003, 0.6 * d["h0"])
    _check(pos, d["m"].astype(np.float32), h, np.arange(0, 5003, 3, dtype=np.int32), 16, leaf_size=leaf)


def test_octree_chains_outgrow_the_first_capacity(cuda_device):
    """Pairs 2^-20 apart with leaves of one particle: chains of 20 levels under every pair,
    more nodes than the build first makes room for."""
    rng = np.random.default_rng(sphgen.SEED_BASE + 3)
    a = rng.random((1500, 3)) * 0.99
    pos = np.concatenate([a, a + 2.0 ** -20])
    _check(pos, np.full(3000, 1 / 3000, np.float32), np.full(3000, 0.08), np.arange(0, 3000, 2, dtype=np.int32), 16,
           leaf_size=1)


def test_forest_beyond_its_capacity_is_an_error(cuda_device):
    """The batch's node arrays are fixed: the same chains there are EOVERFLOW."""
    import torch

    import paper_1810_09898_gb300 as sg

    rng = np.random.default_rng(sphgen.SEED_BASE + 3)
    a = rng.random((1500, 3)) * 0.99
    n = 3000
    B = sg.Batch([0, n], leaf_size=1)
    dev = "cuda"
    z = lambda *s: torch.zeros(s, device=dev)  # noqa: E731
    io = {"pos": torch.as_tensor(np.concatenate([a, a + 2.0 ** -20]), device=dev), "m": z(n) + 1 / n, "vel": z(n, 3),
          "u": z(n) + 1, "h": torch.full((n,), 0.08, dtype=torch.float64, device=dev), "rho": z(n) + 1, "drhodh": z(n),
          "fgrad": z(n) + 1, "nngb": torch.zeros(n, dtype=torch.int32, device=dev), "acc": z(n, 3), "dudt": z(n)}
    with pytest.raises(sg.SphgrpError, match="EOVERFLOW"):
        B.run(io)
    B.close()


@pytest.mark.parametrize("n", [1, 2, 255, 256, 257, 1023, 1024, 1025, (1 << 17) - 1, 1 << 17, (1 << 17) + 1,
                               (1 << 20) - 1, 1 << 20, (1 << 20) + 4097])
def test_sort_sizes(cuda_device, n):
    """Edges of the radix tiles and of the tile-size rule; a twentieth of the particles share
    cells (stable order), in both entry points."""
    import torch

    import paper_1810_09898_gb300 as sg

    rng = np.random.default_rng(sphgen.SEED_BASE + n)
    pos = rng.random((n, 3))
    k = n // 20
    pos[:k] = pos[rng.integers(0, n, k)]
    ref = oracle.hilbert_keys(pos)
    order = oracle.stable_order(ref)
    p = torch.as_tensor(pos, device="cuda")
    keys = torch.empty(n, dtype=torch.int64, device="cuda")
    perm = torch.empty(n, dtype=torch.int32, device="cuda")
    ctx = sg.Context(n)
    calls = [lambda: ctx.sfc_keys_sort(p, keys, perm)]
    if n <= 1 << 19:
        calls.append(lambda: sg.sfc_keys_sort_static(p, keys, perm))
    for call in calls:
        keys.zero_()
        perm.zero_()
        call()
        assert np.array_equal(perm.cpu().numpy(), order)
        assert np.array_equal(keys.cpu().numpy().astype(np.uint64), ref[order])
    ctx.close()


def test_individual_walks_are_counted_once(cuda_device):
    """stats: one walk per particle and pass in the individual form, both loops."""
    d = sphgen.make("uniform", 3001, config=1)
    G = Gpu(d["pos"], d["m"].astype(np.float32))
    act = np.arange(0, 3001, 2, dtype=np.int32)
    h = np.full(3001, d["h0"])
    st = G.density(act, h, 0, 0, 1)["stats"]
    assert st["walks"] == st["members"] == len(act)
    st = G.density(act, h, 1, 0, 1)["stats"]
    assert st["walks"] == st["members"] > len(act)
    one = np.ones(3001, np.float32)
    st = G.hydro(act, h, one, one, np.zeros((3001, 3), np.float32), one, 0, 1)["stats"]
    assert st["walks"] == st["members"] == len(act)
    G.ctx.close()
