"""Inputs at the limits of what the calls take.  References are the FP64 oracle's."""

import numpy as np
import pytest

import oracle
import sphgen
from gpu_common import Gpu

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
