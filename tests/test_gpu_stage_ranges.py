"""The finite-volume stages (marching, generic, MUSCL) at the edges of the number range and with
values that are not finite.

The sums over a voxel's faces are formed in fixed point where the terms' exponents allow it and in
FP64 elsewhere, and the MUSCL edge states square their momenta only in the middle of the range.  The
Euler equations are homogeneous of degree one in Q at a fixed dt, so the oracle's result at scale 1,
times 2^k, is the reference at every scale, within the 1e-12 rule of the other stage tests."""
import numpy as np
import pytest

from gpu_util import assert_parity, dev, host, require_cuda
from helpers import arena, from_grid, single_level, to_grid, voxel_mask
from paper_2608_19273_gb300 import dh, synth

pytestmark = pytest.mark.gpu

# stage: (scheme of the oracle, halo, patches per axis, patch size)
STAGES = {"march8": (0, 1, (2, 2, 2), 8), "march16": (0, 1, (1, 2, 1), 16), "generic6": (0, 1, (3, 2, 2), 6),
          "generic5": (0, 1, (2, 3, 1), 5), "muscl8": (2, 2, (2, 2, 2), 8)}


def _state(orc, mesh, seed=11):
    rng = np.random.default_rng(seed)
    m = voxel_mask(mesh)
    n = int(m.sum())
    prim = arena(mesh, 5)
    prim[0, m] = rng.uniform(0.5, 1.5, n)
    prim[1:4, m] = rng.uniform(-1.0, 1.0, (3, n))
    prim[4, m] = rng.uniform(0.5, 1.5, n)
    return orc.prim2con(synth.PDE_EULER3D, prim, mesh.var_stride)


def _run(torch, mesh, scheme, halo, q, dt):
    with dh.Plan(synth.PDE_EULER3D, 3, mesh.patches, halo, mesh.var_stride) as plan:
        out = torch.zeros(q.shape, dtype=torch.float64, device="cuda")
        lam = torch.zeros(1, dtype=torch.float64, device="cuda")
        d_dt = torch.tensor([dt], dtype=torch.float64, device="cuda")
        f = dh.patch_update_fv_muscl if scheme == 2 else dh.patch_update_fv
        f(plan, dev(torch, q), None, out, None, None, d_dt, 0.0, 1.0, 1.0, 0.0, lam)
        return host(out), float(host(lam)[0])


@pytest.mark.parametrize("k", [-960, -700, -300, 300, 700, 1005])
@pytest.mark.parametrize("stage", list(STAGES))
def test_scaled_states(orc, stage, k):
    torch = require_cuda()
    scheme, halo, n, p = STAGES[stage]
    mesh = single_level(n, p, 1.0 / 32)
    q = _state(orc, mesh)
    ref = np.zeros_like(q)
    lam_ref = orc.stage(scheme, synth.PDE_EULER3D, 3, mesh.patches, halo, mesh.var_stride, q, out=ref, dt=1e-3,
                        a=0, b=1, g=1, want_lam=True)
    got, lam = _run(torch, mesh, scheme, halo, np.ldexp(q, k), 1e-3)
    assert_parity(np.ldexp(got, -k), ref, voxel_mask(mesh), what=f"{stage} 2^{k}")
    assert abs(lam - lam_ref) <= 1e-13 * lam_ref


@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("stage", list(STAGES))
def test_not_finite(orc, stage, bad):
    """An energy that is not finite reaches its voxel and the voxels across its faces, and none outside
    the stencil (MUSCL: two voxels along each axis)."""
    torch = require_cuda()
    scheme, halo, n, p = STAGES[stage]
    mesh = single_level(n, p, 1.0 / 32)
    q = _state(orc, mesh)
    G = to_grid(mesh, q[4])
    at = (G.shape[0] - 1, p - 1, 2)  # next to a patch boundary and the periodic wrap
    G[at] = bad
    from_grid(mesh, G, q[4])
    got, _ = _run(torch, mesh, scheme, halo, q, 1e-3)
    hit = np.zeros(G.shape, bool)
    for v in range(5):
        hit |= ~np.isfinite(to_grid(mesh, got[v]))
    centre = np.zeros(G.shape, bool)
    centre[at] = True
    near, far = centre.copy(), centre.copy()
    for ax in range(3):
        for o in (-1, 1):
            near |= np.roll(centre, o, ax)
            far |= np.roll(centre, o, ax) | (np.roll(centre, 2 * o, ax) if scheme == 2 else centre)
    assert np.all(hit[near])
    assert not np.any(hit[~far])
