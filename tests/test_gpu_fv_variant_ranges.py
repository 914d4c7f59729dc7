"""The first-order FV variants that a plan does not start with, at the ends of their ranges: columns of 256
planes, the edges of the number range and values that are not finite (the start variant's own tests are
in test_gpu_max_patch.py and test_gpu_stage_ranges.py)."""
import numpy as np
import pytest

from gpu_util import assert_parity, dev, host, require_cuda
from helpers import from_grid, single_level, to_grid, voxel_mask
from paper_2608_19273_gb300 import dh, synth
from test_gpu_stage_ranges import _state

pytestmark = pytest.mark.gpu


def _run(torch, mesh, q, dt, fv_var):
    with dh.Plan(synth.PDE_EULER3D, 3, mesh.patches, 1, mesh.var_stride) as plan:
        dh.dh_plan_set_variant(plan, fv_var, 0, 0)
        out = torch.zeros(q.shape, dtype=torch.float64, device="cuda")
        lam = torch.zeros(1, dtype=torch.float64, device="cuda")
        d_dt = torch.tensor([dt], dtype=torch.float64, device="cuda")
        dh.patch_update_fv(plan, dev(torch, q), None, out, None, None, d_dt, 0.0, 1.0, 1.0, 0.0, lam)
        torch.cuda.synchronize()
        assert dh.dh_plan_errors(plan) == 0
        return host(out), float(host(lam)[0])


def test_columns_of_256_planes(orc):
    """One self-periodic patch of 256^3 marched in columns of 256 planes: 16x16 with plain loads, 16x16 and
    32x8 with TMA-staged planes, and four 8x8 columns per CTA."""
    torch = require_cuda()
    p = 256
    mesh = single_level((1, 1, 1), p, 1.0 / p)
    q = orc.prim2con(synth.PDE_EULER3D, synth.euler_prims(mesh, 84), mesh.var_stride)
    ref = np.zeros_like(q)
    lam_ref = orc.stage(0, synth.PDE_EULER3D, 3, mesh.patches, 1, mesh.var_stride, q, out=ref, dt=0.2 / p, a=0, b=1,
                        g=1, want_lam=True)
    for fv_var in (2, 34, 42, 18):
        got, lam = _run(torch, mesh, q, 0.2 / p, fv_var)
        assert_parity(got, ref, voxel_mask(mesh), what=f"p=256 variant {fv_var}")
        assert abs(lam - lam_ref) <= 1e-14 * lam_ref


# tile class by class: 16x16 columns, four 8x8 columns, 32x8 columns, TMA-staged 16x16 and 32x8
TILES = {"16x16": ((1, 2, 1), 16, 2), "four 8x8": ((3, 1, 1), 8, 2), "32x8": ((1, 1, 1), 32, 10),
         "tma 16x16": ((1, 2, 1), 16, 34), "tma 32x8": ((1, 1, 1), 32, 42)}


@pytest.mark.parametrize("k", [-960, -700, 700, 1005])
@pytest.mark.parametrize("tile", list(TILES))
def test_scaled_states(orc, tile, k):
    """The Euler equations are homogeneous of degree one in Q at a fixed dt: the oracle's result at scale
    1, times 2^k."""
    torch = require_cuda()
    n, p, fv_var = TILES[tile]
    mesh = single_level(n, p, 1.0 / 32)
    q = _state(orc, mesh)
    ref = np.zeros_like(q)
    lam_ref = orc.stage(0, synth.PDE_EULER3D, 3, mesh.patches, 1, mesh.var_stride, q, out=ref, dt=1e-3, a=0, b=1, g=1,
                        want_lam=True)
    got, lam = _run(torch, mesh, np.ldexp(q, k), 1e-3, fv_var)
    assert_parity(np.ldexp(got, -k), ref, voxel_mask(mesh), what=f"{tile} 2^{k}")
    assert abs(lam - lam_ref) <= 1e-13 * lam_ref


@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("tile", list(TILES))
def test_not_finite(orc, tile, bad):
    """An energy that is not finite reaches its voxel and the voxels across its faces, and no others."""
    torch = require_cuda()
    n, p, fv_var = TILES[tile]
    mesh = single_level(n, p, 1.0 / 32)
    q = _state(orc, mesh)
    G = to_grid(mesh, q[4])
    at = (G.shape[0] - 1, p - 1, 2)
    G[at] = bad
    from_grid(mesh, G, q[4])
    got, _ = _run(torch, mesh, q, 1e-3, fv_var)
    hit = np.zeros(G.shape, bool)
    for v in range(5):
        hit |= ~np.isfinite(to_grid(mesh, got[v]))
    near = np.zeros(G.shape, bool)
    near[at] = True
    near = near | sum((np.roll(near, o, ax) for ax in range(3) for o in (-1, 1)), np.zeros(G.shape, bool))
    assert np.array_equal(hit, near)
