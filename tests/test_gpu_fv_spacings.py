"""Levels that share a patch size but not a spacing, in the first-order FV stage.

A 256-thread tile of 8x8 columns takes four columns of up to four patches, which the work lists put
together by patch size alone: with these meshes one tile holds columns of two spacings.  Every
patch has to be advanced with its own dx, within the 1e-12 rule of the other stage tests."""
import numpy as np
import pytest

from gpu_util import assert_parity, dev, host, require_cuda
from helpers import voxel_mask
from paper_2608_19273_gb300 import dh, synth

pytestmark = pytest.mark.gpu

# 27 + 8 patches of one column (the seventh tile: three columns of the first level, one of the
# second); 1 + 1 patches of nine columns (the third tile: one and three)
MESHES = {"p8": [synth.Level((3, 3, 3), 8, 1.0 / 64, 0), synth.Level((2, 2, 2), 8, 1.0 / 128, 1)],
          "p24": [synth.Level((1, 1, 1), 24, 1.0 / 64, 0), synth.Level((1, 1, 1), 24, 1.0 / 128, 1)]}


def _state(orc, pde, mesh, seed):
    """(conserved state, material arena or None)"""
    if pde == synth.PDE_SRHD3D:
        prim = synth.srhd_initial(mesh, seed, wmax=3.0)
        return orc.prim2con(pde, prim, mesh.var_stride), prim
    if pde in (synth.PDE_ADV_FLUX, synth.PDE_ADV_NCP):
        rng = np.random.default_rng(seed)
        return rng.uniform(0.5, 1.5, (1, mesh.var_stride)), rng.uniform(-1.0, 1.0, (3, mesh.var_stride))
    return orc.prim2con(pde, synth.euler_prims(mesh, seed), mesh.var_stride), None


def _stage_check(orc, pde, dim, mesh, fv_var, what):
    torch = require_cuda()
    qs, mat = _state(orc, pde, mesh, 41)
    q0, _ = _state(orc, pde, mesh, 42)
    acc0 = np.random.default_rng(43).normal(size=qs.shape)
    ref, ref_acc = np.zeros_like(qs), acc0.copy()
    orc.stage(0, pde, dim, mesh.patches, 1, mesh.var_stride, qs, q0=q0, out=ref, acc=ref_acc, mat=mat, dt=1e-3, a=0.75,
              b=0.25, g=0.25, d=1 / 6)
    with dh.Plan(pde, dim, mesh.patches, 1, mesh.var_stride) as plan:
        if fv_var is not None:
            dh.dh_plan_set_variant(plan, fv_var, 0, 0)
        out, acc = torch.zeros(qs.shape, dtype=torch.float64, device="cuda"), dev(torch, acc0)
        d_dt = torch.tensor([1e-3], dtype=torch.float64, device="cuda")
        dh.patch_update_fv(plan, dev(torch, qs), dev(torch, q0), out, acc, None if mat is None else dev(torch, mat), d_dt,
                           0.75, 0.25, 0.25, 1 / 6)
        got, got_acc = host(out), host(acc)
    m = voxel_mask(mesh)
    assert_parity(got, ref, m, what=f"{what} out")
    assert_parity(got_acc, ref_acc, m, what=f"{what} acc")


# None: the variant that a plan starts with; then every kernel form, the persistent grid (4) and every
# tile set (bits 3-4)
@pytest.mark.parametrize("fv_var", [None, 0, 1, 2, 3, 6, 7, 10, 11, 14, 16, 18, 22, 26])
@pytest.mark.parametrize("name", list(MESHES))
def test_euler3d_stage_two_spacings(orc, name, fv_var):
    mesh = synth.make_mesh(MESHES[name], dim=3)
    _stage_check(orc, synth.PDE_EULER3D, 3, mesh, fv_var, f"{name} variant {fv_var}")


@pytest.mark.parametrize("pde", [synth.PDE_ADV_FLUX, synth.PDE_ADV_NCP, synth.PDE_SRHD3D, synth.PDE_EULER2D])
def test_other_systems_two_spacings(orc, pde):
    dim = 2 if pde == synth.PDE_EULER2D else 3
    levels = MESHES["p8"]
    if dim == 2:
        levels = [synth.Level((3, 3, 1), 8, 1.0 / 64, 0), synth.Level((2, 2, 1), 8, 1.0 / 128, 1)]
    _stage_check(orc, pde, dim, synth.make_mesh(levels, dim=dim), 2, f"pde {pde}")


@pytest.mark.parametrize("name", list(MESHES))
def test_noalloc_two_spacings(orc, name):
    torch = require_cuda()
    mesh = synth.make_mesh(MESHES[name], dim=3)
    qs, _ = _state(orc, synth.PDE_EULER3D, mesh, 44)
    ref = np.zeros_like(qs)
    orc.stage(0, synth.PDE_EULER3D, 3, mesh.patches, 1, mesh.var_stride, qs, out=ref, dt=1e-3, a=0, b=1, g=1)
    out = torch.zeros(qs.shape, dtype=torch.float64, device="cuda")
    d_dt = torch.tensor([1e-3], dtype=torch.float64, device="cuda")
    dh.patch_update_fv_noalloc(3, 3, mesh.patches, mesh.var_stride, None, dev(torch, qs), None, out, None, None, d_dt,
                               0.0, 1.0, 1.0, 0.0)
    torch.cuda.synchronize()
    assert_parity(host(out), ref, voxel_mask(mesh), what=f"noalloc {name}")


@pytest.mark.parametrize("fv_var", [2, 6, 10, 18])
@pytest.mark.parametrize("coupled", [False, True])
def test_steps_two_spacings(orc, coupled, fv_var):
    """Two SSP-RK3 steps, levels by themselves (stage-sum form, W handed over) and coupled with
    reflux and restriction: 125 coarse patches, so that the first fine ones share a tile with the last."""
    torch = require_cuda()
    mesh = synth.coupled_mesh(5, 8, 1.0 / 40, 1, 2) if coupled else synth.make_mesh(MESHES["p8"], dim=3)
    if coupled:
        prim = synth.coupled_fields(mesh, np.random.default_rng(45), [(1.0, 0.5)] + [(0.0, 0.5)] * 3 + [(1.0, 0.5)])
        q = orc.prim2con(synth.PDE_EULER3D, prim, mesh.var_stride)
    else:
        q, _ = _state(orc, synth.PDE_EULER3D, mesh, 45)
    ref = q.copy()
    orc.rk_steps(0, synth.PDE_EULER3D, 3, mesh.patches, 1, mesh.var_stride, ref, rk=3, steps=2, cfl=0.4)
    with dh.Plan(synth.PDE_EULER3D, 3, mesh.patches, 1, mesh.var_stride) as plan:
        dh.dh_plan_set_variant(plan, fv_var, 0, 0)
        Q = dev(torch, q)
        U1, U2 = torch.zeros_like(Q), torch.zeros_like(Q)
        R = None if coupled else torch.zeros_like(Q)
        lam = torch.zeros(1, dtype=torch.float64, device="cuda")
        dt = torch.zeros(1, dtype=torch.float64, device="cuda")
        dh.max_wave_speed(plan, Q, None, lam)
        for _ in range(2):
            dh.dh_rk_step(plan, 0, 3, Q, U1, U2, R, None, dt, lam, 0.4, 0.0)
        got = host(Q)
    assert_parity(got, ref, voxel_mask(mesh), what=f"steps, coupled={coupled}, variant {fv_var}")
