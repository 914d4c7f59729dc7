"""The second-order FV stage's two forms of an edge state (momenta squared first where density and energy of
all of a tile's voxels and halos lie within 2^-500 and 2^500, velocities first elsewhere), side by side in
one launch, and the values that its variant call takes."""
import numpy as np
import pytest

from gpu_util import dev, host, require_cuda
from helpers import single_level, to_grid
from paper_2608_19273_gb300 import dh, synth
from test_gpu_stage_ranges import _state

pytestmark = pytest.mark.gpu


def _near_max(G):
    """The largest magnitude among the voxels that the stencil of a voxel reads."""
    G = np.abs(G)
    M = G.copy()
    for ax in range(3):
        for o in (-2, -1, 1, 2):
            M = np.maximum(M, np.roll(G, o, ax))
    return M


@pytest.mark.parametrize("k", [-600, 520, 600])
def test_tiles_of_both_forms(orc, k):
    """Four patches of 8^3 in a row, the first scaled by 2^k: its tiles and those of its neighbours, which read
    it, take one form, the third patch's the other.  Every value is compared with the oracle's relative
    to the largest value that its stencil reads (1e-12, as the other stage tests), with q0 and acc."""
    torch = require_cuda()
    mesh = single_level((4, 1, 1), 8, 1.0 / 32)
    q, q0 = _state(orc, mesh), _state(orc, mesh, seed=12)
    first = slice(int(mesh.patches[0]["offset"]), int(mesh.patches[0]["offset"]) + 512)
    q[:, first] = np.ldexp(q[:, first], k)
    q0[:, first] = np.ldexp(q0[:, first], k)
    acc0 = q0.copy()
    a, b, g, d = 0.75, 0.25, 0.25, 1 / 6
    ref, ref_acc = np.zeros_like(q), acc0.copy()
    orc.stage(2, synth.PDE_EULER3D, 3, mesh.patches, 2, mesh.var_stride, q, q0=q0, out=ref, acc=ref_acc, dt=1e-3, a=a, b=b,
              g=g, d=d)
    assert np.all(np.isfinite(ref))
    with dh.Plan(synth.PDE_EULER3D, 3, mesh.patches, 2, mesh.var_stride) as plan:
        out, acc = torch.zeros(q.shape, dtype=torch.float64, device="cuda"), dev(torch, acc0)
        d_dt = torch.tensor([1e-3], dtype=torch.float64, device="cuda")
        dh.patch_update_fv_muscl(plan, dev(torch, q), dev(torch, q0), out, acc, None, d_dt, a, b, g, d)
        got, got_acc = host(out), host(acc)
    scale = np.max([_near_max(to_grid(mesh, q[v])) for v in range(5)], axis=0)
    for v in range(5):
        for x, r in ((got, ref), (got_acc, ref_acc)):
            assert np.all(np.abs(to_grid(mesh, x[v]) - to_grid(mesh, r[v])) <= 1e-12 * scale)


def test_variant_values():
    require_cuda()
    mesh = single_level((2, 2, 2), 8, 1.0 / 32)
    with dh.Plan(synth.PDE_EULER3D, 3, mesh.patches, 2, mesh.var_stride) as plan:
        for v in (0, 1, 2):
            dh.dh_plan_set_variant_muscl(plan, v)
        for v in (-1, 3):
            with pytest.raises(dh.DhError):
                dh.dh_plan_set_variant_muscl(plan, v)
