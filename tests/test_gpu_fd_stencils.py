"""The linear stencils of the finite-difference stage (sixth differences and first derivatives of one
variable) against extended precision, relative to the values that each of them reads."""
import numpy as np
import pytest

from gpu_util import dev, host, require_cuda
from helpers import arena, from_grid, single_level, to_grid
from paper_2608_19273_gb300 import dh, synth

pytestmark = pytest.mark.gpu

DX = 2.0 ** -4


def _stencil(G, fd_var, sigma=0.0, speed=None):
    """One stage of dq/dt + a . grad q = 0 from the field G (grid [z][y][x]) with out = L dt, dt = 1."""
    torch = require_cuda()
    n = G.shape[0]
    mesh = single_level((2, 2, 2), n // 2, DX)
    q = from_grid(mesh, G, arena(mesh, 1)[0])[None].copy()
    mat = arena(mesh, 3)
    for d, a in (speed or {}).items():
        mat[d] = a
    with dh.Plan(synth.PDE_ADV_NCP, 3, mesh.patches, 3, mesh.var_stride) as plan:
        dh.dh_plan_set_variant(plan, 2, 0, fd_var)
        d_q = dev(torch, q)
        d_out = torch.zeros_like(d_q)
        dt = torch.ones(1, dtype=torch.float64, device="cuda")
        dh.patch_update_fd_ko(plan, d_q, None, d_out, None, dev(torch, mat), dt, 0.0, 0.0, 1.0, 0.0, sigma)
        return to_grid(mesh, host(d_out)[0])


def _at(G, axis, o):
    """The field's values o voxels further along an axis of the grid."""
    return np.roll(G, -o, axis)


def _interior(G):
    """Voxels whose stencils do not reach across the periodic wrap."""
    m = np.zeros(G.shape, bool)
    m[3:-3, 3:-3, 3:-3] = True
    return m


@pytest.mark.parametrize("fd_var", [0, 2])
@pytest.mark.parametrize("kind", ["linear", "cubic", "odd", "odd_spread"])
def test_exact_zeros(kind, fd_var):
    """The weights of the sixth differences annihilate polynomials up to degree five along an axis and
    odd data about a voxel.  On integers, and on pairs +x, -x, no operation of either form rounds,
    so the result is exactly 0 also where signs mix."""
    rng = np.random.default_rng(21)
    n = 16
    k = np.arange(n) - 8.0
    z, y, x = np.meshgrid(k, k, k, indexing="ij")
    where = _interior(x)
    if kind == "linear":
        G = 3.0 * x - 2.0 * y + 5.0 * z + 1.0
    elif kind == "cubic":
        G = x ** 3 - 4.0 * y ** 3 + 2.0 * z * z - 7.0 * x + 3.0
    else:  # odd about the plane x = 0, where the centre and its neighbours along y and z are 0
        H = rng.uniform(-1.0, 1.0, (n, n, n))
        if kind == "odd_spread":
            H *= 2.0 ** rng.integers(-40, 41, H.shape)
        G = np.where(x > 0, H, 0.0)
        G[:, :, 1:8] = -G[:, :, 15:8:-1]
        where &= x == 0
    G = np.ascontiguousarray(G)
    out = _stencil(G, fd_var, sigma=0.5)
    assert np.all(out[where] == 0.0)
