"""Shear of a slow flow under a uniform pressure: the momentum's own fluxes are many binades below the
pressure, which acts on both faces of a voxel alike.  What the faces exchange has to be as exact
relative to the momentum as where no pressure is near, in every first- and second-order FV kernel.

Fields: rho = p = 1, momentum m along axis a only, varying along the other two and not along a.  No
velocity crosses a face that separates different m, and the faces along a see equal states, so
    out = m + dt/(2 dx) sum over b != a of s [(m_R - m_L) of the upper face - the same of the lower one],
(m_L, m_R: the voxels' values, or their limited edge values for MUSCL), s the sound speed (the flow
changes it by M^2 < u).  With u = 2^-53 each of the four face values rounds by at most 4 u |m| s, s by a
few u of itself, and with dt s/dx = 0.3 and MUSCL's differences of at most 2 |m| the update stays within
16 u of the largest |m|."""
import numpy as np
import pytest

from gpu_util import dev, host, require_cuda
from helpers import arena, from_grid, single_level, to_grid
from paper_2608_19273_gb300 import dh, synth

pytestmark = pytest.mark.gpu

U = 2.0 ** -53
# kernel: (PDE, scheme, patches per axis, patch size, fv_var)
KERNELS = {"column8": (3, 0, (2, 2, 2), 8, None), "column16": (3, 0, (1, 1, 1), 16, 2), "four columns": (3, 0, (2, 2, 2), 8, 2),
           "tma": (3, 0, (1, 1, 1), 32, 34), "generic": (3, 0, (2, 2, 2), 6, None), "muscl": (3, 2, (2, 2, 2), 8, None),
           "srhd": (5, 0, (1, 1, 1), 16, None)}


def _minmod(a, b):
    return np.where(a * b <= 0, 0, np.where(np.abs(a) < np.abs(b), a, b))


@pytest.mark.parametrize("a", [0, 1, 2])
@pytest.mark.parametrize("mach", [2.0 ** -26, 2.0 ** -30])
@pytest.mark.parametrize("kernel", list(KERNELS))
def test_shear_under_uniform_pressure(kernel, mach, a):
    torch = require_cuda()
    pde, scheme, n, p, fv_var = KERNELS[kernel]
    mesh = single_level(n, p, 2.0 ** -5)
    N = n[0] * p
    rng = np.random.default_rng(51)
    ax = 2 - a  # axis of the grid [z][y][x]
    shape = [N] * 3
    shape[ax] = 1
    m = np.broadcast_to(mach * rng.uniform(-1.0, 1.0, shape), (N, N, N)).copy()
    q = np.zeros((5, N, N, N))
    mat = None
    if pde == synth.PDE_EULER3D:
        q[0], q[4] = 1.0, 2.5
        q[1 + a] = m
        s = np.sqrt(np.longdouble(1.4))
    else:  # D = W rho, S = rho h W^2 v, tau = rho h W^2 - p - D: W = 1 to rounding
        h = 1.0 + 2.5
        q[0], q[4] = 1.0, 1.5
        q[1 + a] = m
        w = np.zeros_like(q)
        w[0], w[4] = 1.0, 1.0
        w[1 + a] = m / h
        mat = np.stack([from_grid(mesh, g, arena(mesh, 1)[0]) for g in w])
        s = np.sqrt(np.longdouble(5.0) / 3 / np.longdouble(h))
    Q = np.stack([from_grid(mesh, np.ascontiguousarray(g), arena(mesh, 1)[0]) for g in q])
    dx, dt = 2.0 ** -5, 0.3 * 2.0 ** -5 / float(s)
    with dh.Plan(pde, 3, mesh.patches, 2 if scheme == 2 else 1, mesh.var_stride) as plan:
        if fv_var is not None:
            dh.dh_plan_set_variant(plan, fv_var, 0, 0)
        out = torch.zeros(Q.shape, dtype=torch.float64, device="cuda")
        d_dt = torch.tensor([dt], dtype=torch.float64, device="cuda")
        f = dh.patch_update_fv_muscl if scheme == 2 else dh.patch_update_fv
        f(plan, dev(torch, Q), None, out, None, None if mat is None else dev(torch, mat), d_dt, 0.0, 1.0, 1.0, 0.0)
        got = to_grid(mesh, host(out)[1 + a])
    L = m.astype(np.longdouble)
    ref = L.copy()
    for b in range(3):
        if b == ax:
            continue
        up, dn = np.roll(L, -1, b), np.roll(L, 1, b)
        sig = _minmod(L - dn, up - L) if scheme == 2 else np.zeros_like(L)
        jump = (up - np.roll(sig, -1, b) / 2) - (L + sig / 2)  # of the upper face
        ref += np.longdouble(dt) / (2 * np.longdouble(dx)) * s * (jump - np.roll(jump, 1, b))
    assert np.max(np.abs(got - ref)) <= 16 * U * np.max(np.abs(m))


@pytest.mark.parametrize("kernel", [k for k in KERNELS if k != "srhd"])
def test_contact_at_rest_is_kept(kernel):
    """A density that varies under a uniform pressure with no flow: only the density changes.  The energy's
    face value Q_L (u_L + s) + Q_R (u_R - s) is there the rounding of E s, at most u E s, and with
    dt s/dx <= 1/6 the six of a voxel move the energy by at most 6 x u E s x dt/(2 dx) <= u E/2, no more than
    half a unit in its last place: the update rounds to the same energy, and the momentum stays exactly 0."""
    torch = require_cuda()
    pde, scheme, n, p, fv_var = KERNELS[kernel]
    mesh = single_level(n, p, 2.0 ** -5)
    N = n[0] * p
    rho = np.random.default_rng(52).uniform(0.5, 1.5, (N, N, N))
    q = np.zeros((5, N, N, N))
    q[0], q[4] = rho, 2.6875
    Q = np.stack([from_grid(mesh, np.ascontiguousarray(g), arena(mesh, 1)[0]) for g in q])
    s_max = np.sqrt(1.4 * 0.4 * 2.6875 / rho.min())
    with dh.Plan(pde, 3, mesh.patches, 2 if scheme == 2 else 1, mesh.var_stride) as plan:
        if fv_var is not None:
            dh.dh_plan_set_variant(plan, fv_var, 0, 0)
        out = torch.zeros(Q.shape, dtype=torch.float64, device="cuda")
        d_dt = torch.tensor([0.16 * 2.0 ** -5 / s_max], dtype=torch.float64, device="cuda")
        f = dh.patch_update_fv_muscl if scheme == 2 else dh.patch_update_fv
        f(plan, dev(torch, Q), None, out, None, None, d_dt, 0.0, 1.0, 1.0, 0.0)
        got = np.stack([to_grid(mesh, g) for g in host(out)])
    assert np.array_equal(got[1:], q[1:])
    assert not np.array_equal(got[0], rho)
