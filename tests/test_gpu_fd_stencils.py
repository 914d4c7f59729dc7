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


def _field(kind, n, rng):
    G = rng.uniform(-1.0, 1.0, (n, n, n))
    if kind == "tails":  # neighbours a few binades apart
        G *= 2.0 ** rng.integers(-5, 6, G.shape)
    elif kind == "spread":
        G *= 2.0 ** rng.integers(-60, 61, G.shape)
    elif kind == "huge":
        G *= 2.0 ** 1010
    elif kind == "tiny":
        G *= 2.0 ** -980
    elif kind == "edge_low":
        G *= 2.0 ** rng.integers(-947, -940, G.shape)
    elif kind == "subnormal":
        G *= 2.0 ** -1040
    elif kind.startswith("steep"):  # a factor 2^4 from voxel to voxel along one axis
        i = np.arange(n, dtype=float).reshape([n if a == 2 - int(kind[-1]) else 1 for a in range(3)])
        G *= 2.0 ** (4 * i)
    return G


KINDS = ["unit", "tails", "spread", "huge", "tiny", "edge_low", "subnormal", "steep0", "steep1", "steep2"]


@pytest.mark.parametrize("fd_var", [0, 2])
@pytest.mark.parametrize("d", [0, 1, 2])
@pytest.mark.parametrize("kind", KINDS)
def test_derivatives(kind, d, fd_var):
    """out = -a_d D_d q / (12 dx), D q = (q_-2 - q_+2) + 8 (q_+1 - q_-1).  With M the largest magnitude of
    the four values and u = 2^-53 the FP64 form errs by at most 8 u 2M (the inner difference), 2 u M
    (the outer one) and the rounding of a result of at most 18 M: 36 u M in all.  In fixed point a term
    loses less than one unit, and the weights' magnitudes sum to 18: within that bound where the
    units are at most 2 u M.  1/(12 dx), two products and the update round once each."""
    G = _field(kind, 16, np.random.default_rng(31))
    a = 0.5
    out = _stencil(G, fd_var, speed={d: a})
    ax, u = 2 - d, np.longdouble(2.0) ** -53
    L = G.astype(np.longdouble)
    D = 8 * (_at(L, ax, 1) - _at(L, ax, -1)) + (_at(L, ax, -2) - _at(L, ax, 2))
    M = np.maximum.reduce([np.abs(_at(L, ax, o)) for o in (-2, -1, 1, 2)])
    ref = -a * D / (12 * np.longdouble(DX))
    bound = a / (12 * np.longdouble(DX)) * 36 * u * M + 5 * u * np.abs(ref) + np.longdouble(2.0) ** -1072
    assert np.all(np.abs(out - ref) <= bound)


@pytest.mark.parametrize("fd_var", [0, 2])
@pytest.mark.parametrize("kind", KINDS)
def test_sixth_differences_by_distance(kind, fd_var):
    """The FP64 form T_3 - 6 T_2 + 15 T_1, with T_r = S_r - 6c of values of magnitude at most M_r, rounds in
    each T_r by at most u (3 x 2 + 4 + 6 + 6 + 12) M_r, in the inner product by u (72 M_2 + 12 M_3) and once
    more: u (510 M_1 + 276 M_2 + 46 M_3).  The result may be no further off than that."""
    G = _field(kind, 16, np.random.default_rng(32))
    out = _stencil(G, fd_var, sigma=0.5)
    u = np.longdouble(2.0) ** -53
    L = G.astype(np.longdouble)
    ref, M = -60 * L, {}
    for r, w in ((1, 15), (2, -6), (3, 1)):
        vals = [_at(L, ax, o) for ax in range(3) for o in (-r, r)]
        ref = ref + w * sum(vals)
        M[r] = np.maximum.reduce([np.abs(v) for v in vals + [L]])
    ko = np.longdouble(0.5) / (64 * np.longdouble(DX))
    bound = ko * u * (510 * M[1] + 276 * M[2] + 46 * M[3]) + 3 * u * np.abs(ko * ref) + np.longdouble(2.0) ** -1072
    assert np.all(np.abs(out - ko * ref) <= bound)


def _fma(a, b, c):
    return (np.longdouble(a) * b.astype(np.longdouble) + c.astype(np.longdouble)).astype(np.float64)


@pytest.mark.parametrize("sigmas", [2, 6, 8, 12, 16])
def test_pulse_tail_no_further_off_than_fp64(sigmas):
    """A Gaussian pulse of width 6.4 voxels, around `sigmas` widths from its centre, where the field is
    steep along the radius: the mean error of every stencil is no larger than that of the FP64
    operations on the same values (10% for the two means being those of single samples)."""
    n = 32
    k = np.arange(n) - n / 2.0
    off = 6.4 * sigmas / np.sqrt(3.0)
    z, y, x = np.meshgrid(k + off, k + off + 0.37, k + off - 0.21, indexing="ij")
    G = np.exp(-0.5 * (x * x + y * y + z * z) / 6.4 ** 2)
    L, c = G.astype(np.longdouble), G
    where = _interior(G)
    v = [[_at(G, 2 - d, o) for o in (-3, -2, -1, 1, 2, 3)] for d in range(3)]
    V = [[a.astype(np.longdouble) for a in row] for row in v]
    two = 2.0 * c
    six = (two + two) + two
    T = [((v[0][3 - r] + v[0][2 + r]) + (v[1][3 - r] + v[1][2 + r])) + (v[2][3 - r] + v[2][2 + r]) - six for r in (1, 2, 3)]
    S = [sum(V[d][3 - r] + V[d][2 + r] for d in range(3)) for r in (1, 2, 3)]
    checks = [("sixth differences", S[2] - 6 * S[1] + 15 * S[0] - 60 * L, _fma(15.0, T[0], _fma(-6.0, T[1], T[2])),
               {"sigma": 64 * DX}, 1.0)]
    for d in range(3):
        ref = 8 * (V[d][3] - V[d][2]) + (V[d][1] - V[d][4])
        checks.append((f"derivative {d}", ref, _fma(8.0, v[d][3] - v[d][2], v[d][1] - v[d][4]), {"speed": {d: -1.0}},
                       1.0 / (12.0 * DX)))
    for what, ref, fp64, args, scale in checks:
        got = _stencil(G, 0, **args)
        err = np.abs(got - scale * ref)[where] / np.abs(L)[where]
        err64 = np.abs(fp64 * scale - scale * ref)[where] / np.abs(L)[where]
        assert err.mean() <= 1.1 * err64.mean(), f"{what}: {err.mean():.3e}, FP64 {err64.mean():.3e}"
