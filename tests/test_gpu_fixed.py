"""The fixed-point sums of the finite-difference stage at the edges of their range."""
import numpy as np
import pytest

from gpu_util import dev, host, require_cuda
from helpers import arena, from_grid, single_level, to_grid
from paper_2608_19273_gb300 import dh, synth

pytestmark = pytest.mark.gpu

WEIGHTS = {0: -20, 1: 15, 2: -6, 3: 1}


def _field(kind, n, rng):
    G = rng.uniform(-1.0, 1.0, (n, n, n))
    if kind == "spread":  # neighbours up to 2^120 apart: alignment beyond 63 bits
        G *= 2.0 ** rng.integers(-60, 61, G.shape)
    elif kind == "tails":  # neighbours a few binades apart
        G *= 2.0 ** rng.integers(-3, 4, G.shape)
    elif kind == "huge":  # beyond the fixed-point exponents: FP64 operations
        G *= 2.0 ** 1013
    elif kind == "tiny":
        G *= 2.0 ** -980
    elif kind == "edge_low":  # the smallest exponents on both sides of the rule
        G *= 2.0 ** rng.integers(-947, -940, G.shape)
    elif kind == "subnormal":
        G *= 2.0 ** -1040
    elif kind == "spike":
        G = np.where(rng.uniform(size=G.shape) < 0.02, G, 0.0)
    elif kind == "zero_sign":
        G = np.where(G < 0, -0.0, 0.0)
    return G


@pytest.mark.parametrize("fd_var", [0, 2])
@pytest.mark.parametrize("kind", ["unit", "spread", "tails", "huge", "tiny", "edge_low", "subnormal", "spike", "zero_sign"])
def test_sixth_differences(kind, fd_var):
    """out = sigma/(64 dx) sum_d delta6_d q against the same sum in extended precision.  With M the
    largest magnitude of the 19 values, their alignment costs at most 192 x 2^-54 M (the weights'
    magnitudes sum to 192, two guard bits), the FP64 form at most 8 roundings of partial sums of 18 M
    weighed by at most 15; the conversion and the product round once each."""
    torch = require_cuda()
    mesh = single_level((2, 1, 2), 8, 2.0 ** -4) if kind == "spike" else single_level((2, 2, 2), 8, 2.0 ** -4)
    if kind == "spike":
        mesh = single_level((2, 2, 2), 16, 2.0 ** -4)
    n = 16 if kind != "spike" else 32
    rng = np.random.default_rng(5)
    G = _field(kind, n, rng)
    q = from_grid(mesh, G, arena(mesh, 1)[0])[None].copy()
    sigma = 2.0 ** -3
    with dh.Plan(synth.PDE_ADV_NCP, 3, mesh.patches, 3, mesh.var_stride) as plan:
        dh.dh_plan_set_variant(plan, 2, 0, fd_var)
        d_q = dev(torch, q)
        d_out = torch.zeros_like(d_q)
        dt = torch.ones(1, dtype=torch.float64, device="cuda")
        dh.patch_update_fd_ko(plan, d_q, None, d_out, None, dev(torch, arena(mesh, 3)), dt, 0.0, 0.0, 1.0, 0.0, sigma)
        out = to_grid(mesh, host(d_out)[0])
    L = G.astype(np.longdouble)
    ref, M = np.zeros_like(L), np.abs(G)
    for ax in range(3):
        for o in range(-3, 4):
            ref += WEIGHTS[abs(o)] * np.roll(L, o, ax)
            M = np.maximum(M, np.abs(np.roll(G, o, ax)))
    ko = sigma / (64.0 * 2.0 ** -4)
    far = 192 * 2.0 ** -54 if kind not in ("huge", "tiny", "subnormal", "edge_low") else 8 * 18 * 15 * 2.0 ** -53
    bound = ko * (far * M + 2.0 ** -52 * np.abs(ref)).astype(np.longdouble) + np.longdouble(2.0) ** -1074
    assert np.all(np.abs(out - ko * ref) <= bound)
    if kind == "zero_sign":
        assert np.all(out == 0.0)


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_not_finite(bad):
    """A value that is not finite reaches exactly the results whose stencil holds it."""
    torch = require_cuda()
    mesh = single_level((2, 2, 2), 8, 2.0 ** -4)
    G = np.random.default_rng(6).uniform(-1.0, 1.0, (16, 16, 16))
    G[5, 9, 15] = bad
    q = from_grid(mesh, G, arena(mesh, 1)[0])[None].copy()
    with dh.Plan(synth.PDE_ADV_NCP, 3, mesh.patches, 3, mesh.var_stride) as plan:
        d_q = dev(torch, q)
        d_out = torch.zeros_like(d_q)
        dt = torch.ones(1, dtype=torch.float64, device="cuda")
        dh.patch_update_fd_ko(plan, d_q, None, d_out, None, dev(torch, arena(mesh, 3)), dt, 0.0, 0.0, 1.0, 0.0, 0.1)
        out = to_grid(mesh, host(d_out)[0])
    hit = np.zeros(G.shape, bool)
    for ax in range(3):
        for o in range(-3, 4):
            hit |= ~np.isfinite(np.roll(G, o, ax))
    assert np.array_equal(~np.isfinite(out), hit)
