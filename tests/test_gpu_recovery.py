"""con2prim's stopping rule on bit patterns and the split of patches over CTAs; the seed network's
training kernels at the edges of their tiles."""
import numpy as np
import pytest

from gpu_util import dev, host, require_cuda
from helpers import arena, single_level, voxel_mask
from paper_2608_19273_gb300 import dh, synth

pytestmark = pytest.mark.gpu


def _states(orc, n, seed=3):
    rng = np.random.default_rng(seed)
    W = 1 + 9 * rng.uniform(size=n)
    d = rng.normal(size=(3, n))
    v = np.sqrt(1 - 1 / W ** 2) * d / np.sqrt((d ** 2).sum(0))
    prim = np.concatenate([np.exp(rng.uniform(-2, 2, (1, n))), v, np.exp(rng.uniform(-2, 2, (1, n)))])
    return prim, orc.prim2con(synth.PDE_SRHD3D, np.ascontiguousarray(prim), n)


@pytest.mark.parametrize("tol", [0.3, 2.0 ** -8, 1e-3, 1e-6, 1e-9, 1e-12])
@pytest.mark.parametrize("seed", ["cold", "previous", "exact"])
def test_stopping_rule(orc, tol, seed):
    """Same iteration counts as the oracle's FP64 test.  The iterates agree to rounding, a few 1e-12
    relative for these states (Lorentz factors up to 10), and a step is that close to the limit in at
    most one state of a thousand for tol >= 1e-9; at 1e-12 the counts may differ by one."""
    torch = require_cuda()
    n = 4099
    prim, cons = _states(orc, n)
    prev = {"cold": None, "previous": prim[4] * 1.03, "exact": prim[4].copy()}[seed]
    ref, st_ref, it_ref, _ = orc.con2prim(cons, n, p_prev=prev, tol=tol)
    out = torch.zeros((5, n), dtype=torch.float64, device="cuda")
    st = torch.zeros(n, dtype=torch.uint8, device="cuda")
    it = torch.zeros(n, dtype=torch.int32, device="cuda")
    dh.con2prim_flat(dev(torch, cons), out, n, n, None if prev is None else dev(torch, prev), None, tol=tol,
                     status=st, iters=it)
    got, st, it = host(out), host(st), host(it)
    assert np.array_equal(st, st_ref)
    if tol >= 1e-9:
        assert np.mean(it != it_ref) <= 1e-3
    assert np.max(np.abs(it - it_ref)) <= 1
    same = it == it_ref
    assert np.max(np.abs(got[:, same] - ref[:, same]) / np.maximum(np.abs(ref[:, same]), 1e-3)) <= 1e-9


@pytest.mark.parametrize("n, p", [((2, 1, 1), 40), ((1, 1, 1), 64), ((3, 2, 1), 5), ((9, 8, 8), 8)])
def test_patch_split(orc, n, p):
    """The patch kernels cover every voxel once whatever the number of CTAs per patch: the recovery
    equals the flat one bitwise and the wave speed the oracle's."""
    torch = require_cuda()
    mesh = single_level(n, p, 1.0 / 64)
    m = voxel_mask(mesh)
    vs = mesh.var_stride
    prim, cons = _states(orc, vs)
    d_cons = dev(torch, cons)
    with dh.Plan(synth.PDE_SRHD3D, 3, mesh.patches, 1, vs) as plan:
        a = torch.full((5, vs), 7.0, dtype=torch.float64, device="cuda")
        fails = torch.zeros(1, dtype=torch.int32, device="cuda")
        dh.con2prim(plan, d_cons, a, None, None, fail_count_dev=fails)
        lam = torch.zeros(1, dtype=torch.float64, device="cuda")
        dh.max_wave_speed(plan, d_cons, a, lam)
        a, lam, fails = host(a), float(host(lam)[0]), int(host(fails)[0])
    b = torch.zeros((5, vs), dtype=torch.float64, device="cuda")
    dh.con2prim_flat(d_cons, b, vs, vs)
    assert np.array_equal(a[:, m], host(b)[:, m])
    assert np.all(a[:, ~m] == 7.0)
    assert fails == 0
    ref = orc.max_wave_speed(synth.PDE_SRHD3D, 3, mesh.patches, vs, cons, np.ascontiguousarray(a))
    assert abs(lam - ref) <= 1e-14 * ref


def _net(rng):
    w = np.zeros(1224, np.float32)
    w[:1217] = rng.normal(size=1217).astype(np.float32) * 0.3
    w[1220:1223] = 1.0
    return w


@pytest.mark.parametrize("B", [1, 63, 64, 65, 129, 517])
def test_gradient_batches(orc, B):
    """Gradient entries against the oracle's: chains of 32 FP32 products cost some 1e-5 of the largest
    entry, and the residuals, off by up to 5e-6 of themselves' scale 1, scale every entry; the partial
    rows start off a 16-byte boundary."""
    torch = require_cuda()
    rng = np.random.default_rng(B)
    w, off = _net(rng), 5
    x = rng.normal(size=(off + B, 3)).astype(np.float32)
    t = rng.normal(size=off + B).astype(np.float32)
    loss, ref = orc.mlp_loss_grad(w[:1217].astype(np.float64), x[off:].astype(np.float64), t[off:].astype(np.float64))
    part = torch.empty(((B + 63) // 64) * 1224 + 1, dtype=torch.float32, device="cuda")[1:]
    grad = torch.zeros(1224, dtype=torch.float32, device="cuda")
    dh.dh_mlp_grad(dev(torch, w), dev(torch, x), dev(torch, t), off, B, part, grad)
    g = host(grad)
    tol = 1e-5 + 5e-6 / np.sqrt(loss)
    assert abs(g[1217] - loss) <= 2 * tol * loss
    assert np.max(np.abs(g[:1217] - ref)) <= tol * np.max(np.abs(ref))


@pytest.mark.parametrize("log", [True, False])
def test_training_equals_its_parts(log):
    """Three steps of training equal gradient, loss and Adam called one by one, bit for bit."""
    torch = require_cuda()
    rng = np.random.default_rng(9)
    w0, n, B = _net(rng), 330, 129
    x, t = dev(torch, rng.normal(size=(n, 3)).astype(np.float32)), dev(torch, rng.normal(size=n).astype(np.float32))
    part = torch.empty(3 * 1224, dtype=torch.float32, device="cuda")
    new = lambda: (dev(torch, w0), torch.zeros(1224, device="cuda"), torch.zeros(1224, device="cuda"))  # noqa: E731
    w, m, v = new()
    grad, losses = torch.zeros(1224, device="cuda"), []
    for k in range(3):
        dh.dh_mlp_grad(w, x, t, (k % 2) * B, B, part, grad)
        losses.append(grad[1217].clone())
        dh.dh_mlp_adam(w, m, v, grad, k + 1)
    w2, m2, v2 = new()
    loss = torch.zeros(3, device="cuda")
    dh.dh_mlp_train(w2, m2, v2, x, t, n, B, 3, 0, 1e-3, part, grad, loss if log else None)
    assert torch.equal(w, w2) and torch.equal(m, m2) and torch.equal(v, v2)
    if log:
        assert torch.equal(loss, torch.stack(losses))
