"""The work that a user of the library has it do, as cases that can be timed.

Every case goes through the public entry points of ``paper_2608_19273_gb300.dh`` on a plan with its
default kernels (no tuner), as a program that has just created its plan runs it.  Inputs are smooth
seeded fields made on the GPU.  ``exact`` states the same step in plain torch in 64 bits on the
global periodic grid of each level, without the library.

Meshes are texts, one term per refinement level: ``"16x8x8:16:128"`` is a periodic box of 16 x 8 x 8
patches of 16 voxels per axis with a voxel spacing of 1/128 (2D: ``"8x8:16:128"``).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2608_19273_gb300 import dh, synth

DEV = "cuda"
F64 = torch.float64
GAMMA_E, GAMMA_R = 1.4, 5.0 / 3.0   # ratio of specific heats: Euler, relativistic
DAMP, KAPPA, SIGMA = 0.1, 0.1, 0.1  # wave damping, lapse coupling, Kreiss-Oliger strength
CFL_FV, CFL_FD = 0.4, 0.25

# FP64 operations per voxel and whole time step (add, sub, mul, div, sqrt = 1; halo work excluded)
FLOPS = {("euler2", 1): 114, ("euler3", 3): 534, ("muscl3", 3): 1107, ("wave", 4): 1103, ("gw59", 4): 17472,
         ("srhd", 3): 671 + 3 * 72 + 30}


# --------------------------------------------------------------------------- the cases
def listed():
    return [
        # 2D Euler on 64 patches of 16^2, ten forward-Euler steps replayed as one graph: the smallest
        # problem, where launches and latency count
        {"name": "euler2d_small", "kind": "euler", "dim": 2, "scheme": 0, "rk": 1, "steps": 10, "graph": True,
         "levels": "8x8:16:128"},
        # 3D Euler on the AMR-like mix of 8^3, 16^3 and 32^3 patches (10.5 M voxels), two SSP-RK3 steps
        # replayed as a graph: the library's main use
        {"name": "euler3d_mix", "kind": "euler", "dim": 3, "scheme": 0, "rk": 3, "steps": 2, "graph": True,
         "levels": "16x16x16:8:128,16x8x8:16:128,8x4x4:32:128"},
        # 3D Euler on 16,384 cells of 6^3 voxels, the paper's typical cell size (not a multiple of 8)
        {"name": "euler3d_cells6", "kind": "euler", "dim": 3, "scheme": 0, "rk": 3, "steps": 2, "graph": True,
         "levels": "32x32x16:6:192"},
        # second-order (MUSCL) 3D Euler on the mix with a quarter of its patches, one step called eagerly
        {"name": "euler3d_muscl", "kind": "euler", "dim": 3, "scheme": 2, "rk": 3, "steps": 1, "graph": False,
         "levels": "16x8x8:8:128,8x8x4:16:128,4x4x2:32:128"},
        # 3D Euler on two coupled refinement levels (prolongation, reflux, restriction), two steps as a graph
        {"name": "euler3d_coupled", "kind": "coupled", "nc": 8, "p": 16, "lo": 2, "m": 4, "steps": 2},
        # damped wave system with variable speed, FD4 + Kreiss-Oliger, one RK4 step on 2048 patches of 16^3
        {"name": "wave3d", "kind": "wave", "steps": 1, "levels": "16x16x8:16:128"},
        # the 59-unknown gravitational-wave system on patches of 24^3 and 16^3 (3.8 M voxels), one RK4 step
        {"name": "gw59", "kind": "gw59", "steps": 1, "levels": "4x4x4:24:192,6x6x6:16:192,8x8x8:16:256"},
        # relativistic hydro, one SSP-RK3 step with its recoveries and wave speed on 4096 patches of 16^3
        {"name": "srhd3d", "kind": "srhd", "steps": 1, "levels": "16x16x16:16:256"},
        # con2prim of a million independent states (initial data, tables) with the learned seed
        {"name": "con2prim_learned", "kind": "con2prim", "n": 1048576, "seeding": "learned"},
        # training the learned seed: 20 Adam steps of batch 4096
        {"name": "mlp_train", "kind": "mlp", "n": 262144, "batch": 4096, "steps": 20},
        # a caller whose patches are the paper's array-of-structs blocks on the device, halo included:
        # gather, one forward-Euler stage with the wave speed of its result, scatter
        {"name": "aoas_stage", "kind": "aoas", "halo": 1, "levels": "16x16x16:8:128,16x8x8:16:128"},
        # a caller whose blocks live in page-locked host memory: one offloaded SSP-RK3 step
        {"name": "offload_step", "kind": "offload", "halo": 1, "steps": 1, "staged": False,
         "levels": "8x8x8:8:128,8x4x4:16:128"},
    ]


def _spread(rng, lo, hi):
    """A whole number between lo and hi, even in its logarithm."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _box(rng, voxels, p, dim):
    """Patches per axis of a box of about `voxels` voxels in patches of p."""
    K = max(1.0, voxels / p ** dim)
    n = []
    for a in range(dim - 1):
        n.append(max(1, round(K ** (1.0 / (dim - a)) * math.exp(rng.uniform(-0.35, 0.35)))))
        K = max(1.0, K / n[-1])
    n.append(max(1, int(K)))
    return "x".join(map(str, n)) + ":%d:%d" % (p, rng.choice((64, 100, 128, 192, 256)))


def _mix(rng, voxels, sizes, dim, most=3):
    k = rng.randint(1, most)
    return ",".join(_box(rng, voxels / k, rng.choice(sizes), dim) for _ in range(k))


def draw(rng):
    kind = rng.choice(("euler2", "euler3", "cells", "muscl", "coupled", "wave", "gw59", "srhd", "con2prim", "mlp",
                       "aoas", "offload"))
    if kind == "euler2":
        sizes = rng.choice(((8, 16, 24, 32), (5, 10, 12, 20, 27)))
        return {"kind": "euler", "dim": 2, "scheme": 0, "rk": rng.choice((1, 3)), "steps": rng.randint(2, 12),
                "graph": True, "levels": _mix(rng, _spread(rng, 4000, 400000), sizes, 2, 2)}
    if kind == "euler3":
        return {"kind": "euler", "dim": 3, "scheme": 0, "rk": 3, "steps": rng.randint(1, 2),
                "graph": rng.random() < 0.7,
                "levels": _mix(rng, _spread(rng, 30000, 8000000), (8, 16, 24, 32, 40, 64), 3)}
    if kind == "cells":
        p = rng.choice((3, 4, 5, 6, 7, 10, 12, 20))
        most = min(3500000, 16000 * p ** 3)
        return {"kind": "euler", "dim": 3, "scheme": 0, "rk": 3, "steps": rng.randint(1, 2), "graph": True,
                "levels": _box(rng, _spread(rng, 20000, most), p, 3)}
    if kind == "muscl":
        return {"kind": "euler", "dim": 3, "scheme": 2, "rk": 3, "steps": 1, "graph": rng.random() < 0.5,
                "levels": _mix(rng, _spread(rng, 30000, 2500000), (8, 16, 24, 32, 40), 3)}
    if kind == "coupled":
        nc = rng.randint(4, 7)
        m = rng.randint(1, nc - 3)
        return {"kind": "coupled", "nc": nc, "p": rng.choice((8, 16)), "lo": rng.randint(1, nc - 1 - m), "m": m,
                "steps": rng.randint(1, 2)}
    if kind == "wave":
        return {"kind": "wave", "steps": rng.randint(1, 2),
                "levels": _mix(rng, _spread(rng, 30000, 4000000), (8, 16, 24, 32), 3, 2)}
    if kind == "gw59":
        return {"kind": "gw59", "steps": 1, "levels": _mix(rng, _spread(rng, 20000, 1500000), (8, 16, 24, 32), 3, 2)}
    if kind == "srhd":
        sizes = rng.choice(((8, 16, 24, 32), (8, 16, 24, 32), (6, 12, 10)))
        return {"kind": "srhd", "steps": 1, "levels": _mix(rng, _spread(rng, 30000, 8000000), sizes, 3, 2)}
    if kind == "con2prim":
        return {"kind": "con2prim", "n": _spread(rng, 5000, 8000000),
                "seeding": rng.choice(("learned", "previous", "refined", "cold"))}
    if kind == "mlp":
        batch = _spread(rng, 256, 16384)
        return {"kind": "mlp", "n": batch * rng.randint(2, 16) + rng.randint(0, 63), "batch": batch,
                "steps": rng.randint(2, 20)}
    if kind == "aoas":
        return {"kind": "aoas", "halo": rng.randint(0, 3),
                "levels": _mix(rng, _spread(rng, 30000, 6000000), rng.choice(((8, 16, 32), (6, 12, 20))), 3, 2)}
    return {"kind": "offload", "halo": rng.randint(0, 2), "steps": rng.randint(1, 2), "staged": rng.random() < 0.5,
            "levels": _mix(rng, _spread(rng, 30000, 600000), (8, 16, 32), 3, 2)}


# --------------------------------------------------------------------------- meshes and layouts
def _levels(text, dim):
    out = []
    for li, term in enumerate(text.split(",")):
        n, p, inv = term.split(":")
        n = tuple(int(s) for s in n.split("x"))
        out.append(synth.Level(n if dim == 3 else (n[0], n[1], 1), int(p), 1.0 / int(inv), li))
    return out


def _voxels(case):
    if case["kind"] == "coupled":
        return (case["nc"] ** 3 + (2 * case["m"]) ** 3) * case["p"] ** 3
    if "levels" not in case:
        return case["n"]
    dim = case.get("dim", 3)
    return sum(lv.n[0] * lv.n[1] * lv.n[2] * lv.p ** dim for lv in _levels(case["levels"], dim))


def _grid(lv, dim):
    """(z, y, x) voxels of a level's global grid."""
    return (lv.n[2] * lv.p if dim == 3 else 1, lv.n[1] * lv.p, lv.n[0] * lv.p)


def _block(n, align):
    return (n + align - 1) // align * align


def _to_blocks(G, lv, dim):
    """(V, Z, Y, X) -> (V, patches, voxels of a patch), x fastest in both."""
    V, p, pz, (nx, ny, nz) = G.shape[0], lv.p, lv.p if dim == 3 else 1, lv.n
    return G.reshape(V, nz, pz, ny, p, nx, p).permute(0, 1, 3, 5, 2, 4, 6).reshape(V, nx * ny * nz, pz * p * p)


def _to_arena(grids, levels, dim, var_stride):
    """The arena (V, var_stride) of one global grid per level; the space between blocks is 0."""
    out = torch.zeros(grids[0].shape[0], var_stride, dtype=F64, device=DEV)
    off = 0
    for G, lv in zip(grids, levels):
        B = _to_blocks(G, lv, dim)
        V, K, n = B.shape
        pad = _block(n, 16)
        out[:, off:off + K * pad].view(V, K, pad)[:, :, :n] = B
        off += K * pad
    return out


def _gen(seed):
    return torch.Generator(device="cpu").manual_seed(int(seed))


def _fourier(gen, shape, mid, amp, modes=4, kmax=4):
    """mid + amp sum_m a_m sin(2 pi k_m . x / L + phi_m) / sum a_m on a periodic grid (z, y, x)."""
    a = torch.rand(modes, generator=gen, dtype=F64)
    phi = torch.rand(modes, generator=gen, dtype=F64) * 2 * math.pi
    f = torch.zeros(shape, dtype=F64, device=DEV)
    for m in range(modes):
        k = torch.randint(-kmax, kmax + 1, (3,), generator=gen)
        if not k.any():
            k[0] = 1
        ph = [2 * math.pi * int(k[ax]) * (torch.arange(n, dtype=F64, device=DEV) + 0.5) / n
              for ax, n in enumerate(shape)]
        if shape[0] == 1:
            ph[0].zero_()
        f += float(a[m]) * torch.sin(ph[0][:, None, None] + ph[1][None, :, None] + ph[2][None, None, :]
                                     + float(phi[m]))
    return mid + amp * f / float(a.sum())


def _euler_cons(rho, u, p):
    kin = sum(x * x for x in u)
    return torch.stack([rho] + [rho * x for x in u] + [p / (GAMMA_E - 1) + 0.5 * rho * kin])


def _euler_grid(gen, shape, dim):
    """rho, p in [0.5, 1.5], velocities in [-0.5, 0.5], as conserved quantities."""
    rho = _fourier(gen, shape, 1.0, 0.5)
    u = [_fourier(gen, shape, 0.0, 0.5) for _ in range(dim)]
    return _euler_cons(rho, u, _fourier(gen, shape, 1.0, 0.5))


def _srhd_cons(w):
    rho, v, p = w[0], w[1:4], w[4]
    W2 = 1 / (1 - (v * v).sum(0))
    rhoh = rho + GAMMA_R / (GAMMA_R - 1) * p
    D = rho * W2.sqrt()
    return torch.cat([D[None], rhoh * W2 * v, (rhoh * W2 - p - D)[None]])


def _srhd_grid(gen, shape):
    """Primitives: ln rho, ln p smooth on [ln 0.1, ln 10], Lorentz factors up to 10."""
    f = [_fourier(gen, shape, 0.0, math.log(10.0)) for _ in range(2)]
    W = 1 + 9 * _fourier(gen, shape, 0.5, 0.5)
    n = torch.stack([_fourier(gen, shape, 0.0, 1.0) for _ in range(3)])
    n = n / (n * n).sum(0).sqrt().clamp_min(1e-12)
    speed = (1 - 1 / (W * W)).clamp_min(0).sqrt()
    return torch.cat([f[0].exp()[None], speed * n, f[1].exp()[None]])


def _srhd_states(gen, n):
    """Independent primitives: rho, p log-uniform on [0.1, 10], W uniform on [1, 10], any direction."""
    r = torch.rand(3, n, generator=gen, dtype=F64).to(DEV)
    d = torch.randn(3, n, generator=gen, dtype=F64).to(DEV)
    W = 1 + 9 * r[2]
    v = (1 - 1 / (W * W)).sqrt() * d / (d * d).sum(0).sqrt()
    ln = lambda x: torch.exp((2 * x - 1) * math.log(10.0))  # noqa: E731
    return torch.cat([ln(r[0])[None], v, ln(r[1])[None]])


def _wave_grid(gen, shape, lv):
    """Gaussian pulse phi, Pi = 0, psi = grad phi; speed c in [0.5, 2]."""
    L = [n * lv.dx for n in shape]
    x0 = [(0.25 + 0.5 * float(torch.rand(1, generator=gen))) * s for s in L]
    x = [((torch.arange(n, dtype=F64, device=DEV) + 0.5) * lv.dx) for n in shape]
    r = [x[0][:, None, None] - x0[0], x[1][None, :, None] - x0[1], x[2][None, None, :] - x0[2]]
    g = torch.exp(-(r[0] ** 2 + r[1] ** 2 + r[2] ** 2) / (2 * 0.05 ** 2))
    q = torch.stack([g, torch.zeros_like(g)] + [-r[2 - a] / 0.05 ** 2 * g for a in range(3)])
    s = [torch.sin(2 * math.pi * x[a] / L[a]) for a in range(3)]
    return q, (1.25 + 0.75 * s[0][:, None, None] * s[1][None, :, None] * s[2][None, None, :])[None]


def _gw_grid(gen, shape):
    """Flat space (lapse 1, everything else 0) with smooth perturbations of every unknown."""
    q = torch.empty(59, *shape, dtype=F64, device=DEV)
    for v in range(59):
        q[v] = _fourier(gen, shape, 1.0 if v == 55 else 0.0, 1e-3)
    return q


def _gw_coupling(gen):
    return (torch.rand(11, 11, generator=gen, dtype=F64) * 2 - 1) * 0.1


def _inputs(case, seed):
    """The initial data of a mesh case as global grids, one list per quantity group."""
    gen = _gen(seed)
    dim = case.get("dim", 3)
    if case["kind"] == "coupled":
        nC = case["nc"] * case["p"]
        a, w = case["lo"] * case["p"], case["m"] * case["p"]
        C = _euler_grid(gen, (nC,) * 3, 3)
        Fi = C[:, a:a + w, a:a + w, a:a + w]
        for ax in (1, 2, 3):
            Fi = Fi.repeat_interleave(2, ax)
        f = _fourier(gen, Fi.shape[1:], 1.0, 0.02)  # detail that only the fine level has
        return {"q": [C, Fi * f]}
    levels = _levels(case["levels"], dim)
    shapes = [_grid(lv, dim) for lv in levels]
    if case["kind"] == "wave":
        got = [_wave_grid(gen, s, lv) for s, lv in zip(shapes, levels)]
        return {"q": [g[0] for g in got], "mat": [g[1] for g in got]}
    if case["kind"] == "gw59":
        return {"C": _gw_coupling(gen), "q": [_gw_grid(gen, s) for s in shapes]}
    if case["kind"] == "srhd":
        w = [_srhd_grid(gen, s) for s in shapes]
        return {"q": [_srhd_cons(x) for x in w], "mat": w}
    return {"q": [_euler_grid(gen, s, dim) for s in shapes]}


def _mesh(case):
    if case["kind"] == "coupled":
        return synth.coupled_mesh(case["nc"], case["p"], 1.0 / 128, case["lo"], case["m"])
    return synth.make_mesh(_levels(case["levels"], case.get("dim", 3)), case.get("dim", 3))


# --------------------------------------------------------------------------- prepare and run
_PDE = {"wave": dh.PDE_WAVE3D, "gw59": dh.PDE_GW59, "srhd": dh.PDE_SRHD3D}


def _network(gen):
    """Initial weights of the seed network (uniform by fan-in, zero biases), statistics 0 and 1."""
    w = torch.zeros(dh.MLP_LEN)
    u = lambda n, fan: (torch.rand(n, generator=gen) * 2 - 1) / math.sqrt(fan)  # noqa: E731
    w[:96], w[128:1152], w[1184:1216] = u(96, 3), u(1024, 32), u(32, 32)
    w[1220:1223] = 1.0
    return w


def _features(cons, p):
    """Raw network inputs (n, 3) and targets in 32 bits."""
    D, E = cons[0], cons[0] + cons[4]
    S = (cons[1:4] ** 2).sum(0).sqrt()
    return torch.stack([S / E, D / E, torch.log(E / D)], 1).float().contiguous(), torch.log(p / E).float()


def _standardized(w, x):
    w[1217:1220] = x.double().mean(0).float().cpu()
    w[1220:1223] = x.double().std(0, unbiased=False).float().cpu()
    return w


def prepare(case, seed):
    kind = case["kind"]
    if kind == "mlp":
        return _prepare_mlp(case, seed)
    if kind == "con2prim":
        return _prepare_con2prim(case, seed)
    mesh, ins = _mesh(case), _inputs(case, seed)
    dim = case.get("dim", 3)
    pde = _PDE.get(kind, dh.PDE_EULER3D if dim == 3 else dh.PDE_EULER2D)
    scheme = 1 if kind in ("wave", "gw59") else case.get("scheme", 0)
    params = {"wave": [DAMP], "srhd": [GAMMA_R]}.get(kind)
    if kind == "gw59":
        params = np.concatenate([[KAPPA], ins["C"].numpy().ravel()])
    halo = 3 if scheme == 1 else (2 if scheme == 2 else 1)
    plan = dh.dh_plan_create(pde, dim, mesh.patches, halo, mesh.var_stride, params)
    s = {"case": case, "plan": plan, "scheme": scheme}
    q = _to_arena(ins["q"], mesh.levels, dim, mesh.var_stride)
    s["mat"] = _to_arena(ins["mat"], mesh.levels, dim, mesh.var_stride) if "mat" in ins else None
    if kind in ("aoas", "offload"):
        return _prepare_blocks(case, s, mesh, ins)
    s["q"] = q
    s["u1"], s["u2"], s["acc"] = torch.empty_like(q), torch.empty_like(q), torch.empty_like(q)
    s["dt"], s["lam"] = torch.zeros(1, dtype=F64, device=DEV), torch.zeros(1, dtype=F64, device=DEV)
    s["cfl"] = CFL_FD if scheme == 1 else CFL_FV
    s["rk"] = {"wave": 4, "gw59": 4}.get(kind, case.get("rk", 3))
    if kind == "srhd":
        dh.dh_plan_set_con2prim(plan, seed_refine=3)
    dh.max_wave_speed(plan, q, s["mat"], s["lam"])
    s["graph"] = case.get("graph", kind == "coupled")
    if s["graph"]:
        dh.dh_graph_capture(plan, scheme, s["rk"], case["steps"], q, s["u1"], s["u2"], s["acc"], s["mat"], s["dt"],
                            s["lam"], s["cfl"], SIGMA, stream=torch.cuda.Stream())
    return s


def _prepare_blocks(case, s, mesh, ins):
    """One array-of-structs block per patch, halo included, in one allocation (device or pinned host)."""
    h, addr, parts = case["halo"], [], []
    for G, lv in zip(ins["q"], mesh.levels):
        B = _to_blocks(G, lv, 3)
        V, K, n = B.shape
        P = lv.p + 2 * h
        full = torch.zeros(K, P, P, P, V, dtype=F64, device=DEV)
        full[:, h:h + lv.p, h:h + lv.p, h:h + lv.p] = B.reshape(V, K, lv.p, lv.p, lv.p).permute(1, 2, 3, 4, 0)
        addr.append((K, P ** 3 * V))
        parts.append(full.reshape(-1))
    flat = torch.cat(parts)
    if case["kind"] == "offload":
        host = torch.empty(flat.shape, dtype=F64, pin_memory=True)
        host.copy_(flat)
        flat = host
    s["blocks"] = flat
    at, table = flat.data_ptr(), []
    for K, size in addr:
        table += [at + 8 * size * k for k in range(K)]
        at += 8 * size * K
    V, dev = 5, dict(dtype=F64, device=DEV)
    s["arena"] = torch.zeros(V, mesh.var_stride, **dev)
    s["lam"], s["dt"] = torch.zeros(1, **dev), torch.full((1,), 1e-3, **dev)
    s["u1"] = torch.zeros_like(s["arena"])
    if case["kind"] == "aoas":
        s["table"] = torch.tensor(table, dtype=torch.int64, device=DEV)
        return s
    s["u2"], s["acc"] = torch.empty_like(s["arena"]), torch.empty_like(s["arena"])
    (dh.dh_offload_bind_staged if case["staged"] else dh.dh_offload_bind)(s["plan"], table, V, h)
    return s


def _prepare_mlp(case, seed):
    gen = _gen(seed)
    w = _srhd_states(gen, case["n"])
    x, t = _features(_srhd_cons(w), w[4])
    net = _standardized(_network(gen), x).to(DEV)
    nb = (case["batch"] + 63) // 64
    return {"case": case, "w": net, "m": torch.zeros_like(net), "v": torch.zeros_like(net), "x": x, "t": t,
            "partials": torch.empty(nb * dh.MLP_LEN, device=DEV), "grad": torch.empty(dh.MLP_LEN, device=DEV),
            "loss": torch.empty(case["steps"], device=DEV)}


def _prepare_con2prim(case, seed):
    gen = _gen(seed)
    w = _srhd_states(gen, case["n"])
    cons = _srhd_cons(w).contiguous()
    s = {"case": case, "cons": cons, "prim": torch.empty_like(cons), "mlp": None, "prev": None, "refine": 0,
         "status": torch.empty(case["n"], dtype=torch.uint8, device=DEV)}
    if case["seeding"] in ("previous", "refined"):  # the pressure of a step before: a few per cent off
        s["prev"] = (w[4] * (1 + 0.05 * torch.rand(case["n"], generator=gen, dtype=F64).to(DEV))).contiguous()
        s["refine"] = 3 if case["seeding"] == "refined" else 0
    if case["seeding"] == "learned":  # a network trained before on states of the same kind
        m = _prepare_mlp({"n": 65536, "batch": 4096, "steps": 200}, 1)
        _train(m)
        s["mlp"], s["refine"] = m["w"], 3
    return s


def _train(s):
    c = s["case"]
    dh.dh_mlp_train(s["w"], s["m"], s["v"], s["x"], s["t"], c["n"], c["batch"], c["steps"], 0, 1e-3, s["partials"],
                    s["grad"], s["loss"])


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "mlp":
        _train(s)
        return [s["w"], s["m"], s["v"], s["loss"]]
    if kind == "con2prim":
        dh.con2prim_flat(s["cons"], s["prim"], case["n"], case["n"], s["prev"], s["mlp"], GAMMA_R,
                         status=s["status"], seed_refine=s["refine"])
        return [s["prim"], s["status"]]
    plan = s["plan"]
    if kind == "aoas":
        dh.dh_gather_aoas(plan, s["table"], 5, case["halo"], s["arena"])
        dh.patch_update_fv(plan, s["arena"], None, s["u1"], None, None, s["dt"], 0.0, 1.0, 1.0, 0.0, s["lam"])
        dh.dh_scatter_aoas(plan, s["u1"], s["table"], 5, case["halo"])
        return [s["blocks"], s["u1"], s["lam"]]
    if kind == "offload":
        dh.dh_offload_run(plan, 0, 3, case["steps"], s["arena"], s["u1"], s["u2"], s["acc"], s["dt"], s["lam"],
                          CFL_FV, 0.0, 5)
        return [s["blocks"], s["lam"]]
    if s["graph"]:
        dh.dh_graph_launch(plan)
    else:
        for _ in range(case["steps"]):
            dh.dh_rk_step(plan, s["scheme"], s["rk"], s["q"], s["u1"], s["u2"], s["acc"], s["mat"], s["dt"], s["lam"],
                          s["cfl"], SIGMA)
    out = [s["q"], s["lam"]]
    return out + [s["mat"]] if kind == "srhd" else out


def work(case):
    kind, n = case["kind"], _voxels(case)
    if kind == "mlp":  # forward, backward and weight gradients: 6 FP32 FLOP per weight and sample
        return {"bytes": 16.0 * case["batch"] * case["steps"], "flops": 6.0 * 1152 * case["batch"] * case["steps"]}
    if kind == "con2prim":
        its = {"learned": 2.0, "refined": 2.0, "previous": 4.0, "cold": 6.5}[case["seeding"]]
        prev = 8 if case["seeding"] in ("previous", "refined") else 0
        return {"bytes": (81.0 + prev) * n, "flops": (24 + 24 * its) * n}
    if kind == "aoas":  # blocks -> arena, stage, arena -> blocks: the state is read and written once
        return {"bytes": 80.0 * n, "flops": 178.0 * n}
    if kind == "offload":
        return {"bytes": 80.0 * n, "flops": 534.0 * n * case["steps"]}
    rk = {"wave": 4, "gw59": 4}.get(kind, case.get("rk", 3))
    name = {"wave": "wave", "gw59": "gw59", "srhd": "srhd"}.get(kind, "euler3")
    if kind == "euler":
        name = "muscl3" if case["scheme"] == 2 else "euler%d" % case["dim"]
    flops = FLOPS.get((name, rk), 114 * rk)
    values = {"wave": 11, "gw59": 118, "srhd": 20, "euler2": 8}.get(name, 10)
    return {"bytes": 8.0 * values * n, "flops": float(flops * n * case["steps"])}


# --------------------------------------------------------------------------- the same in plain torch
def _sh(a, ax, k):
    return torch.roll(a, k, ax)


def _euler_parts(Q, d):
    """Flux and largest speed along direction d (0 = x) of conserved states (V, ...)."""
    rho, E = Q[0], Q[-1]
    p = (GAMMA_E - 1) * (E - 0.5 * (Q[1:-1] ** 2).sum(0) / rho)
    u = Q[1 + d] / rho
    F = Q * u
    F[1 + d] += p
    F[-1] += p * u
    return F, u.abs() + (GAMMA_E * p / rho).sqrt()


def _srhd_parts(Q, w, d):
    v, p = w[1 + d], w[4]
    F = Q * v
    F[1 + d] += p
    F[4] = Q[1 + d] - Q[0] * v
    v2 = (w[1:4] ** 2).sum(0)
    cs2 = GAMMA_R * p / (w[0] + GAMMA_R / (GAMMA_R - 1) * p)
    disc = (1 - v2) * (1 - v2 * cs2 - v * v * (1 - cs2))
    return F, (v.abs() * (1 - cs2) + (cs2 * disc).sqrt()) / (1 - v2 * cs2)


def _rusanov(L, R, pL, pR):
    return 0.5 * (pL[0] + pR[0]) - 0.5 * torch.maximum(pL[1], pR[1]) * (R - L)


def _fv_L(Q, dx, dim, parts, muscl=False):
    out = torch.zeros_like(Q)
    for d in range(dim):
        ax = Q.ndim - 1 - d
        if muscl:
            a, b = Q - _sh(Q, ax, 1), _sh(Q, ax, -1) - Q
            s = torch.where(a * b > 0, torch.where(a.abs() < b.abs(), a, b), torch.zeros_like(a))
            L, R = _sh(Q + 0.5 * s, ax, 1), Q - 0.5 * s
            F = _rusanov(L, R, parts(L, d), parts(R, d))
        else:
            P = parts(Q, d)
            L = _sh(Q, ax, 1)
            F = _rusanov(L, Q, (_sh(P[0], ax, 1), _sh(P[1], P[1].ndim - 1 - d, 1)), P)
        out -= (_sh(F, ax, -1) - F) / dx
    return out


def _one(x):
    return torch.tensor([x], dtype=F64)


def _euler_speed(grids, dim):
    return max(float(_euler_parts(Q, d)[1].max()) for Q in grids for d in range(dim))


def _coupled_L(C, Fi, dxc, a, w):
    """L on the coarse box and on the refined block [a, a + w)^3 of coarse voxels at half the spacing."""
    LC, LF = torch.zeros_like(C), torch.zeros_like(Fi)
    blk = slice(a, a + w)
    for d in range(3):
        ax = 3 - d
        P = _euler_parts(C, d)
        F = _rusanov(_sh(C, ax, 1), C, (_sh(P[0], ax, 1), _sh(P[1], ax - 1, 1)), P)
        halos = []
        for at in (a - 1, a + w):  # the coarse layers next to the block, prolonged
            at = [slice(None)] + [slice(at, at + 1) if x == ax else blk for x in (1, 2, 3)]
            h = C[at]
            for x in (1, 2, 3):
                if x != ax:
                    h = h.repeat_interleave(2, x)
            halos.append(h)
        pad = torch.cat([halos[0], Fi, halos[1]], ax)
        n = Fi.shape[ax]
        lo, hi = pad.narrow(ax, 0, n + 1), pad.narrow(ax, 1, n + 1)
        G = _rusanov(lo, hi, _euler_parts(lo, d), _euler_parts(hi, d))
        LF -= (G.narrow(ax, 1, n) - G.narrow(ax, 0, n)) / (dxc / 2)
        for at, side in ((a, 0), (a + w, n)):  # the fine fluxes replace the coarse one
            m = G.narrow(ax, side, 1)
            for x in (1, 2, 3):
                if x != ax:
                    m = m.unflatten(x, (-1, 2)).mean(x + 1)
            F[[slice(None)] + [slice(at, at + 1) if x == ax else blk for x in (1, 2, 3)]] = m
        LC -= (_sh(F, ax, -1) - F) / dxc
    return LC, LF


def _restrict(C, Fi, a, w):
    m = Fi.unflatten(3, (-1, 2)).mean(4).unflatten(2, (-1, 2)).mean(3).unflatten(1, (-1, 2)).mean(2)
    C[:, a:a + w, a:a + w, a:a + w] = m


def _ssp3(q, dt, op, fix=lambda u: None):
    """One SSP-RK3 step of the list of grids q."""
    def stage(a, b, c, u):
        out = [a * x + b * y + c * dt * z for x, y, z in zip(q, u, op(u))]
        fix(out)
        return out
    u = stage(0.0, 1.0, 1.0, q)
    u = stage(0.75, 0.25, 0.25, u)
    return stage(1 / 3, 2 / 3, 2 / 3, u), u


def _d1(f, ax, dx):
    return ((_sh(f, ax, 2) - _sh(f, ax, -2)) + 8 * (_sh(f, ax, -1) - _sh(f, ax, 1))) / (12 * dx)


def _ko(f, dx):
    out = torch.zeros_like(f)
    for ax in range(f.ndim - 3, f.ndim):
        out += (_sh(f, ax, 3) + _sh(f, ax, -3)) - 6 * (_sh(f, ax, 2) + _sh(f, ax, -2)) \
            + 15 * (_sh(f, ax, 1) + _sh(f, ax, -1)) - 20 * f
    return SIGMA / (64 * dx) * out


def _wave_L(q, c, dx):
    L = _ko(q, dx)
    L[0] += q[1]
    L[1] += c * c * sum(_d1(q[2 + a], 2 - a, dx) for a in range(3)) - DAMP * q[1]
    for a in range(3):
        L[2 + a] += _d1(q[1], 2 - a, dx)
    return L


def _gw_L(q, C, dx):
    """psi_a,i at 5a + 2 + i; direction i lies along array axis 2 - i."""
    L = torch.empty_like(q)
    for v in range(59):
        L[v] = _ko(q[v], dx)
    al, be = q[55], q[56:59]
    dal = [_d1(al, 2 - i, dx) for i in range(3)]
    src = [q[5 * a] * q[5 * a + 1] for a in range(11)]
    for a in range(11):
        phi, Pi = 5 * a, 5 * a + 1
        psi = [q[5 * a + 2 + i] for i in range(3)]
        dPi = [_d1(q[Pi], 2 - i, dx) for i in range(3)]
        L[phi] += al * q[Pi] + sum(be[i] * psi[i] for i in range(3))
        L[Pi] += al * sum(_d1(psi[i], 2 - i, dx) for i in range(3)) + sum(be[i] * dPi[i] for i in range(3)) \
            + al * sum(float(C[a, b]) * src[b] for b in range(11))
        for i in range(3):
            L[5 * a + 2 + i] += al * dPi[i] + q[Pi] * dal[i] + sum(be[k] * _d1(psi[i], 2 - k, dx) for k in range(3))
        for i in range(3):
            L[56 + i] += 0.75 * psi[i] * q[Pi]
        L[55] -= KAPPA * al * al * q[Pi] ** 2
    return L


def _rk4(q, dt, op):
    k = op(q)
    out, u = q + dt / 6 * k, q + 0.5 * dt * k
    k = op(u)
    out, u = out + dt / 3 * k, q + 0.5 * dt * k
    k = op(u)
    out, u = out + dt / 3 * k, q + dt * k
    return out + dt / 6 * op(u)


def _c2p(cons, p=None):
    """Primitives of conserved states by Newton's method on the pressure, iterated to rest."""
    D, S2, E = cons[0], (cons[1:4] ** 2).sum(0), cons[0] + cons[4]
    lo = (S2.sqrt() - E).clamp_min(0)
    gf = (GAMMA_R - 1) / GAMMA_R
    p = torch.maximum((1 + 1e-8) * lo + 1e-300, (GAMMA_R - 1) * cons[4]) if p is None else p
    for _ in range(40):
        y = E + p
        r = (1 - S2 / y ** 2).sqrt()
        f = gf * (y - S2 / y - D * r) - p
        df = gf * (1 + S2 / y ** 2 - D * S2 / (y ** 3 * r)) - 1
        pn = p - f / df
        p = torch.where(pn > lo, pn, 0.5 * (p + lo))
    v = cons[1:4] / (E + p)
    return torch.cat([(D * (1 - (v * v).sum(0)).sqrt())[None], v, p[None]])


def _exact_mlp(case, seed):
    s = _prepare_mlp(case, seed)
    w0, x, t = s["w"].double(), s["x"].double(), s["t"].double()
    x = (x - w0[1217:1220]) / w0[1220:1223]
    w = w0[:1217].clone().requires_grad_(True)
    m, v = torch.zeros(1217, dtype=F64, device=DEV), torch.zeros(1217, dtype=F64, device=DEV)
    loss, nb, B = [], case["n"] // case["batch"], case["batch"]
    lr, b1, b2, eps = (float(np.float32(z)) for z in (1e-3, 0.9, 0.999, 1e-8))
    for k in range(case["steps"]):
        at = (k % nb) * B
        h = torch.tanh(x[at:at + B] @ w[:96].view(32, 3).T + w[96:128])
        h = torch.tanh(h @ w[128:1152].view(32, 32).T + w[1152:1184])
        y = h @ w[1184:1216] + w[1216]
        e = ((y - t[at:at + B]) ** 2).mean()
        g, = torch.autograd.grad(e, w)
        loss.append(e.detach())
        with torch.no_grad():
            m = b1 * m + (1 - b1) * g
            v = b2 * v + (1 - b2) * g * g
            w -= lr * (m / (1 - b1 ** (k + 1))) / ((v / (1 - b2 ** (k + 1))).sqrt() + eps)
    full = lambda a, tail: torch.cat([a.detach(), tail])  # noqa: E731
    z = torch.zeros(7, dtype=F64, device=DEV)
    return [full(w, w0[1217:]), full(m, z), full(v, z), torch.stack(loss)]


def exact(case, seed):
    kind = case["kind"]
    if kind == "mlp":
        return _exact_mlp(case, seed)
    if kind == "con2prim":
        w = _srhd_states(_gen(seed), case["n"])
        return [_c2p(_srhd_cons(w), w[4]), None]
    ins = _inputs(case, seed)
    q, dim = ins["q"], case.get("dim", 3)
    mesh = _mesh(case)
    levels, vs = mesh.levels, mesh.var_stride
    arena = lambda g: _to_arena(g, levels, dim, vs)  # noqa: E731
    dx_min = min(lv.dx for lv in levels)
    if kind == "coupled":
        a, w = case["lo"] * case["p"], case["m"] * case["p"]
        for _ in range(case["steps"]):
            dt = CFL_FV * dx_min / 3 / _euler_speed(q, 3)
            q, _u = _ssp3(q, dt, lambda u: _coupled_L(u[0], u[1], levels[0].dx, a, w),
                          lambda u: _restrict(u[0], u[1], a, w))
        return [arena(q), _one(_euler_speed(q, 3))]
    if kind in ("euler", "offload", "aoas"):
        muscl = case.get("scheme", 0) == 2
        op = lambda u: [_fv_L(x, lv.dx, dim, _euler_parts, muscl) for x, lv in zip(u, levels)]  # noqa: E731
        for _ in range(case.get("steps", 1)):
            dt = 1e-3 if kind == "aoas" else CFL_FV * dx_min / dim / _euler_speed(q, dim)
            if kind == "aoas" or case.get("rk", 3) == 1:
                q = [x + dt * y for x, y in zip(q, op(q))]
            else:
                q, _u = _ssp3(q, dt, op)
        lam = _euler_speed(q, dim)
        if kind == "euler":
            return [arena(q), _one(lam)]
        h, parts = case["halo"], []
        for G, lv in zip(q, levels):
            B = _to_blocks(G, lv, 3)
            V, K, n = B.shape
            P = lv.p + 2 * h
            full = torch.zeros(K, P, P, P, V, dtype=F64, device=DEV)
            full[:, h:h + lv.p, h:h + lv.p, h:h + lv.p] = B.reshape(V, K, lv.p, lv.p, lv.p).permute(1, 2, 3, 4, 0)
            parts.append(full.reshape(-1))
        return [torch.cat(parts), arena(q), _one(lam)] if kind == "aoas" else [torch.cat(parts), _one(lam)]
    if kind == "srhd":
        w = [_c2p(x, g[4]) for x, g in zip(q, ins["mat"])]
        speed = lambda q, w: max(float(_srhd_parts(x, y, d)[1].max()) for x, y in zip(q, w) for d in range(3))  # noqa: E731
        lam = speed(q, w)
        now = {"w": w}

        def op(u):
            if u is not q:
                now["w"] = [_c2p(x, g[4]) for x, g in zip(u, now["w"])]
            out = []
            for x, y, lv in zip(u, now["w"], levels):
                out.append(_fv_L(x, lv.dx, 3, lambda Q, d, y=y: _srhd_parts(Q, y, d)))
            return out
        q1, _u = _ssp3(q, CFL_FV * dx_min / 3 / lam, op)
        return [arena(q1), _one(lam), arena(now["w"])]
    if kind == "wave":
        lam = max(float(c.max()) for c in ins["mat"])
        dt = CFL_FD * dx_min / 3 / lam
        for _ in range(case["steps"]):
            q = [_rk4(x, dt, lambda u, c=c, lv=lv: _wave_L(u, c[0], lv.dx)) for x, c, lv in zip(q, ins["mat"], levels)]
        return [arena(q), _one(lam)]
    gw_speed = lambda q: max(float((x[55] + x[56 + d].abs()).max()) for x in q for d in range(3))  # noqa: E731
    dt = CFL_FD * dx_min / 3 / gw_speed(q)
    q = [_rk4(x, dt, lambda u, lv=lv: _gw_L(u, ins["C"], lv.dx)) for x, lv in zip(q, levels)]
    return [arena(q), _one(gw_speed(q))]
