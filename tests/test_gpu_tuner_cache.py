"""Saved choices of the autotuner: which plan takes which, and what happens to one that does not fit."""
import json

import numpy as np
import pytest

from gpu_util import require_cuda
from paper_2608_19273_gb300 import dh, synth

pytestmark = pytest.mark.gpu


def _mesh(gap):
    """Eight patches of 16^3 back to back, or with a gap between them (no TMA staging then)."""
    mesh = synth.make_mesh([synth.Level((2, 2, 2), 16, 1.0 / 32, 0)], dim=3)
    if gap:
        mesh.patches["offset"] += 16 * np.arange(8)
        mesh.var_stride += 128
    return mesh


def _tune(torch, mesh, pde, scheme, cache):
    nq, halo = (5, 1) if pde == synth.PDE_EULER3D else (synth.PDE_NQ[pde], 3)
    mat = torch.full((max(synth.PDE_NM[pde], 1), mesh.var_stride), 0.5, dtype=torch.float64, device="cuda")
    with dh.Plan(pde, 3, mesh.patches, halo, mesh.var_stride) as plan:
        q = torch.ones((nq, mesh.var_stride), dtype=torch.float64, device="cuda")
        q[nq - 1] = 2.5
        dt = torch.tensor([1e-3], dtype=torch.float64, device="cuda")
        return dh.dh_autotune(plan, scheme, q, torch.empty_like(q), mat if synth.PDE_NM[pde] else None, dt, reps=1,
                              cache_path=str(cache))


@pytest.mark.parametrize("pde,scheme,key,value", [(synth.PDE_EULER3D, 0, "fv_var", 34), (synth.PDE_WAVE3D, 1, "fd_var", 6)])
def test_choice_a_plan_refuses_is_timed_anew(tmp_path, pde, scheme, key, value):
    """A TMA-staged choice under the key of a plan that cannot run it."""
    torch = require_cuda()
    cache = tmp_path / "tune.jsonl"
    mesh = _mesh(gap=True)
    _tune(torch, mesh, pde, scheme, cache)
    line = json.loads(cache.read_text().splitlines()[-1])
    line[key] = value
    cache.write_text(json.dumps(line) + "\n")
    choice = _tune(torch, mesh, pde, scheme, cache)
    assert not choice[3] and (choice[0] if key == "fv_var" else choice[2]) != value
    assert _tune(torch, mesh, pde, scheme, cache)[3]  # the new choice was saved


@pytest.mark.parametrize("pde,scheme", [(synth.PDE_EULER3D, 0), (synth.PDE_WAVE3D, 1)])
def test_choices_of_plans_with_and_without_tma_are_apart(tmp_path, pde, scheme):
    torch = require_cuda()
    cache = tmp_path / "tune.jsonl"
    assert not _tune(torch, _mesh(gap=False), pde, scheme, cache)[3]
    assert not _tune(torch, _mesh(gap=True), pde, scheme, cache)[3]
    assert _tune(torch, _mesh(gap=False), pde, scheme, cache)[3]


def test_choice_saved_for_other_kernels_is_not_taken(tmp_path):
    """A line as it was written before the key named the kernels' revision."""
    torch = require_cuda()
    cache = tmp_path / "tune.jsonl"
    mesh = _mesh(gap=False)
    _tune(torch, mesh, synth.PDE_WAVE3D, 1, cache)
    line = json.loads(cache.read_text().splitlines()[-1])
    parts = [x for x in line["key"].split("|") if not x.startswith(("rev=", "tma="))]
    line["key"], line["fd_var"] = "|".join(parts), 20
    cache.write_text(json.dumps(line) + "\n")
    choice = _tune(torch, mesh, synth.PDE_WAVE3D, 1, cache)
    assert not choice[3]


@pytest.mark.parametrize("pde,scheme,halo,count", [(synth.PDE_EULER3D, 2, 2, 1), (synth.PDE_GW59, 1, 3, 1),
                                                   (synth.PDE_ADV_NCP, 1, 3, 2), (synth.PDE_WAVE3D, 1, 3, 6)])
def test_candidates_are_different_kernels(pde, scheme, halo, count):
    """One candidate for each kernel that the values of a variant launch."""
    torch = require_cuda()
    mesh = _mesh(gap=False)
    nq, nm = synth.PDE_NQ[pde], synth.PDE_NM[pde]
    with dh.Plan(pde, 3, mesh.patches, halo, mesh.var_stride) as plan:
        q = torch.ones((nq, mesh.var_stride), dtype=torch.float64, device="cuda")
        q[nq - 1] = 2.5
        mat = torch.full((nm, mesh.var_stride), 0.5, dtype=torch.float64, device="cuda") if nm else None
        dt = torch.tensor([1e-3], dtype=torch.float64, device="cuda")
        choice = dh.dh_autotune(plan, scheme, q, torch.empty_like(q), mat, dt, reps=1)
        assert len([t for t in choice[4] if t > 0]) == count


@pytest.mark.parametrize("pde,same", [(synth.PDE_GW59, [(0, 2), (0, 4), (0, 6)]), (synth.PDE_ADV_NCP, [(0, 4), (2, 6), (0, 12), (0, 20)])])
def test_values_that_share_a_kernel(pde, same):
    """fd_var values that select TMA staging, for systems it is not compiled for: the ring's results bit for bit."""
    torch = require_cuda()
    mesh = _mesh(gap=False)
    nq, nm = synth.PDE_NQ[pde], synth.PDE_NM[pde]
    rng = np.random.default_rng(61)
    q = torch.from_numpy(rng.uniform(0.5, 1.5, (nq, mesh.var_stride))).cuda()
    mat = torch.from_numpy(rng.uniform(0.5, 1.5, (nm, mesh.var_stride))).cuda() if nm else None
    dt = torch.tensor([1e-3], dtype=torch.float64, device="cuda")
    outs = {}
    with dh.Plan(pde, 3, mesh.patches, 3, mesh.var_stride) as plan:
        for v in sorted({v for pair in same for v in pair}):
            dh.dh_plan_set_variant(plan, 2, 0, v)
            outs[v] = torch.zeros_like(q)
            dh.patch_update_fd_ko(plan, q, None, outs[v], None, mat, dt, 0.0, 1.0, 1.0, 0.0, 0.1)
    for a, b in same:
        assert torch.equal(outs[a], outs[b])
