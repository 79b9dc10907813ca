"""Calls of PVScore and PVScoreXYZ that are not recorded (no_grad, inference_mode, an input without gradient) evaluate
energies alone: no gradient buffer is allocated, and the library is not asked for one."""
import contextlib

import pytest

import pvsynth as S
from tests import _gpu as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("xyz", [False, True])
@pytest.mark.parametrize("mode", ["no_grad", "inference_mode", "plain", "recorded"])
def test_energy_only_where_nothing_is_recorded(xyz, mode):
    import torch
    from paper_2506_20043_gb300 import api
    ctx = G.context()
    w = S.tiny()
    gs = ctx.build_grids(G.receptor32(w.receptors[0]), [G.box32(w.boxes[0][0])], list(range(11)))
    lig = ctx.ligand(G.ligand32(S.ligand_centered(S.make_ligand(24, 5, 24))))
    n = 4096
    x = torch.tensor(S.random_poses(n, w.boxes[0][0], lig.n_rot, 3), dtype=torch.float32, device="cuda")
    fn = api.PVScore
    if xyz:
        x, fn = ctx.pose_coords(lig, x), api.PVScoreXYZ
    x.requires_grad_(mode != "plain")
    guard = {"no_grad": torch.no_grad, "inference_mode": torch.inference_mode}.get(mode, contextlib.nullcontext)
    energy = ctx.score_xyz(gs, lig, 0, x.detach(), grad=False)[0] if xyz else ctx.score(gs, lig, 0, x.detach(), grad=False)[0]
    torch.cuda.synchronize()
    torch.cuda.reset_peak_memory_stats()
    before = torch.cuda.memory_allocated()
    with guard():
        e = fn.apply(x, ctx, gs, lig, 0)
    torch.cuda.synchronize()
    extra = torch.cuda.max_memory_allocated() - before
    assert torch.equal(e, energy) and e.requires_grad == (mode == "recorded")
    gradient = x.numel() * x.element_size()
    if mode == "recorded":
        assert extra >= gradient
    else:
        assert extra < gradient // 4        # the energies: one of 12 or of 72 floats per pose
