"""Scores do not depend on how many poses a call has: calls around whole rounds of the resident warps (152 SMs by
28 warps on the largest part this is built for) give each pose the bits it has in small calls."""
import pytest
import torch

import pvsynth as S
from tests import _gpu as G

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", params=[(20, 4), (64, 26)])
def site(request):
    ctx = G.context()
    w = S.tiny()
    gs = ctx.build_grids(G.receptor32(w.receptors[0]), [G.box32(w.boxes[0][0])], list(range(11)))
    lig = ctx.ligand(G.ligand32(S.ligand_centered(S.make_ligand(*request.param, 5))))
    poses = torch.tensor(S.random_poses(8600, w.boxes[0][0], lig.n_rot, 3), dtype=torch.float32, device="cuda")
    xyz = ctx.pose_coords(lig, poses)
    run = lambda a, b: [*ctx.score(gs, lig, 0, poses[a:b], parts=True), *ctx.score_xyz(gs, lig, 0, xyz[a:b]),  # noqa: E731
                        *ctx.score_value_grad(gs, lig, 0, poses[a:b]), ctx.pose_coords(lig, poses[a:b])]
    parts = [run(a, a + 100) for a in range(0, 8600, 100)]
    return run, [torch.cat(v) for v in zip(*parts)]


@pytest.mark.parametrize("n", [1, 3, 4, 5, 151, 153, 607, 608, 609, 4255, 4256, 4257, 8511, 8513, 8600])
def test_scores_do_not_depend_on_the_number_of_poses(site, n):
    run, ref = site
    for got, want in zip(run(0, n), ref):
        assert torch.equal(got, want[:n])
