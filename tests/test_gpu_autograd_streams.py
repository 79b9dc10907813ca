"""PVScore and PVScoreXYZ through a context on a side stream: the gradient is right for a caller who waits for that
stream, and for work that follows the backward pass on the stream it ran on, although the score kernels are
still queued behind other work when the backward pass is issued."""
import pytest

import pvsynth as S
from tests import _gpu as G

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def site():
    import torch
    from paper_2506_20043_gb300 import api
    G.context()
    side = torch.cuda.Stream()
    ctx = api.Context(0, stream=side)
    w = S.tiny()
    gs = ctx.build_grids(G.receptor32(w.receptors[0]), [G.box32(w.boxes[0][0])], list(range(11)))
    lig = ctx.ligand(G.ligand32(S.ligand_centered(S.make_ligand(24, 5, 24))))
    poses = torch.tensor(S.random_poses(500, w.boxes[0][0], lig.n_rot, 3), dtype=torch.float32, device="cuda")
    weight = torch.linspace(-2.0, 3.0, 500, device="cuda")
    torch.cuda.synchronize()
    xyz = ctx.pose_coords(lig, poses)
    torch.cuda.synchronize()
    refs = ctx.score_backward(gs, lig, 0, poses, weight)[0], ctx.score_xyz(gs, lig, 0, xyz, grad_energy=weight)[1]
    torch.cuda.synchronize()
    return ctx, side, gs, lig, (poses, xyz), weight, [r.clone() for r in refs]


@pytest.mark.parametrize("which", [0, 1])
@pytest.mark.parametrize("wait", ["context", "current", "saved on the host"])
def test_gradients_of_a_context_on_a_side_stream(site, which, wait):
    import torch
    from paper_2506_20043_gb300 import api
    ctx, side, gs, lig, inputs, weight, refs = site
    fn = (api.PVScore, api.PVScoreXYZ)[which]
    x = inputs[which].clone().requires_grad_()
    nans = [torch.full_like(x, float("nan")) for _ in range(8)]     # what memory handed out next holds
    torch.cuda.synchronize()
    del nans
    with torch.cuda.stream(side):
        torch.cuda._sleep(200_000_000)                              # a tenth of a second
    if wait == "context":
        g, = torch.autograd.grad(fn.apply(x, ctx, gs, lig, 0), x, weight)
        side.synchronize()
    elif wait == "saved on the host":                               # hooks copy the gradient as soon as it is saved
        with torch.autograd.graph.save_on_cpu():
            e = fn.apply(x, ctx, gs, lig, 0)
        g, = torch.autograd.grad(e, x, weight)
    else:
        fn.apply(x * 1.0, ctx, gs, lig, 0).backward(weight)         # a node after it, on the current stream
        g = x.grad
    got = g.cpu()
    torch.cuda.synchronize()
    assert torch.equal(got, refs[which].cpu())
