"""PVScore and PVScoreXYZ keep the gradient that the forward pass evaluates: it has the bits of the library's
vector-Jacobian products (tests/test_gpu_score.py holds those against the oracle), for every shape and
type the functions take, and what they refused they still refuse."""
import numpy as np
import pytest

import pvsynth as S
from tests import _gpu as G

pytestmark = pytest.mark.gpu


def _site(n_atoms, n_rot, packed):
    ctx = G.context()
    w = S.tiny()
    gs = ctx.build_grids(G.receptor32(w.receptors[0]), [G.box32(w.boxes[0][0])], list(range(11)))
    lig = ctx.ligand(G.ligand32(S.ligand_centered(S.make_ligand(n_atoms, n_rot, n_atoms))))
    return ctx, gs.pack() if packed else gs, lig, w.boxes[0][0]


@pytest.mark.parametrize("n_atoms, n_rot, packed, n", [(1, 0, False, 1), (12, 2, True, 7), (32, 8, True, 300), (33, 5, False, 65),
                                                       (64, 26, True, 33)])
def test_gradients_are_the_library_products(n_atoms, n_rot, packed, n):
    import torch
    from paper_2506_20043_gb300 import api
    ctx, gs, lig, box = _site(n_atoms, n_rot, packed)
    poses = torch.tensor(S.random_poses(n, box, lig.n_rot, 3), dtype=torch.float32, device="cuda")
    xyz = ctx.pose_coords(lig, poses)
    w = torch.linspace(-2.0, 3.0, n, device="cuda")
    for fn, x, ref in ((api.PVScore, poses, lambda: ctx.score_backward(gs, lig, 0, poses, w)[0]),
                       (api.PVScoreXYZ, xyz, lambda: ctx.score_xyz(gs, lig, 0, xyz, grad_energy=w)[1])):
        energy = ctx.score(gs, lig, 0, poses, grad=False)[0] if fn is api.PVScore else ctx.score_xyz(gs, lig, 0, xyz)[0]
        a = x.clone().requires_grad_()
        e = fn.apply(a, ctx, gs, lig, 0)
        assert torch.equal(e, energy)
        g, = torch.autograd.grad(e, a, w, retain_graph=True)
        assert torch.equal(g, ref())
        assert torch.equal(torch.autograd.grad(e, a, w)[0], g)          # the graph can be walked again
        b = x.double().requires_grad_()                                  # another input type
        fn.apply(b, ctx, gs, lig, 0).backward(w)
        assert b.grad.dtype == torch.float64 and torch.equal(b.grad.float(), g)
        c = x.t().contiguous().t().requires_grad_() if x.dim() == 2 else x.reshape(n, -1).clone().requires_grad_()
        fn.apply(c, ctx, gs, lig, 0).sum().backward()                    # strided poses; flat coordinates
        assert c.grad.shape == c.shape
        ones, = torch.autograd.grad(fn.apply(a, ctx, gs, lig, 0).sum(), a)
        assert torch.equal(c.grad.reshape(ones.shape), ones)
        with torch.no_grad():
            assert not fn.apply(a, ctx, gs, lig, 0).requires_grad


def test_second_derivatives_and_changed_inputs_are_refused():
    import torch
    from paper_2506_20043_gb300 import api
    ctx, gs, lig, box = _site(20, 4, False)
    poses = torch.tensor(S.random_poses(5, box, lig.n_rot, 3), dtype=torch.float32, device="cuda")
    a = poses.clone().requires_grad_()
    g, = torch.autograd.grad(api.PVScore.apply(a, ctx, gs, lig, 0).sum(), a, create_graph=True)
    with pytest.raises(RuntimeError):
        g.sum().backward()
    b = poses.clone().requires_grad_()
    c = b * 1.0
    e = api.PVScore.apply(c, ctx, gs, lig, 0).sum()
    c.add_(1.0)
    with pytest.raises(RuntimeError):
        e.backward()
