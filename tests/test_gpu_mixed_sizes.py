"""Calls over items of very different sizes, whose launches are cut into runs (pv_runs.h): every item gives what
a call gives whose launches are not cut, wherever the large one stands."""
import numpy as np
import pytest

import pvsynth as S
from tests import _gpu as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("at", [0, 31, 60])
def test_point_sets(at):
    import torch
    ctx, rng = G.context(), np.random.default_rng(4)

    def points(n):
        return (torch.tensor(rng.uniform(0, max(1.0, (n / 0.02) ** (1 / 3)), (n, 3)), dtype=torch.float32, device="cuda"),
                torch.tensor(rng.uniform(0, 1, n), dtype=torch.float32, device="cuda"))

    sets = [points(n) for n in [0] + [7 * (i % 9) + 1 for i in range(59)]]
    sets.insert(at, points(80000))
    for got, (p, s) in zip(ctx.cluster_many(sets), sets):
        a, b = got.read(), ctx.cluster(p, s).read()
        for k in ("cluster", "size", "first"):
            np.testing.assert_array_equal(a[k], b[k])
        for k in ("score", "center"):       # float64 sums in any order, rounded to float32
            np.testing.assert_allclose(a[k], b[k], rtol=3e-7, atol=0)


@pytest.mark.parametrize("at", [0, 20, 40])
def test_receptors(at):
    ctx = G.context()
    recs = [G.receptor32(S.make_receptor(20 + i, i)) for i in range(40)]
    recs.insert(at, G.receptor32(S.make_receptor(60000, 3)))
    for got, rec in zip(ctx.surfaces(recs), recs):
        one = ctx.surface(rec)
        assert np.array_equal(got.sources(), one.sources()) and got.points().equal(one.points())


@pytest.mark.parametrize("at", [0, 33, 66])
def test_boxes(at):
    import torch
    ctx, rng = G.context(), np.random.default_rng(8)
    rec = G.receptor32(S.make_receptor(3000, 5))
    boxes = [G.box32(S.Box(rng.uniform(-12, 12, 3), np.full(3, 5.0 + 0.1 * i), 0.375)) for i in range(66)]
    large = G.box32(S.Box(np.zeros(3), np.array([70.0, 68.0, 71.0]), 0.375))
    boxes.insert(at, large)
    types = [0, 1, 3, 6, 8]
    gs = ctx.build_grids(rec, boxes, types)
    lig = ctx.ligand(G.ligand32(S.ligand_centered(S.make_ligand(20, 4, 2))))
    types_all = sorted(set(types) | set(lig.xs_types.tolist()))
    packed, plain = ctx.build_grids(rec, boxes, types_all).pack(), ctx.build_grids(rec, boxes, types_all)
    for p in sorted({0, 1, at, 32, 33, 34, 65, 66}):
        # a call of two boxes, in one launch; receptor atoms are binned over the region of all a call's boxes, so the
        # large one keeps the order of the sums
        one = ctx.build_grids(rec, [boxes[p], large], types)
        for t in types:
            np.testing.assert_array_equal(gs.read_map(p, t), one.read_map(0, t))
        poses = torch.tensor(S.random_poses(200, boxes[p], lig.n_rot, 5), dtype=torch.float32, device="cuda")
        a, b = ctx.score(packed, lig, p, poses), ctx.score(plain, lig, p, poses)
        assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])
