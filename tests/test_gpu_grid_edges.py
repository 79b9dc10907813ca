"""Edges of the receptor binning of the grid cache, against the FP64 oracle's direct sums at sampled
nodes (the grid tolerance of tests/_gpu.py): atom counts around a block's, boxes whose rows of binning
cells are longer than a warp, receptors mostly outside every box, dense and far-away ones."""
import numpy as np
import pytest

import oracle as O
import pvsynth as S
from tests import _gpu as G

pytestmark = pytest.mark.gpu


def _receptor(n, density, seed, shift=0.0):
    r = S.make_receptor(n, seed, density=density)
    return G.receptor32(S.Receptor(r.xyz + shift, r.element, r.donor, r.acceptor))


def _box(center, size, spacing=0.375):
    return G.box32(S.Box(np.asarray(center, float), np.asarray(size, float), spacing))


CASES = {
    "one atom": (_receptor(1, 0.05, 1), [_box((0.5, 0, 0), (4, 4, 4))]),
    "127 atoms": (_receptor(127, 0.05, 2), [_box((0, 0, 0), (5, 7, 6))]),
    "129 atoms, all types in one cell's reach": (_receptor(129, 0.8, 3), [_box((0, 0, 0), (3, 3, 3))]),
    "dense": (_receptor(6000, 1.5, 4), [_box((0, 0, 0), (4.2, 4.9, 3.4))]),
    "long rows": (_receptor(4000, 0.05, 5), [_box((-18, 0, 0), (6, 6, 6)), _box((80, 1, -60), (6, 6, 6)),
                                             _box((10, 5, 5), (9, 3, 3))]),
    "mostly outside": (_receptor(8000, 0.05, 6), [_box((24, 24, 24), (3, 3, 3))]),
    "far away": (_receptor(1000, 0.05, 7, shift=1000.0), [_box((1000, 1002, 999), (6, 6, 6))]),
    "coarse": (_receptor(3000, 0.05, 8), [_box((0, 0, 0), (40, 30, 22), 4.0)]),
}


@pytest.mark.parametrize("name", list(CASES))
def test_binned_receptor_gives_the_direct_sums(name):
    rec, boxes = CASES[name]
    types = [0, 1, 4, 9, 10]
    gs = G.context().build_grids(rec, boxes, types)
    rt = O.xs_type_receptor(rec)
    rng = np.random.default_rng(11)
    for p, b in enumerate(boxes):
        _, dims = O.grid_geometry(b)
        idx = np.concatenate([rng.integers(0, dims, size=(60, 3)), [dims - 1, np.zeros(3, int)]])
        for t in types:
            ref = np.array([O.grid_node_value(rec, rt, b, t, *i) for i in idx])
            got = gs.read_map(p, t)[idx[:, 2], idx[:, 1], idx[:, 0]]
            assert G.close(got, ref).all(), (p, t, np.abs(got - ref).max())


@pytest.mark.parametrize("types", [[10], [0], [1], [2, 5], [3, 7], [0, 10], [1, 4, 8], [6, 9, 10], [0, 1, 6], [2, 10]])
def test_maps_do_not_depend_on_the_other_types_asked_for(types):
    """Each set of element classes has its own map kernel: a type's map has the same bits in all."""
    rec, boxes = _receptor(1500, 0.3, 9), [_box((0, 0, 0), (6.4, 4.9, 7.2)), _box((2, 1, 0), (3.0, 3.1, 2.6))]
    every = G.context().build_grids(rec, boxes, list(range(11)))
    some = G.context().build_grids(rec, boxes, types)
    for p in range(len(boxes)):
        for t in types:
            np.testing.assert_array_equal(some.read_map(p, t), every.read_map(p, t))


def _offset_context(shift):
    """A context whose device memory starts `shift` bytes past the torch allocator's blocks."""
    import torch
    from paper_2506_20043_gb300 import _capi as A
    from paper_2506_20043_gb300 import api
    ctx = api.Context(0, torch_allocator=False)
    alloc = A.ALLOC_FN(lambda n, stream, _: torch.cuda.caching_allocator_alloc(int(n) + shift, 0, stream) + shift)
    free = A.FREE_FN(lambda p, _s, _u: torch.cuda.caching_allocator_delete(p - shift))
    ctx._keep += [alloc, free]
    ctx._check(ctx.lib.pv_context_set_allocator(ctx.h, alloc, free, None), "pv_context_set_allocator")
    return ctx


@pytest.mark.parametrize("shift", [0, 16])
def test_packed_cells_of_ragged_boxes_hold_the_plain_corners(shift):
    """Boxes of 1 to 27 cells per axis packed in one launch, in 32-byte and in 16-byte aligned memory:
    a lookup in the packed cells gives the bits of one in the plain maps, over the whole box and beyond."""
    import torch
    ctx = _offset_context(shift)
    sizes = [(0.3, 0.3, 0.3), (3.0, 3.0, 3.0), (0.375, 4.0, 10.0), (10.0, 0.5, 3.1), (5.2, 6.1, 3.4)]
    boxes = [_box((0.3 * i, -0.2 * i, 0.1), s) for i, s in enumerate(sizes)]
    lig = ctx.ligand(S.Ligand(np.zeros((1, 3)), np.zeros(1, np.uint8), np.zeros(1, np.uint8), np.zeros(1, np.uint8),
                              np.zeros((0, 2), np.int32), np.zeros(0, np.uint8)))
    rec = _receptor(800, 0.05, 10)
    plain, packed = ctx.build_grids(rec, boxes, [0, 3, 10]), ctx.build_grids(rec, boxes, [0, 3, 10]).pack()
    rng = np.random.default_rng(0)
    for p, s in enumerate(sizes):
        at = np.zeros((4096, 7), np.float32)
        at[:, :3] = np.asarray(boxes[p].center) + (rng.random((4096, 3)) - 0.5) * (np.asarray(s) + 0.4)
        at[:, 3] = 1.0
        x = torch.tensor(at, device="cuda")
        for a, b in zip(ctx.score(plain, lig, p, x)[:2], ctx.score(packed, lig, p, x)[:2]):
            assert torch.equal(a, b)


@pytest.mark.parametrize("n_atoms,packed", [(40, False), (4400, True), (9000, False)])
def test_appended_pockets_past_an_inline_table(n_atoms, packed):
    """Appends that take a set from 1 over 63, 64 and 65 to 67 pockets, where its pocket table moves out of
    the maps' memory, with receptors that go up in one piece and in several: maps and lookups in the packed
    cells have the bits of a set built from the appended boxes alone."""
    import torch
    ctx = G.context()
    rec = _receptor(n_atoms, 0.3, 12)
    lig = ctx.ligand(S.Ligand(np.zeros((1, 3)), np.zeros(1, np.uint8), np.zeros(1, np.uint8), np.zeros(1, np.uint8),
                              np.zeros((0, 2), np.int32), np.zeros(0, np.uint8)))
    boxes = [_box((0.4 * i - 12, 1, 0), (2.6, 3.0 + 0.1 * (i % 5), 2.2)) for i in range(67)]
    parts = [(0, 1), (1, 63), (63, 64), (64, 65), (65, 67)]
    gs = ctx.build_grids(rec, boxes[:1], [0, 9])
    if packed:
        gs.pack()
    for lo, hi in parts[1:]:
        assert gs.append(rec, boxes[lo:hi]) == lo
    if not packed:
        gs.pack()
    at = np.zeros((500, 7), np.float32)
    at[:, 3] = 1.0
    rng = np.random.default_rng(13)
    for lo, hi in parts:
        alone = ctx.build_grids(rec, boxes[lo:hi], [0, 9]).pack()
        for p in {lo, hi - 1}:
            for t in (0, 9):
                np.testing.assert_array_equal(gs.read_map(p, t), alone.read_map(p - lo, t))
            at[:, :3] = np.asarray(boxes[p].center) + (rng.random((500, 3)) - 0.5) * 3
            x = torch.tensor(at, device="cuda")
            for a, b in zip(ctx.score(gs, lig, p, x)[:2], ctx.score(alone, lig, p - lo, x)[:2]):
                assert torch.equal(a, b)
