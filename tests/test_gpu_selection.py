"""The selection's batches of candidates against a plain greedy filter over the chains' bests (sorted by SF, ties by
chain), at chain counts around a batch, and rescoring against the oracle's direct sum over the whole receptor."""
import numpy as np
import pytest
import torch

import oracle as O
import pvsynth as S
from tests import _gpu as G

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def site():
    ctx = G.context()
    w = S.tiny()
    rec, box = G.receptor32(w.receptors[0]), G.box32(w.boxes[0][0])
    ligs = [G.ligand32(S.ligand_centered(S.make_ligand(n, t, n))) for n, t in ((20, 4), (40, 6), (1, 0))]
    return ctx, rec, ctx.build_grids(rec, [box], list(range(11))), ligs, [ctx.ligand(l) for l in ligs]


@pytest.mark.parametrize("chains, top_k, rmsd_min", [(1, 1, 1.0), (7, 9, 1.0), (8, 3, 0.0), (9, 32, 2.0), (100, 9, 4.0),
                                                     (65, 32, 0.5), (40, 5, 50.0)])
def test_selection_is_the_greedy_filter(site, chains, top_k, rmsd_min):
    ctx, _, gs, _, pls = site
    r = ctx.dock(gs, pls, [0], chains=chains, steps=6, seed=3, top_k=top_k, rmsd_min=rmsd_min)
    pots, es = r.chain_records()
    for i, pl in enumerate(pls):
        xyz = ctx.pose_coords(pl, torch.tensor(pots[i, :, :7 + pl.n_rot], device="cuda")).cpu().numpy().astype(np.float64)
        kept = []
        for c in np.lexsort((np.arange(chains), es[i])):
            d = [np.sqrt(np.square(xyz[c] - xyz[k]).sum() / pl.n_atoms) for k in kept]
            assert all(abs(v - rmsd_min) > 1e-4 for v in d) or rmsd_min == 0.0       # no decision on the edge
            if len(kept) < top_k and all(v >= rmsd_min for v in d):
                kept.append(c)
        assert list(r.poses[i]["chain"][:r.n_kept[i]]) == kept


def test_rescoring_sums_every_receptor_atom_in_reach(site):
    ctx, rec, gs, ligs, pls = site
    kw = dict(chains=20, steps=5, seed=4, top_k=4)
    base, r = ctx.dock(gs, pls, [0], **kw), ctx.dock(gs, pls, [0], rescore=True, **kw)
    rt = O.xs_type_receptor(rec)
    for i, lig in enumerate(ligs):
        G.check_rescored(r, i, O.OracleLigand(lig), rec, rt, base)
