"""Docks of few chains, one CTA per chain with line-search trials evaluated ahead by the CTA's other warps, against
the one warp per chain of a fixed search variant (held to the oracle by tests/test_gpu_dock.py): the same bits and
the same counts of evaluations, from one chain to more than run at once, for the ligand sizes of every evaluation
path, both layouts, the consistency check, rounds, and line searches of one, few and many trials."""
import numpy as np
import pytest

import pvsynth as S
from tests import _gpu as G

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def site():
    ctx = G.context()
    rec, boxes = S._carved(2000, 3, (6.0, 7.0), 5, 14.0)
    return ctx, ctx.build_grids(G.receptor32(rec), [G.box32(b) for b in boxes], list(range(11))).pack()


def _sms():
    import torch
    return torch.cuda.get_device_properties(0).multi_processor_count


@pytest.mark.parametrize("sizes, pockets, chains, steps, kw", [
    ([(17, 0)], [0], 1, 20, {}), ([(32, 8)], [1], 8, 12, {}), ([(33, 9)], [0, 1, 2], 5, 10, {}),
    ([(64, 15)], [2], 3, 8, dict(map_layout=0)), ([(30, 6), (20, 1), (47, 11)], [0, 2], 7, 10, {}),
    ([(24, 5)], [0], 9, 14, dict(focc=3)), ([(40, 7)], [1], 9, 10, dict(focc=4, map_layout=0)),
    ([(20, 4)], [0], 6, 11, dict(steps_per_round=4)), ([(20, 4)], [0], 6, 8, dict(bfgs_max_trials=1)),
    ([(20, 4)], [0], 6, 8, dict(bfgs_max_trials=3)), ([(20, 4)], [0], 6, 8, dict(bfgs_max_trials=60)),
    ([(26, 5)], [0], 4, 0, {}), ([(26, 5)], [0], 4, 8, dict(use_graph=0, rescore=1)),
    ([(18, 2)], [0], "all", 4, {}), ([(18, 2)], [0], "more", 4, {})])
def test_foreseen_trials_do_not_change_a_chain(site, sizes, pockets, chains, steps, kw):
    ctx, gs = site
    chains = {"all": 2 * _sms(), "more": 2 * _sms() + 1}.get(chains, chains)
    ligs = [ctx.ligand(G.ligand32(S.ligand_centered(S.make_ligand(n, t, 90 + n)))) for n, t in sizes]
    run = dict(chains=chains, steps=steps, seed=4, top_k=3, **kw)
    r, base = ctx.dock(gs, ligs, pockets, **run), ctx.dock(gs, ligs, pockets, search_variant=0, **run)
    assert r.status_code == 0 and r.stats()[0] == base.stats()[0]
    for a, b in zip(r.chain_records(), base.chain_records()):
        np.testing.assert_array_equal(a, b)
    np.testing.assert_array_equal(r.poses, base.poses)
