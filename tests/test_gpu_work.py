"""How the batched search hands its chains to warps: for jobs from one chain to several waves, one ligand and more
ligands than a CTA stages at a time, chain counts that divide into nothing, every step-block split: the
same bits as one warp per CTA (tests/test_gpu_dock.py holds that form against the oracle)."""
import numpy as np
import pytest

import pvsynth as S
from tests import _gpu as G

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def site():
    ctx = G.context()
    rec, boxes = S._carved(2000, 3, (6.0, 7.0), 5, 14.0)
    gs = ctx.build_grids(G.receptor32(rec), [G.box32(b) for b in boxes], list(range(11))).pack()
    big = [ctx.ligand(G.ligand32(S.ligand_centered(S.make_ligand(n, t, 40 + n)))) for n, t in
           ((20, 4), (45, 9), (9, 0), (33, 6), (12, 3), (60, 12), (1, 0))]
    small = [ctx.ligand(G.ligand32(S.ligand_centered(S.make_ligand(n, t, 70 + n)))) for n, t in ((16, 4), (8, 1), (13, 3))]
    return ctx, gs, big, small


def _same(ctx, gs, ligs, pockets, base_kw, **kw):
    run = dict(chains=kw.pop("chains"), steps=kw.pop("steps"), seed=9, top_k=3)
    base, r = ctx.dock(gs, ligs, pockets, **run, **base_kw), ctx.dock(gs, ligs, pockets, **run, **kw)
    assert r.status_code == 0 and (r.stats()[2] == 0).all() and r.stats()[0] == base.stats()[0]
    for a, b in zip(r.chain_records(), base.chain_records()):
        np.testing.assert_array_equal(a, b)
    np.testing.assert_array_equal(r.poses, base.poses)
    for i in range(len(ligs)):
        np.testing.assert_array_equal(r.ranking(i), base.ranking(i))


@pytest.mark.parametrize("n_ligs, chains, steps, kw", [
    (1, 1, 9, {}), (1, 153, 5, {}), (1, 1700, 17, {}), (2, 31, 12, {}), (7, 64, 20, {}), (7, 300, 9, {}),
    (7, 37, 12, dict(search_variant=3)), (7, 37, 30, dict(search_variant=1, warps_per_cta=3)), (5, 50, 11, dict(focc=3)),
    (7, 33, 26, dict(warps_per_cta=16, search_variant=0)), (3, 40, 10, dict(steps_per_round=3)),
    (4, 29, 8, dict(mode="plain_warp")), (7, 90, 12, dict(map_layout=0))])
def test_chains_end_the_same_however_they_are_handed_out(site, n_ligs, chains, steps, kw):
    ctx, gs, big, _ = site
    base = dict(search_variant=0, warps_per_cta=1, map_layout=1, **({"focc": kw["focc"]} if "focc" in kw else {}))
    _same(ctx, gs, big[:n_ligs], [0, 1, 2], base, chains=chains, steps=steps, **kw)


@pytest.mark.parametrize("n_ligs, chains, steps, kw", [
    (1, 1, 6, {}), (3, 77, 14, {}), (3, 1001, 9, {}), (2, 5, 30, dict(warps_per_cta=2)), (3, 50, 10, dict(search_variant=7))])
def test_half_warp_chains_end_the_same(site, n_ligs, chains, steps, kw):
    ctx, gs, _, small = site
    _same(ctx, gs, small[:n_ligs], [0, 1, 2], dict(search_variant=4, warps_per_cta=1, map_layout=1), chains=chains, steps=steps,
          **kw)
