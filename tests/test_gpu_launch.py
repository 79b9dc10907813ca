"""Which search kernel a dock runs and what it reports of the launch (DockResult.launched, launch_shape): few chains
of whole-warp ligands with the shape left free in the kernel of their own, everything else in the round kernel or
the thread-per-chain one; a reported shape can be asked for. The jobs that a free shape sends elsewhere reach the
round kernel's queue and the autotuner here with the variant fixed, or with more chains."""
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
    ligs = {n: ctx.ligand(G.ligand32(S.ligand_centered(S.make_ligand(n, t, 90 + n)))) for n, t in
            ((14, 3), (20, 4), (22, 5), (24, 11), (45, 9))}
    return ctx, gs, ligs


def _sms():
    import torch
    return torch.cuda.get_device_properties(0).multi_processor_count


@pytest.mark.parametrize("atoms, pockets, chains, kw, kernel, warps", [
    (20, [0], 1, {}, "few", 8), (45, [0, 1], 3, {}, "few", 8), (24, [0], "2 per SM", {}, "few", 8),
    (24, [0], "and one", {}, "round", None), (24, [0, 1, 2], 2000, dict(search_variant=3), "round", 28),
    (45, [0, 1, 2], 2000, dict(search_variant=1), "round", 20), (14, [0], 1, {}, "round", 1),
    (24, [0], 8, dict(search_variant=0), "round", 1), (24, [0], 8, dict(warps_per_cta=2), "round", 2),
    (24, [0], 200, dict(mode="plain"), "plain", 4), (24, [0, 1], 200, dict(mode="plain_warp", search_variant=1), "round", 2),
    (24, [0], 200, dict(mode="plain_warp", search_variant=1, warps_per_cta=4), "round", 4)])
def test_the_launch_that_ran_is_reported(site, atoms, pockets, chains, kw, kernel, warps):
    ctx, gs, ligs = site
    chains = {"2 per SM": 2 * _sms(), "and one": 2 * _sms() + 1}.get(chains, chains)
    lanes16 = atoms == 14
    r = ctx.dock(gs, [ligs[atoms]], pockets, chains=chains, steps=2, seed=1, **kw)
    name, w, ctas = r.launched()
    assert name == {"few": "search_few_kernel", "round": "search_round_kernel", "plain": "plain_search_kernel"}[kernel]
    assert warps is None or w == warps
    n = len(pockets) * chains
    if kernel == "few":
        assert ctas == n
    elif kernel == "plain":
        assert ctas == -(-chains // 128)
    else:
        assert 1 <= ctas <= min(n, _sms() * (16 if "warps_per_cta" in kw else 1))
    v, accepted = r.launch_shape()
    again = ctx.dock(gs, [ligs[atoms]], pockets, chains=chains, steps=2, seed=1, search_variant=v, warps_per_cta=accepted)
    assert (v >= 4) == (again.launch_shape()[0] >= 4) and again.launch_shape()[1] == accepted
    if kernel != "plain" and not lanes16:
        np.testing.assert_array_equal(r.chain_records()[1], again.chain_records()[1])


@pytest.mark.parametrize("chains, steps", [(103, 9), (400, 20)])
def test_the_autotuner_chooses_either_layout_with_the_same_bits(site, chains, steps):
    ctx, gs, ligs = site
    assert 3 * chains > 2 * _sms()
    lig = ligs[22]
    r = ctx.dock(gs, [lig], [0, 1, 2], chains=chains, steps=steps, seed=3)
    v, w = r.launch_shape()
    assert r.launched()[0] == "search_round_kernel" and r.map_layout() in (0, 1)
    for layout in (0, 1):
        ref = ctx.dock(gs, [lig], [0, 1, 2], chains=chains, steps=steps, seed=3, map_layout=layout, search_variant=v, warps_per_cta=w)
        np.testing.assert_array_equal(r.chain_records()[1], ref.chain_records()[1])


@pytest.mark.parametrize("atoms, chains, steps, kw", [
    ([45], 1, 9, {}), ([20, 45], 31, 12, {}), ([45, 24, 22], 5, 40, {}), ([24], 101, 20, dict(steps_per_round=7))])
def test_small_jobs_from_the_queue(site, atoms, chains, steps, kw):
    ctx, gs, ligs = site
    run = dict(chains=chains, steps=steps, seed=9, top_k=3, **kw)
    js = [ligs[n] for n in atoms]
    r = ctx.dock(gs, js, [0, 1, 2], search_variant=1, **run)
    base = ctx.dock(gs, js, [0, 1, 2], search_variant=0, warps_per_cta=1, **run)
    assert r.launched()[0] == "search_round_kernel" and r.status_code == 0 and r.stats()[0] == base.stats()[0]
    for a, b in zip(r.chain_records(), base.chain_records()):
        np.testing.assert_array_equal(a, b)
