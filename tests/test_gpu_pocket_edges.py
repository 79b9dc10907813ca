"""Edges of the pocket side's batched kernels: neighbour lists that overflow, more cell rows than a warp's lanes,
lattices of one to 1,024 points, receptors of very different sizes in one call, and device-resident
receptors that the host checks used to read; points against the FP64 oracle as in test_gpu_pocket.py."""
import numpy as np
import pytest

import pvsynth as S
from tests import _gpu as G
from tests.test_gpu_pocket import _check_sas, _params

pytestmark = pytest.mark.gpu


def _receptor(n, density, seed):
    return G.receptor32(S.make_receptor(n, seed, density=density))


@pytest.mark.parametrize("n, density, n_sphere, probe, radius", [
    (1, 0.05, 1024, 1.6, None), (5, 0.05, 1, 1.6, None), (300, 0.05, 33, 1.6, None), (257, 0.05, 96, 0.0, None),
    (700, 0.6, 64, 1.6, None),            # about 700 spheres in reach of one: the list overflows
    (200, 0.002, 40, 10.0, 9.5),          # spheres of 19.5 A: some 20 cells of 4 A per axis in reach
    (64, 5.0, 100, 1.6, None)])           # one or two cells hold every atom
def test_sas_points_at_the_edges(n, density, n_sphere, probe, radius):
    rec = _receptor(n, density, n)
    rad = None if radius is None else np.full(n, radius, np.float32)
    surf = G.context().surface(rec, radius=rad, params=_params(n_sphere=n_sphere, probe=probe))
    _check_sas(rec, surf, n_sphere, probe=probe, radii=None if rad is None else rad.astype(np.float64))


def test_receptors_of_very_different_sizes_in_one_call():
    ctx = G.context()
    recs = [_receptor(n, 0.05, n) for n in (1, 3000, 33, 700)]
    for surf, rec in zip(ctx.surfaces(recs), recs):
        one = ctx.surface(rec)
        assert np.array_equal(surf.sources(), one.sources()) and surf.points().equal(one.points())
        props = np.arange(2.0 * rec.n, dtype=np.float32).reshape(rec.n, 2)
        for a, b in zip(surf.features(props), one.features(props)):
            assert a.equal(b)


@pytest.mark.parametrize("what, value", [("xyz", float("nan")), ("xyz", float("inf")), ("xyz", 2e6), ("radius", 0.0),
                                         ("radius", 11.0), ("radius", float("nan"))])
def test_device_receptors_are_checked(what, value):
    import torch
    from paper_2506_20043_gb300.api import PVError
    ctx = G.context()
    r = _receptor(50, 0.05, 1)
    dev = S.Receptor(torch.tensor(r.xyz, dtype=torch.float32, device="cuda"), *(torch.tensor(a, device="cuda") for a in
                                                                               (r.element, r.donor, r.acceptor)))
    rad = torch.full((50,), 1.7, device="cuda")
    good = ctx.surface(dev, radius=rad).n_points
    if what == "xyz":
        dev.xyz[17, 1] = value
    else:
        rad[49] = value
    with pytest.raises(PVError, match="ARG"):
        ctx.surface(dev, radius=rad)
    with pytest.raises(PVError, match="ARG"):
        ctx.surfaces([r, dev], radii=[None, rad])
    assert ctx.surface(r, radius=np.full(50, 1.7, np.float32)).n_points == good


@pytest.mark.parametrize("n_props", [1, 8, 9, 17])
def test_feature_columns_do_not_depend_on_their_chunk(n_props):
    """Eight columns go to one launch row: a column has the same bits alone and among others."""
    ctx = G.context()
    rec = _receptor(900, 0.05, 3)
    surf = ctx.surface(rec)
    props = np.random.default_rng(0).uniform(-1, 1, (rec.n, n_props)).astype(np.float32)
    feat, prot = surf.features(props)
    for q in range(n_props):
        f, p = surf.features(props[:, q:q + 1])
        assert f[:, 0].equal(feat[:, q]) and p.equal(prot)
