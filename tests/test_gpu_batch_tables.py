"""Batches whose blocks hold the tables of every band chunk, and batches whose
blocks hold one at a time (many bands, large tables): views along an axis, inclined
and mixed, with and without the learned proposal, against single images, bit for
bit."""
import functools

import numpy as np
import pytest

import paper_1010_5534_gb300 as air
import scenes

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

INCLINED = scenes.random_views(83, 2)
VIEWS = {"inclined": INCLINED, "axis": [scenes.axis_view("-x"), scenes.axis_view("+y")],
         "mixed": INCLINED + [scenes.axis_view("+z")]}


@functools.lru_cache(maxsize=1)
def grid(n_bands, n_tbins):
    air.build()
    return air.Grid(scenes.cone_shock_amr(6, n_base=32, brick=8, levels=2, thickness=0.08, kappa0=0.4,
                                          e_lo=0.5, n_bands=n_bands, n_tbins=n_tbins))


def same(a, b, what):
    assert a["n_steps"] == b["n_steps"] and a["n_out"] == b["n_out"], what
    for k in ("level", "i", "j", "coldens", "intensity", "p"):
        assert torch.equal(a[k], b[k]), (what, k)


@pytest.mark.parametrize("n_bands,n_tbins", [(16, 255), (32, 64), (33, 255), (48, 128), (64, 64), (64, 255)])
@pytest.mark.parametrize("views", sorted(VIEWS))
def test_batch_is_the_single_images(n_bands, n_tbins, views):
    g = grid(n_bands, n_tbins)
    vs = VIEWS[views]
    ref = [g.render_adaptive(v, 24, 3, 0.35, include_interior=True) for v in vs]
    for bpt in (0, 2, 8, 16):
        for a, b in zip(g.render_batch(vs, 24, 3, 0.35, include_interior=True, bands_per_thread=bpt), ref):
            same(a, b, (bpt, views))


@pytest.mark.parametrize("n_bands,n_tbins", [(3, 64), (12, 64), (33, 64), (64, 255)])
@pytest.mark.parametrize("views", sorted(VIEWS))
def test_learned_batch_is_the_single_images(n_bands, n_tbins, views):
    g = grid(n_bands, n_tbins)
    vs = VIEWS[views]
    net = air.MLP(scenes.mlp_init(7, scale=0.5))
    ref = [g.render_adaptive(v, 24, 3, 0.35, include_interior=True) for v in vs]
    imgs, stats = g.render_batch_learned(vs, 24, 3, 0.35, net, include_interior=True)
    for a, b in zip(imgs, ref):
        same(a, b, views)
    assert stats["proposed_rays"] > 0
    for v, b in zip(vs, ref):  # and one view at a time
        a, st = g.render_learned(v, 24, 3, 0.35, net, include_interior=True)
        same(a, b, views)
    net.close()


def test_blocks_of_many_bands_are_not_fewer():
    """A batch of 64 bands with large tables takes little longer than with small
    ones: the tables of all chunks do not fit, and one at a time leaves as many
    blocks resident as small tables do."""
    ms = []
    for n_tbins in (64, 255):
        g = grid(64, n_tbins)
        best = 1e9
        for k in range(6):
            g.profile(True)
            g.render_batch(INCLINED * 4, 64, 3, 0.35, fields=("band_flux",))
            best = min(best, g.profile_read()["batch"][0])
            g.profile(False)
        ms.append(best)
    assert ms[1] < 1.5 * ms[0], ms
