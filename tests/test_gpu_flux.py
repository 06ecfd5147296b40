"""Band flux against exactly rounded sums (math.fsum) of the returned pixels.

Single images: a thread adds at most 32 leaves as a pair of FP32 numbers. With
u = 2^-24 the pair's low part gathers at most 31 u of the sum and rounds at most
31 u of that, 31^2 u^2 < 2^-38 of the sum; everything else is FP64. Batches add
in FP64 throughout: at most 8 + 6 + 8 additions and one per block of 2048 nodes."""
import functools
import math

import numpy as np
import pytest

import paper_1010_5534_gb300 as air
import scenes

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

OBLIQUE = scenes.random_views(81, 2)


def np_(t):
    return t.cpu().numpy() if hasattr(t, "cpu") else np.asarray(t)


@functools.lru_cache(maxsize=None)
def cone(n_bands):
    air.build()
    return scenes.cone_shock_amr(6, n_base=32, brick=8, levels=2, thickness=0.08, kappa0=0.4, e_lo=0.5,
                                 n_bands=n_bands)


def exact(r, view, n0):
    leaf = np_(r["is_leaf"]).astype(bool)
    w = 0.25 ** np_(r["level"])[leaf].astype(np.float64)
    area = (2.0 * view.half_extent / n0) ** 2
    return np.array([math.fsum(b.astype(np.float64)[leaf] * w) * area for b in np_(r["intensity"])])


def rel(r, view, n0):
    want = exact(r, view, n0)
    got = np_(r["band_flux"])
    assert (got[want == 0] == 0).all() and np.isfinite(got).all()
    return (np.abs(got - want) / np.where(want == 0, 1.0, want)).max()


# pixels of a base image that no sweep refines: below, at and above a chunk (512
# nodes) and a block (8192) of the single image's sums, a block of the batch's
@pytest.mark.parametrize("n0,levels", [(1, 0), (16, 0), (22, 0), (23, 0), (32, 0), (45, 0), (46, 0), (90, 0),
                                       (91, 0), (128, 0), (64, 3)])
@pytest.mark.parametrize("n_bands", [1, 2, 5])
def test_flux_is_the_sum_of_the_leaves(n0, levels, n_bands):
    g = air.Grid(cone(n_bands))
    views = [OBLIQUE[0], scenes.axis_view("+z"), OBLIQUE[1]]
    v = views[0]
    for kw in (dict(), dict(include_interior=True), dict(mem="host")):
        r = g.render_adaptive(v, n0, levels, 0.4, **kw)
        assert rel(r, v, n0) <= 2.0 ** -38, kw
    if levels == 0:
        f = dict(g.render_fixed(v, n0))
        f["is_leaf"], f["level"] = np.ones(n0 * n0, bool), np.zeros(n0 * n0, int)
        assert rel(f, v, n0) <= 2.0 ** -38
    batch = g.render_batch(views, n0, levels, 0.4, include_interior=True)
    n = sum(b["n_out"] for b in batch)
    for b, v in zip(batch, views):
        assert rel(b, v, n0) <= (24 + n / 2048) * 2.0 ** -53
    g.close()


@pytest.mark.parametrize("levels", [0, 2])
def test_flux_beyond_the_range_of_fp32(levels):
    """Finite intensities whose sum exceeds FP32's largest number."""
    s = scenes.random_uniform(9, n=(16, 16, 16), kappa=0.1, with_temp=True, n_bands=2)
    g = air.Grid(s)
    top = np_(g.render_fixed(OBLIQUE[0], 40)["intensity"]).max(axis=1)
    g.close()
    s.lambda_table = (s.lambda_table * (5e37 / top)[:, None]).astype(np.float32)
    g = air.Grid(s)
    r = g.render_adaptive(OBLIQUE[0], 40, levels, 0.4, include_interior=True)
    I = np_(r["intensity"])
    assert np.isfinite(I).all() and I.astype(np.float64).sum() > 2e39
    assert rel(r, OBLIQUE[0], 40) <= 2.0 ** -38
    f = g.render_fixed(OBLIQUE[0], 40)
    f["is_leaf"], f["level"] = np.ones(1600, bool), np.zeros(1600, int)
    assert rel(f, OBLIQUE[0], 40) <= 2.0 ** -38
    for b, v in zip(g.render_batch(OBLIQUE, 40, levels, 0.4, include_interior=True), OBLIQUE):
        assert rel(b, v, 40) <= 64 * 2.0 ** -53
    g.close()
