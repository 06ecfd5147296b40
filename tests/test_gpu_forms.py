"""The march has several kernel forms (bands in registers or in shared memory,
many or few rays, rays along an axis or not, one view or a batch), chosen from
the number of bands, rays and views. They round alike, so whichever form takes
a ray, its column density, band intensities and step count are the same bits;
these tests compare the forms with each other at the edges of each choice. The
values themselves are checked against the FP64 oracle in test_gpu_parity.py."""
import functools

import numpy as np
import pytest

import paper_1010_5534_gb300 as air
import scenes
from oracle import raster as R

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)


def np_(t):
    return t.cpu().numpy() if hasattr(t, "cpu") else np.asarray(t)


def same(a, b, what, keys=("coldens", "intensity", "p")):
    for k in keys:
        x, y = np_(a[k]), np_(b[k])
        assert x.shape == y.shape, (what, k, x.shape, y.shape)
        assert ((x == y) | (np.isnan(x) & np.isnan(y))).all(), (what, k)
    assert a["n_steps"] == b["n_steps"], what


@functools.lru_cache(maxsize=None)
def cone(n_bands, brick=8, **kw):
    air.build()
    kw = dict(dict(n_base=32, levels=2, thickness=0.08, kappa0=0.4, e_lo=0.5), **kw)
    return scenes.cone_shock_amr(6, brick=brick, n_bands=n_bands, **kw)


OBLIQUE = scenes.random_views(71, 1)[0]
BANDS = [1, 2, 3, 4, 5, 8, 9, 15, 16, 17, 31, 32, 33, 40, 64]


@pytest.mark.parametrize("n_bands", BANDS)
def test_bands_per_thread_and_ray_counts(n_bands):
    """Every band width, for a handful of inclined rays and for a full launch."""
    g = air.Grid(cone(n_bands))
    # 1 x 1 and 13 x 13: the forms for few rays; 400 x 400: more threads than
    # the GPU holds for up to 8 bands; the adaptive image: counts on the device
    def images():
        return [g.render_fixed(OBLIQUE, 1), g.render_fixed(OBLIQUE, 13), g.render_fixed(OBLIQUE, 400),
                g.render_adaptive(OBLIQUE, 40, 3, 0.3, include_interior=True)]
    ref = images()
    for bpt in (1, 2, 4, 8, 16):
        g.set_tuning(bands_per_thread=bpt)
        for k, (a, b) in enumerate(zip(images(), ref)):
            same(a, b, f"{n_bands} bands, {bpt} per thread, image {k}")
    g.close()


@pytest.mark.parametrize("n_bands", BANDS)
@pytest.mark.parametrize("view", ["-x", "oblique"])
def test_adaptive_pixels_are_the_fixed_images(n_bands, view):
    """A pixel has the same bits in a sweep of any size and in a fixed image."""
    v = OBLIQUE if view == "oblique" else scenes.axis_view(view)
    g = air.Grid(cone(n_bands))
    a = g.render_adaptive(v, 20, 4, 0.25, refine_on=2, include_interior=True)
    L, i, j = (np_(a[k]).astype(int) for k in ("level", "i", "j"))
    for lev in range(5):
        f = g.render_fixed(v, 20 << lev)
        at = L == lev
        k = (j * (20 << lev) + i)[at]
        assert at.any()
        assert (np_(a["intensity"])[:, at] == np_(f["intensity"])[:, k]).all(), lev
        assert (np_(a["coldens"])[at] == np_(f["coldens"])[k]).all(), lev
    g.close()


def test_bands_do_not_depend_on_their_neighbours():
    """Each band of a 33-band grid is the image of the one-band grid of that band
    (table, opacity): the band's own sums, dark cells included."""
    s = cone(33)
    g = air.Grid(s)
    full = g.render_fixed(OBLIQUE, 61)
    for b in (0, 7, 32):
        one = scenes.Scene(**{f: getattr(s, f) for f in s.__dataclass_fields__})
        one.lambda_table = np.ascontiguousarray(s.lambda_table[b:b + 1].repeat(2, axis=0))
        one.kappa = np.repeat(np.asarray(s.kappa)[b:b + 1], 2)
        h = air.Grid(one)
        r = h.render_fixed(OBLIQUE, 61)
        h.close()
        assert (np_(r["intensity"])[0].view(np.uint32) == np_(full["intensity"])[b].view(np.uint32)).all(), b
        assert (np_(r["coldens"]).view(np.uint32) == np_(full["coldens"]).view(np.uint32)).all(), b
    g.close()


@pytest.mark.parametrize("n_tbins", [2, 64, 255])
def test_table_sizes_of_the_wide_form(n_tbins):
    """64 bands of 255 bins fill the shared memory: more chunks than of 64 bins."""
    g = air.Grid(cone(64, n_tbins=n_tbins))
    vs = scenes.random_views(72, 2)
    batch = g.render_batch(vs, 24, 2, 0.4, include_interior=True)
    ref = [g.render_adaptive(v, 24, 2, 0.4, include_interior=True) for v in vs]
    g.set_tuning(bands_per_thread=2)
    for v, a, b in zip(vs, batch, ref):
        c = g.render_adaptive(v, 24, 2, 0.4, include_interior=True)
        same(a, b, "batch")
        same(c, b, "two bands per thread")
    g.close()


@pytest.mark.parametrize("n_bands", [1, 5, 12])
def test_batches_of_inclined_and_mixed_views(n_bands):
    """A batch of inclined views has a kernel without the axis code; the graph
    captured for it must not serve the next batch, which has an axis view."""
    g = air.Grid(cone(n_bands))
    inclined = scenes.random_views(73, 3)
    mixed = inclined[:2] + [scenes.axis_view("-y")]
    for views in (inclined, mixed, inclined, mixed):
        for b, v in zip(g.render_batch(views, 16, 3, 0.3, include_interior=True), views):
            same(b, g.render_adaptive(v, 16, 3, 0.3, include_interior=True), f"{n_bands} bands")
    g.close()


@pytest.mark.parametrize("brick", [4, 8, 16, 32])
@pytest.mark.parametrize("axis", ["+x", "-x", "+y", "-y", "+z", "-z"])
def test_axis_forms_of_each_brick_size(brick, axis):
    """One-band axis kernels (by axis, brick size and direction) against the
    batched kernel, which walks the same columns in its general form."""
    g = air.Grid(cone(1, brick=brick, n_base=64 if brick == 32 else 32))
    v = scenes.axis_view(axis)
    a = g.render_adaptive(v, 33, 2, 0.3, include_interior=True)
    same(g.render_batch([v], 33, 2, 0.3, include_interior=True)[0], a, (brick, axis))
    g.close()


@pytest.mark.parametrize("shape", [(1, 1, 1), (3, 5, 7), (17, 4, 33)])
@pytest.mark.parametrize("fill", ["zero", "huge", "plain"])
def test_uniform_grids_of_odd_shapes(shape, fill):
    """Chunks of cells that end inside a block; densities of zero (no cell
    emits) and so large that the column density overflows (every cell takes the
    full path)."""
    s = scenes.random_uniform(8, n=shape, kappa=0.5, with_temp=True)
    s.rho = s.rho * {"zero": 0.0, "huge": 3e37, "plain": 1.0}[fill]
    g = air.Grid(s)
    for v in (OBLIQUE, scenes.axis_view("+y")):
        a = g.render_fixed(v, 37)
        b = g.render_batch([v], 37, 0, 0.5)[0]
        same(a, b, (shape, fill))
        if fill == "zero":
            assert not np_(a["coldens"]).any() and not np_(a["intensity"]).any()
    g.close()


@pytest.mark.parametrize("n0,levels", [(32, 1), (64, 2), (91, 1), (128, 1), (130, 2)])
def test_output_at_the_edges_of_its_blocks(n0, levels):
    """Leaves are counted per 1024 and per 8192 nodes: base images of one chunk,
    of exactly eight and sixteen, and ragged ones. The leaves are the interior
    output's leaves in their order; the flux is their sum in FP64 (the order of
    addition alone differs: n eps for n <= 10^6 leaves of one sign)."""
    g = air.Grid(cone(2))
    leaf = g.render_adaptive(OBLIQUE, n0, levels, 0.35)
    full = g.render_adaptive(OBLIQUE, n0, levels, 0.35, include_interior=True)
    sel = np_(full["is_leaf"]).astype(bool)
    assert leaf["n_out"] == sel.sum() == leaf["n_leaves"]
    for k in ("level", "i", "j", "coldens", "p"):
        assert (np_(full[k])[sel] == np_(leaf[k])).all(), k
    assert (np_(full["intensity"])[:, sel] == np_(leaf["intensity"])).all()
    area = (2.0 * OBLIQUE.half_extent / n0) ** 2 * 0.25 ** np_(leaf["level"]).astype(np.float64)
    flux = (np_(leaf["intensity"]).astype(np.float64) * area).sum(axis=1)
    for r in (leaf, full):
        np.testing.assert_allclose(np_(r["band_flux"]), flux, rtol=1e6 * 2.0 ** -52)
    host = g.render_adaptive(OBLIQUE, n0, levels, 0.35, mem="host")
    assert (np_(host["band_flux"]) == np_(leaf["band_flux"])).all()
    g.close()


@pytest.mark.parametrize("mode", ["nearest", "bilinear"])
@pytest.mark.parametrize("n0,levels", [(1, 0), (5, 1), (33, 3)])
def test_raster_through_level_maps(mode, n0, levels):
    """Odd widths (rows that start off a 16-byte boundary) and a tree of one level."""
    g = air.Grid(cone(2))
    r = g.render_adaptive(OBLIQUE, n0, levels, 0.3, include_interior=True)
    img = np_(g.raster("I", band=1, mode=mode))
    val = np_(r["intensity"])[1].astype(np.float64)
    want = R.raster(np_(r["level"]), np_(r["i"]), np_(r["j"]), val, n0, levels, mode)
    assert img.shape == want.shape == (n0 << levels, n0 << levels)
    # (bilinear: FP32 rounding of four products and three sums, as in test_gpu_raster.py)
    tol = 0.0 if mode == "nearest" else 2e-7 * np.abs(want) + 1e-7 * np.abs(want).max()
    assert (np.abs(img - want) <= tol).all()
    g.close()
