"""Grids of more than 8 bands through the calls whose march writes elsewhere than a
plain image's: streamed spectra (staging buffers, offset by the sweep's first node)
and sharded images (slices of a sweep), against the plain image, bit for bit."""
import ctypes as C
import functools

import pytest

import paper_1010_5534_gb300 as air
import scenes

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

VIEWS = {"inclined": scenes.random_views(84, 1)[0], "axis": scenes.axis_view("-z")}


@functools.lru_cache(maxsize=1)
def grid(n_bands):
    air.build()
    return air.Grid(scenes.cone_shock_amr(6, n_base=32, brick=8, levels=2, thickness=0.08, kappa0=0.4,
                                          e_lo=0.5, n_bands=n_bands))


@pytest.mark.parametrize("n_bands", [9, 12, 33])
@pytest.mark.parametrize("view", sorted(VIEWS))
def test_streamed_spectra_of_many_bands(n_bands, view):
    g, v = grid(n_bands), VIEWS[view]
    ref = g.render_adaptive(v, 40, 3, 0.3, include_interior=True)
    got, spec = g.render_adaptive_spectra(v, 40, 3, 0.3)
    assert got["n_steps"] == ref["n_steps"]
    for k in ("level", "i", "j", "coldens", "p", "band_flux"):
        assert torch.equal(got[k], ref[k]), k
    assert torch.equal(spec, ref["intensity"].cpu())


@pytest.mark.parametrize("n_bands", [9, 12, 33])
@pytest.mark.parametrize("view", sorted(VIEWS))
@pytest.mark.parametrize("rank,world", [(0, 2), (1, 2), (2, 3)])
def test_sharded_image_of_many_bands(n_bands, view, rank, world):
    """One rank's call, the other ranks' slices filled in from the plain image."""
    g, v = grid(n_bands), VIEWS[view]
    ref = g.render_adaptive(v, 40, 3, 0.3, include_interior=True)
    ref = {k: t.clone() if hasattr(t, "clone") else t for k, t in ref.items()}

    def exchange(user, first, count, nb, N, I, stride, p, steps):
        lo, hi = first + count * rank // world, first + count * (rank + 1) // world

        def fill(ptr, src):
            dst = torch.as_tensor(air._DeviceArray(ptr, first + count, "<f4"), device="cuda")
            for a, b in ((first, lo), (hi, first + count)):
                dst[a:b] = src[a:b]
        fill(N, ref["coldens"])
        fill(p, ref["p"])
        for b in range(nb):
            fill(I + 4 * b * stride, ref["intensity"][b])
        torch.cuda.current_stream().synchronize()
        return 0

    cb = air.EXCHANGE_FN(exchange)
    buf = g.alloc_image(ref["n_out"], "device", ("level", "i", "j", "coldens", "p", "intensity"))
    im = g._image_of(buf, "device")
    par = air.Params(40, 3, 0.3, 0, 0, -1, 1)
    air._check(air.lib().air_set_stream(g._h, air._stream()))
    air._check(air.lib().air_render_adaptive_sharded(g._h, C.byref(air._view(v)), C.byref(par),
                                                     C.byref(air.Shard(rank, world, cb, None)), C.byref(im)))
    assert im.n_out == ref["n_out"]
    for k, t in buf.items():
        assert torch.equal(t[..., :im.n_out], ref[k]), k
