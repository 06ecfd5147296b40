"""Band flux into device memory at any 4-byte boundary: the values of an aligned
array, and nothing beside them is written."""
import ctypes as C

import pytest

import paper_1010_5534_gb300 as air
import scenes

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)


@pytest.mark.parametrize("n_bands", [1, 3])
@pytest.mark.parametrize("call", ["fixed", "adaptive", "batch"])
@pytest.mark.parametrize("offset", [4, 8, 12])
def test_flux_off_an_8_byte_boundary(n_bands, call, offset):
    air.build()
    g = air.Grid(scenes.random_uniform(3, n=(12, 10, 14), with_temp=True, n_bands=n_bands))
    v = scenes.random_views(2, 1)[0]
    view = air._view(v)
    p = air.Params(20, 2, 0.3, 0, 0, -1, 0)
    L = air.lib()

    def flux(at):
        raw = torch.full((16 + 8 * n_bands + 16,), 0x5a, dtype=torch.uint8, device="cuda")
        im = air.Image()
        im.mem, im.capacity, im.band_flux = air.AIR_DEVICE, 1 << 20, raw.data_ptr() + at
        air._check(L.air_set_stream(g._h, air._stream()))
        if call == "fixed":
            st = L.air_render_fixed(g._h, C.byref(view), 33, -1, C.byref(im))
        elif call == "adaptive":
            st = L.air_render_adaptive(g._h, C.byref(view), C.byref(p), C.byref(im))
        else:
            ims = (air.Image * 1)(im)
            st = L.air_render_batch(g._h, (air.View * 1)(view), 1, C.byref(p), None, ims)
        air._check(st)
        b = raw.cpu()
        end = at + 8 * n_bands
        assert (b[:at] == 0x5a).all() and (b[end:] == 0x5a).all()
        return b[at:end].clone().view(torch.float64)

    want = flux(16)
    assert (want > 0).all()
    assert torch.allclose(flux(offset), want, rtol=1e-14, atol=0) if call == "batch" else \
        torch.equal(flux(offset), want)
    g.close()
