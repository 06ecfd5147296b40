"""Rasters on both sides of the sizes from which the level maps are used (2^21
pixels bilinear, 3 x 2^20 nearest: sides 1448.2 and 1773.6), against the raster
oracle: nearest the same bits, bilinear within FP32 rounding of the four
products and three sums (2e-7 relative, plus 1e-7 of the image maximum)."""
import ctypes as C

import numpy as np
import pytest

import paper_1010_5534_gb300 as air
import scenes
from oracle import raster as R

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)


@pytest.fixture(scope="module")
def grid():
    air.build()
    g = air.Grid(scenes.cone_shock_amr(1, n_base=32, brick=8, levels=2, n_bands=2, e_lo=0.5, kappa0=0.4,
                                       thickness=0.08))
    yield g
    g.close()


@pytest.mark.parametrize("n0,levels", [(725, 1), (1773, 0), (887, 1), (443, 2), (181, 3), (182, 3), (111, 4),
                                       (7, 8), (3, 9)])
def test_raster_on_both_sides_of_the_line(grid, n0, levels):
    v = scenes.random_views(6, 1)[0]
    r = grid.render_adaptive(v, n0, levels, 0.3, include_interior=True)
    lv, i, j, p = (r[k].cpu().numpy() for k in ("level", "i", "j", "p"))
    nf = n0 << levels
    spare = torch.empty(nf * nf + 1, device="cuda")
    for mode in ("nearest", "bilinear"):
        want = R.raster(lv, i, j, p.astype(np.float64), n0, levels, mode)
        got = grid.raster("p", mode=mode)
        # an output that starts off an 8-byte boundary: the same bits
        code = {"nearest": 0, "bilinear": 1}[mode]
        st = air.lib().air_render_raster(grid._h, 1, 0, code, C.c_void_p(spare.data_ptr() + 4), nf * nf)
        assert st == air.AIR_OK
        assert torch.equal(spare[1:].view(nf, nf), got)
        got = got.cpu().numpy()
        tol = 0.0 if mode == "nearest" else 2e-7 * np.abs(want) + 1e-7 * np.abs(want).max()
        assert (np.abs(got - want) <= tol).all(), mode
