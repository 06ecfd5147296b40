"""Grids without an emission table (j = rho^2) and with several bands: every width and
form gives the same bits, and the FP64 oracle's values."""
import numpy as np
import pytest

import oracle
import paper_1010_5534_gb300 as air
import scenes

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

VIEWS = {"inclined": scenes.random_views(87, 1)[0], "axis": scenes.axis_view("-y")}


@pytest.mark.parametrize("kind", ["amr", "uniform"])
@pytest.mark.parametrize("n_bands", [2, 3, 5, 8, 9])
def test_bands_without_a_table(kind, n_bands):
    air.build()
    s = scenes.cone_shock_amr(6, n_base=32, brick=8, levels=1, thickness=0.1, kappa0=0.4, e_lo=0.5,
                              n_bands=n_bands) if kind == "amr" else \
        scenes.random_uniform(4, n=(20, 23, 18), kappa=0.4, with_temp=True, n_bands=n_bands)
    s.emis_mode, s.temp, s.lambda_table = 0, None, None
    g, o = air.Grid(s), oracle.Oracle(s)
    for v in VIEWS.values():
        ref = g.render_adaptive(v, 20, 2, 0.3, include_interior=True)
        ref_f = g.render_fixed(v, 300)
        for bpt in (1, 2, 4, 8, 16):
            g.set_tuning(bands_per_thread=bpt)
            a, f = g.render_adaptive(v, 20, 2, 0.3, include_interior=True), g.render_fixed(v, 300)
            b = g.render_batch([v], 20, 2, 0.3, include_interior=True, bands_per_thread=bpt)[0]
            for k in ("coldens", "intensity", "p"):
                assert torch.equal(a[k], ref[k]) and torch.equal(b[k], ref[k]) and torch.equal(f[k], ref_f[k]), (bpt, k)
        g.set_tuning()
        f, t = g.render_fixed(v, 31), o.fixed(v, 31)
        for got, want in ((f["coldens"], t["col"]), (f["intensity"].T, t["inten"])):
            got = got.cpu().numpy().astype(np.float64)
            assert (np.abs(got - want) <= 1e-5 * np.abs(want) + 1e-7 * np.abs(want).max()).all()
    g.close()
