"""Cells so large that a ray moves less than 1e-30 cells per unit length along every
axis: such a ray counts as at rest, whatever the width of the march. Every width
takes the call and gives the same column densities and step counts."""
import pytest

import paper_1010_5534_gb300 as air
import scenes

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)


@pytest.mark.parametrize("n_bands", [3, 12])
def test_every_width_takes_the_call(n_bands):
    air.build()
    s = scenes.random_uniform(5, n=(4, 4, 4), with_temp=True, n_bands=n_bands)
    s.rho = s.rho * 1e-3
    s.lo, s.hi = (-1e33,) * 3, (1e33,) * 3
    v = scenes.random_views(2, 1)[0]
    v.half_extent = 1e33
    g = air.Grid(s)
    ref = g.render_fixed(v, 5)
    for bpt in (1, 2, 4, 8, 16):
        g.set_tuning(bands_per_thread=bpt)
        r = g.render_fixed(v, 5)
        assert r["n_steps"] == ref["n_steps"] > 0
        assert torch.equal(r["coldens"], ref["coldens"])
    g.close()
