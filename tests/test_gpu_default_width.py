"""Up to 8 bands, setting the number of bands per thread that the default takes
leaves launches of few inclined rays as they are (their bands on more threads),
so the autotuner, which tries the widths one by one, also times the default."""
import numpy as np
import pytest

import paper_1010_5534_gb300 as air
import scenes

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)


@pytest.mark.parametrize("n_bands", [1, 2, 4, 5, 6, 8])
def test_the_default_width_set_is_the_default(n_bands):
    air.build()
    g = air.Grid(scenes.cone_shock_amr(8, n_base=32, brick=8, levels=2, n_bands=n_bands, e_lo=0.5, kappa0=0.4,
                                       thickness=0.08))
    v = scenes.random_views(2, 1)[0]
    width = 1 << (n_bands - 1).bit_length()

    def image(bpt):
        g.set_tuning(bands_per_thread=bpt)
        g.render_adaptive(v, 16, 3, 0.3, include_interior=True)  # sizes the outputs
        g.profile(True)
        r = g.render_adaptive(v, 16, 3, 0.3, include_interior=True)
        march = g.profile_read()["march"][1]
        g.profile(False)
        return r, march

    (a, la), (b, lb) = image(0), image(width)
    assert la == lb  # the same march launches and band sums
    for k in ("level", "i", "j", "coldens", "intensity", "p"):
        assert torch.equal(a[k], b[k]), k
    t = g.autotune(v, 16, 3, 0.3)
    assert t["bands_per_thread"] in [w for w in (1, 2, 4, 8) if w <= width]
    g.close()
