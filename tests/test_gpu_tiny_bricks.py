"""Bricks of one and two cells (and four, for comparison): the axis forms against the
batched kernel's general walk, bit for bit, and every form against the FP64 oracle."""
import functools

import numpy as np
import pytest

import oracle
import paper_1010_5534_gb300 as air
import scenes

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)


@functools.lru_cache(maxsize=2)
def scene(brick, n_bands):
    air.build()
    s = scenes.cone_shock_amr(6, n_base=16, brick=brick, levels=2, thickness=0.1, kappa0=0.4, e_lo=0.5,
                              n_bands=n_bands)
    return s, air.Grid(s)


@pytest.mark.parametrize("brick", [1, 2, 4])
@pytest.mark.parametrize("n_bands", [1, 3, 12])
@pytest.mark.parametrize("view", ["+x", "-x", "+y", "-y", "+z", "-z", "inclined"])
def test_tiny_bricks(brick, n_bands, view):
    s, g = scene(brick, n_bands)
    v = scenes.random_views(85, 1)[0] if view == "inclined" else scenes.axis_view(view)
    a = g.render_adaptive(v, 21, 2, 0.3, include_interior=True)
    b = g.render_batch([v], 21, 2, 0.3, include_interior=True)[0]
    c = g.render_batch([v, scenes.axis_view("+x")], 21, 2, 0.3, include_interior=True)[0]
    for x in (b, c):
        assert x["n_steps"] == a["n_steps"]
        for k in ("level", "i", "j", "coldens", "intensity", "p"):
            assert torch.equal(x[k], a[k]), k
    for res in (9, 33):
        f = g.render_fixed(v, res)
        o = oracle.Oracle(s).fixed(v, res)
        for got, want in ((f["coldens"], o["col"]), (f["intensity"].T, o["inten"])):
            got = got.cpu().numpy().astype(np.float64)
            assert want.max() > 0
            assert (np.abs(got - want) <= 1e-5 * np.abs(want) + 1e-7 * np.abs(want).max()).all()
