"""Leaf output of images around 1024 flux blocks of 8192 nodes, where the leaves in
front of a block stop being added up by the block itself and come from prefix
sums (one launch more), against the interior output's leaves in their order."""
import numpy as np
import pytest

import paper_1010_5534_gb300 as air
import scenes

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)


# 8 388 608 nodes are 1024 flux blocks: 2896^2 lies just below, 2897^2 above
@pytest.mark.parametrize("n0,levels,launches", [(23, 0, 3), (91, 2, 3), (2896, 0, 3), (2897, 0, 4), (2890, 1, 4)])
def test_leaves_in_order(n0, levels, launches):
    air.build()
    s = scenes.random_uniform(10, n=(24, 20, 28), kappa=0.5)
    g = air.Grid(s)
    v = scenes.random_views(82, 1)[0]
    full = g.render_adaptive(v, n0, levels, 0.3, include_interior=True)
    g.profile(True)
    leaf = g.render_adaptive(v, n0, levels, 0.3)
    prof = g.profile_read()
    g.profile(False)
    sel = full["is_leaf"].bool()
    assert leaf["n_out"] == int(sel.sum()) == leaf["n_leaves"]
    for k in ("level", "i", "j", "coldens", "p"):
        assert torch.equal(full[k][sel], leaf[k]), k
    assert torch.equal(full["intensity"][:, sel], leaf["intensity"])
    assert (full["n_out"] > 8388608) == (launches == 4)
    assert prof["output"][1] == launches, prof
    g.close()
