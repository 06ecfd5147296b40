"""Two threads render at once, each its own grid on its own stream, through kernels
whose blocks take different amounts of shared memory: no call fails, and every image
is the one that the grid gives alone."""
import threading

import pytest

import paper_1010_5534_gb300 as air
import scenes

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

VIEWS = scenes.random_views(86, 2)
KEYS = ("coldens", "intensity", "p")


def images(g):
    return [g.render_fixed(VIEWS[0], 30), g.render_fixed(VIEWS[1], 7), g.render_adaptive(VIEWS[1], 12, 2, 0.3)]


def test_two_threads_with_different_tables():
    air.build()
    # (bands, bins): 51 and 53 KB a block in the wide march
    shapes = [(32, 64), (64, 255)]
    grids = [air.Grid(scenes.cone_shock_amr(6, n_base=16, brick=8, levels=1, thickness=0.1, kappa0=0.4,
                                            e_lo=0.5, n_bands=nb, n_tbins=nt)) for nb, nt in shapes]
    ref = [[{k: r[k].clone() for k in KEYS} for r in images(g)] for g in grids]
    torch.cuda.synchronize()
    errors = []

    def work(k):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(60):
                    for r, want in zip(images(grids[k]), ref[k]):
                        for f in KEYS:
                            assert torch.equal(r[f], want[f]), f
        except Exception as e:  # noqa: BLE001
            errors.append(e)

    ts = [threading.Thread(target=work, args=(k,)) for k in range(2)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not errors, errors
    for g in grids:
        g.close()
