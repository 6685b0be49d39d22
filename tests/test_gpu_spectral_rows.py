"""The DDM's spectral shading pass at the edges of its chunks of four bins: bin
counts around multiples of four and of a warp's share, and shadow rays through
so many panes that the glass query list (two queries a path) overflows and the
pass evaluates glass itself. Judge: the megakernel, which walks the same paths
bin by bin in one thread.

Tolerance: both compute every bin by the same float operations; they differ in
the compiler's contraction of the slab formula (a few ulp, amplified at most
some tens of times at grazing angles) and in the order of sums of positive
terms (a few ulp): 1e-5 of a sample's norm.
"""
import numpy as np
import pytest

from paper_1912_06474_gb300 import scenes

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]


def _compare(scene, spec):
    from paper_1912_06474_gb300 import sddm
    ctx = sddm.Context(0)
    ctx.set_scene(scene)
    ctx.build(grid=(2, 2, 1))
    got = {}
    for method in ("megakernel", "ddm"):
        _, st, (sx, prim) = ctx.render([spec], method=method, aov=True)
        got[method] = (sx[0].cpu().numpy().astype(np.float64), prim[0].cpu().numpy(), st)
    ctx.close()
    want, have = got["megakernel"], got["ddm"]
    assert np.array_equal(want[1], have[1])
    err = np.linalg.norm(want[0] - have[0], axis=1)
    assert (err <= 1e-5 * np.linalg.norm(want[0], axis=1) + 1e-9 * np.abs(want[0]).max()).all(), err.max()
    assert np.abs(want[0]).max() > 0
    return have[2]


@pytest.mark.parametrize("L", [2, 3, 4, 5, 8, 31, 33, 64, 65, 193, 256])
@pytest.mark.parametrize("coated", [False, True])
def test_bin_counts(L, coated):
    sc = scenes.tiny_room(L=L, seed=3, coated=coated)
    _compare(sc, scenes.RenderSpec(37, 23, 3, 5, seed=4, camera=sc.camera))


def test_query_list_overflow():
    sc = scenes.tiny_room(L=16, seed=1)
    glass = sc.glass_materials()[0]
    for k in range(4):   # four panes across the whole room between the camera and the lamp
        V, F = scenes.box_mesh((0.01, 0.01, 2.4 + 0.1 * k), (4.99, 3.99, 2.404 + 0.1 * k))
        sc.F = np.concatenate([sc.F, (F + len(sc.V)).astype(np.uint32)])
        sc.V = np.concatenate([sc.V, V.astype(np.float32)])
        sc.mat_id = np.concatenate([sc.mat_id, np.full(len(F), glass, np.uint32)])
        sc.obj_id = np.concatenate([sc.obj_id, np.full(len(F), 100 + k, np.uint32)])
    st = _compare(sc, scenes.RenderSpec(40, 30, 2, 3, seed=2, camera=sc.camera))
    assert st["glass_queries"] > 2 * st["paths"]   # more than one bounce's list holds
