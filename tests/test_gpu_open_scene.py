"""Rays that leave an open scene hit nothing: the megakernel, like the DDM,
reports first-hit triangle -1 and a black sample, although such a ray may have
been tested against triangles on its way (a miss there is no hit at infinity)."""
import numpy as np
import pytest

from paper_1912_06474_gb300 import scenes

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]


@pytest.mark.parametrize("n_tris", [1, 7, 300])
def test_misses(oracle_mod, n_tris):
    from paper_1912_06474_gb300 import sddm
    sc = scenes.random_soup(n_tris, seed=n_tris)
    spec = scenes.RenderSpec(64, 64, 1, 4, seed=1, camera=sc.camera)
    ref = oracle_mod.Oracle(sc).render_pixels(spec, per_sample=True, brute_force=True)
    want, sure = ref["first_prim"].reshape(-1), ref["margin"].reshape(-1) > 1e-5
    assert (want < 0).sum() > 100 and (want >= 0).sum() > 0
    ctx = sddm.Context(0)
    ctx.set_scene(sc)
    for method, grid in (("megakernel", (1, 1, 1)), ("ddm", (2, 2, 2))):
        ctx.build(grid=grid)
        _, _, (sx, prim) = ctx.render([spec], method=method, aov=True)
        got = prim[0].cpu().numpy()
        assert np.array_equal(got[sure], want[sure]), method
        assert np.abs(sx[0].cpu().numpy()[got < 0]).max() == 0
    ctx.close()
