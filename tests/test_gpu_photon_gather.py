"""The DDM's photon-map gather at the edges of its kernels: bin counts on both
sides of a lane's 1, 2, 3 and 8 bins, and vertices with few and with many photons
in reach (a warp or a whole block per path). Judge: the megakernel's gather, a
thread per path over the same photons.

Tolerance: the same photons (counter-based random numbers) whose positions the two
photon passes round differently by a few ulp, so a photon on the rim of a gather
sphere may fall on different sides; each is one of some hundred of a gather's and
few in 1e5 lie that close: 1e-4 of the image's norm.
"""
import numpy as np
import pytest

from paper_1912_06474_gb300 import scenes
from tests.helpers import rel_rmse

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]


@pytest.mark.parametrize("L,photons,radius,caustic", [(16, 3000, 0.1, 0.0), (32, 20000, 0.3, 0.1), (33, 20000, 0.3, 0.0),
                                                      (64, 60000, 0.4, 0.2), (65, 20000, 0.3, 0.1),
                                                      (96, 20000, 0.3, 0.0), (97, 20000, 0.3, 0.1), (256, 8000, 0.4, 0.0)])
def test_gather_matches_megakernel(L, photons, radius, caustic):
    from paper_1912_06474_gb300 import sddm
    sc = scenes.tiny_room(L=L, seed=5)
    spec = scenes.RenderSpec(45, 31, 2, 4, seed=6, camera=sc.camera)
    ctx = sddm.Context(0)
    ctx.set_scene(sc)
    ctx.build(grid=(2, 2, 1))
    img = {}
    for method in ("megakernel", "ddm"):
        im, _, pst = ctx.render_photon_map(spec, photons, radius, method=method, caustic_radius=caustic)
        img[method] = im.cpu().numpy().reshape(-1, 3).astype(np.float64)
        assert pst["stored"] > photons // 4
    ctx.close()
    assert rel_rmse(img["ddm"], img["megakernel"]) <= 1e-4
