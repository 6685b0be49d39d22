"""Renders replayed as CUDA graphs after something has changed that the recorded
kernels hold by value or that each call uploads: the surrogate's trained box, the
seed. The third call of a kind replays the graph that the second recorded; every
image must be the one a context that never recorded anything renders, bit for bit
(the same kernels on the same inputs)."""
import pytest

from paper_1912_06474_gb300 import scenes

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]


def _context(scene, eager=False):
    from paper_1912_06474_gb300 import sddm
    ctx = sddm.Context(0)
    ctx.set_scene(scene)
    ctx.build(grid=(2, 2, 1))
    if eager:
        ctx.set_profiling(eager=True)
    return ctx


def test_replay_after_the_trained_box_changes():
    sc = scenes.tiny_room(L=41, seed=2)
    spec = scenes.RenderSpec(48, 32, 2, 4, seed=5, camera=sc.camera)
    pane = sc.glass_materials()[0]
    d = float(sc.materials[pane].thickness_m)
    ctx, fresh = _context(sc), _context(sc, eager=True)
    ctx.mlp_train(pane, seed=7, thick_min=0.5 * d, thick_max=1.5 * d)
    w = ctx.mlp_get_weights(pane)
    for lo, hi, outside in ((0.5, 1.5, False), (2.0, 3.0, True), (0.25, 1.25, False)):
        ctx.mlp_set_weights(pane, w, thick_min=lo * d, thick_max=hi * d)
        fresh.mlp_set_weights(pane, w, thick_min=lo * d, thick_max=hi * d)
        want, ws = fresh.render([spec], bsdf="mlp")
        for _ in range(3):
            got, st = ctx.render([spec], bsdf="mlp")
            assert st["mlp_batches"] == ws["mlp_batches"] > 0
            assert st["mlp_fallbacks"] == ws["mlp_fallbacks"]
            assert (st["mlp_fallbacks"] == st["mlp_batches"]) == outside
            assert torch.equal(got[0], want[0])
    ctx.close()
    fresh.close()


@pytest.mark.parametrize("bsdf", ["exact", "mlp"])
def test_replay_with_another_seed(bsdf):
    sc = scenes.tiny_room(L=16, seed=3)
    pane = sc.glass_materials()[0]
    ctx, fresh = _context(sc), _context(sc, eager=True)
    if bsdf == "mlp":
        ctx.mlp_train(pane, seed=7)
        fresh.mlp_set_weights(pane, ctx.mlp_get_weights(pane))
    for seed in (1, 1, 1, 2, 3, 2, 1):
        spec = scenes.RenderSpec(40, 24, 2, 4, seed=seed, camera=sc.camera)
        got, want = ctx.render([spec], bsdf=bsdf)[0][0], fresh.render([spec], bsdf=bsdf)[0][0]
        assert torch.equal(got, want)
    ctx.close()
    fresh.close()
