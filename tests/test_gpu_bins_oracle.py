"""Spectral shading, the plain method's persistent warps and the trace's narrow
warps at the edges of their rules, judged by the FP64 oracle (whose loops over bins
share nothing with the kernels' chunks of four):

* bin counts around multiples of four, of a warp's share of chunks and of the count
  from which the plain method's throughput rows leave the chip;
* a glass query list that overflows in the only bounce that has one, and in one of several;
* images around the sizes at which the plain method's warps take 2, 3, 31, 32 and more
  paths a lane set (16 warps on each of 152 SMs), and a batch of renders of different depth;
* scenes around 64 nodes a subdomain, where small waves take narrow warps.

Tolerances are those of tests/test_gpu_render.py: on samples whose decisions are
clear (margin above 1e-5) at most 1 in 1000 off by more than 1e-4 of its norm, the
image within 1e-3."""
import dataclasses

import numpy as np
import pytest

from paper_1912_06474_gb300 import scenes
from tests.helpers import rel_rmse, sample_mismatch

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]

BOTH = (("megakernel", (1, 1, 1)), ("ddm", (2, 2, 1)))


def _against_oracle(oracle_mod, scene, specs, methods=BOTH, pixels=0, **build):
    from paper_1912_06474_gb300 import sddm
    ctx = sddm.Context(0)
    ctx.set_scene(scene)
    oracle = oracle_mod.Oracle(scene)
    rng = np.random.default_rng(0)
    refs = []
    for spec in specs:
        n = spec.width * spec.height
        pix = np.sort(rng.choice(n, pixels, replace=False)).astype(np.uint32) if 0 < pixels < n else None
        refs.append((pix, oracle.render_pixels(spec, pix=pix, per_sample=True, brute_force=True)))
    stats = {}
    for method, grid in methods:
        ctx.build(grid=grid, **build)
        _, stats[method], (sx, prim) = ctx.render(specs, method=method, aov=True)
        for spec, (pix, ref), x, p in zip(specs, refs, sx, prim):
            take = np.arange(spec.width * spec.height) if pix is None else pix
            got = x.cpu().numpy().astype(np.float64).reshape(-1, spec.spp, 3)[take]
            hit = p.cpu().numpy().reshape(-1, spec.spp)[take]
            keep = ref["margin"].reshape(-1) > 1e-5
            assert keep.mean() > 0.9
            assert np.array_equal(hit.reshape(-1)[keep], ref["first_prim"].reshape(-1)[keep]), method
            assert sample_mismatch(got, ref["sample_xyz"], keep, 1e-4).mean() < 1e-3, method
            assert rel_rmse(got.mean(1), ref["xyz"]) <= 1e-3, method
            assert np.linalg.norm(ref["xyz"]) > 0
    ctx.close()
    return stats


@pytest.mark.parametrize("L", [2, 3, 4, 5, 8, 31, 33, 44, 45, 48, 65, 160, 193, 256])
@pytest.mark.parametrize("coated", [False, True])
def test_bin_counts(oracle_mod, L, coated):
    sc = scenes.tiny_room(L=L, seed=3, coated=coated)
    _against_oracle(oracle_mod, sc, [scenes.RenderSpec(37, 23, 3, 5, seed=4, camera=sc.camera)])


@pytest.mark.parametrize("depth", [1, 3])
@pytest.mark.parametrize("coated", [False, True])
def test_query_list_overflow(oracle_mod, depth, coated):
    sc = scenes.tiny_room(L=17, seed=1, coated=coated)
    glass = sc.glass_materials()[0]
    for k in range(4):   # four panes across the whole room between the camera and the lamp
        V, F = scenes.box_mesh((0.01, 0.01, 2.4 + 0.1 * k), (4.99, 3.99, 2.404 + 0.1 * k))
        sc.F = np.concatenate([sc.F, (F + len(sc.V)).astype(np.uint32)])
        sc.V = np.concatenate([sc.V, V.astype(np.float32)])
        sc.mat_id = np.concatenate([sc.mat_id, np.full(len(F), glass, np.uint32)])
        sc.obj_id = np.concatenate([sc.obj_id, np.full(len(F), 100 + k, np.uint32)])
    down = scenes.Camera(pos=(2.5, 2.0, 2.35), look=(2.5, 2.0, 0.0), up=(1.0, 0.0, 0.0), vfov_deg=60.0)
    st = _against_oracle(oracle_mod, sc, [scenes.RenderSpec(40, 30, 2, depth, seed=2, camera=down)])["ddm"]
    # the list holds two queries a path; at depth 1 only the first vertices' shadow rays have any
    assert st["glass_queries"] > 2 * st["paths"]


@pytest.mark.parametrize("L", [16, 48])
@pytest.mark.parametrize("size", [(1, 1, 1), (64, 38, 2), (35, 139, 1), (304, 248, 1), (304, 256, 1), (283, 275, 1),
                                  (300, 200, 3)])
def test_megakernel_paths_per_warp(oracle_mod, L, size):
    sc = scenes.tiny_room(L=L, seed=5)
    _against_oracle(oracle_mod, sc, [scenes.RenderSpec(*size, 5, seed=6, camera=sc.camera)], BOTH[:1], pixels=600)


@pytest.mark.parametrize("L", [16, 48])
def test_megakernel_batch_of_depths(oracle_mod, L):
    sc = scenes.tiny_room(L=L, seed=7)
    specs = [scenes.RenderSpec(20 + 7 * k, 15 + 4 * k, 1 + k % 3, depth, seed=8, render_id=k, camera=sc.camera)
             for k, depth in enumerate((1, 6, 2, 4, 1, 3))]
    _against_oracle(oracle_mod, sc, specs)


@pytest.mark.parametrize("n_tris", [60, 120, 200, 260, 320, 600])
@pytest.mark.parametrize("grid", [(1, 1, 1), (2, 1, 1)])
def test_trace_around_the_narrow_warp_rule(oracle_mod, n_tris, grid):
    sc = scenes.random_soup(n_tris, seed=4)
    rng = np.random.default_rng(4)
    mats = [sc.materials[0], scenes.Material(scenes.EMITTER, Le=np.full(sc.L, 2.0, np.float32))]
    cam = scenes.Camera(pos=(-2.5, 0.3, 0.2), look=(0.5, 0.5, 0.5), vfov_deg=40.0)
    sc = dataclasses.replace(sc, materials=mats, mat_id=(rng.uniform(0, 1, sc.n_tris) < 0.2).astype(np.uint32), camera=cam)
    for size in ((16, 16, 1), (60, 50, 2)):
        _against_oracle(oracle_mod, sc, [scenes.RenderSpec(*size, 3, seed=9, camera=cam)], (("ddm", grid),))
