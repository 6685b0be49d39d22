"""Rounding error of the sums over bins: a wall of 1024 emitters of random spectra
seen directly, so that a sample is sum_i Le_i w_i and nothing else.

A compensated sum rounds its products and its result and nothing on the way. With
rounding errors uniform in half a unit in the last place, its error against 64 bits
has the root mean square sqrt((ulp(result)^2 + sum_i ulp(product_i)^2) / 12); the
tolerance is that plus five standard deviations of a root mean square over 1024
values (5 / sqrt(2 * 1024) = 11 %). Plain sums of four bins between compensated
ones are 1.2 to 1.5 times as far off."""
import numpy as np
import pytest

from paper_1912_06474_gb300 import scenes

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]

SIDE = 32


def _wall(L):
    base = scenes.tiny_room(L=L)
    rng = np.random.default_rng(L)
    mats = [scenes.Material(scenes.LAMBERT, rho=np.full(L, 0.5, np.float32))]
    V, F, M, n = [], [], [], 0

    def add(quad, mat):
        nonlocal n
        v, f = scenes.quad_mesh(*quad)
        V.append(v)
        F.append(np.asarray(f) + n)
        M.append(np.full(len(f), mat))
        n += len(v)

    add([(2, -1, -1), (2, -1, 5), (2, 5, 5), (2, 5, -1)], 0)
    for k in range(SIDE * SIDE):
        y, z = 0.1 * (k % SIDE), 0.1 * (k // SIDE)
        mats.append(scenes.Material(scenes.EMITTER, Le=rng.uniform(0.5, 1.5, L).astype(np.float32)))
        add([(1, y, z), (1, y, z + 0.1), (1, y + 0.1, z + 0.1), (1, y + 0.1, z)], 1 + k)
    M = np.concatenate(M).astype(np.uint32)
    half = 0.05 * SIDE
    cam = scenes.Camera(pos=(0, half, half), look=(1, half, half), ortho_height=2 * half)
    return scenes.Scene(base.lam, base.quad_w, base.cmf, mats, np.concatenate(V).astype(np.float32),
                        np.concatenate(F).astype(np.uint32), M, np.arange(len(M), dtype=np.uint32), cam)


def _ulp(x):
    return np.spacing(np.abs(np.asarray(x, np.float32))).astype(np.float64)


@pytest.mark.parametrize("L", [5, 8, 16, 41, 81])
@pytest.mark.parametrize("method", ["ddm", "megakernel"])
def test_sums_over_bins_round_once(method, L):
    from paper_1912_06474_gb300 import sddm
    sc = _wall(L)
    ctx = sddm.Context(0)
    ctx.set_scene(sc)
    ctx.build(grid=(1, 2, 2))
    spec = scenes.RenderSpec(3 * SIDE, 3 * SIDE, 1, 1, seed=1, camera=sc.camera)
    _, _, (sx, prim) = ctx.render([spec], method=method, aov=True)
    got, prim = sx[0].cpu().numpy().astype(np.float64).reshape(-1, 3), prim[0].cpu().numpy().reshape(-1)
    ctx.close()
    mat = np.where(prim >= 0, sc.mat_id[prim], 0)
    seen, first = np.unique(mat, return_index=True)
    seen, first = seen[seen > 0], first[seen > 0]
    assert len(seen) > 1000
    Le = np.stack([sc.materials[m].Le for m in seen]).astype(np.float64)
    w = (np.asarray(sc.quad_w, np.float64)[:, None] * np.asarray(sc.cmf, np.float64)).astype(np.float32).astype(np.float64)
    p = Le[:, :, None] * w[None]
    want = p.sum(1)
    assert (got[first] > 0).all()
    err = np.sqrt((((got[first] - want) / want) ** 2).mean())
    once = np.sqrt((((_ulp(want) ** 2 + (_ulp(p) ** 2).sum(1)) / 12) / want ** 2).mean())
    print(f"{method} L={L}: rms error {err:.3e}, one rounding of products and result {once:.3e}")
    assert err <= 1.11 * once
