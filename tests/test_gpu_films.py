"""Exact coated glass on both sides of the number of films the dense kernels keep in
registers (three), a mixture of stacks in one scene included, against the FP64 oracle.

Tolerance: that of the coated slab elsewhere, 1e-4 absolute in R and T."""
import dataclasses

import numpy as np
import pytest

from paper_1912_06474_gb300 import scenes

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]


def _pane(room, n_films):
    glass = room.materials[room.glass_materials()[0]]
    films = [glass.layers[k % len(glass.layers)] for k in range(n_films)]
    return dataclasses.replace(glass, layers=films or None)


@pytest.mark.parametrize("stacks", [(1,), (2,), (3,), (4,), (10,), (0, 1, 2, 3), (3, 4), (0, 1, 4, 7)])
def test_table_against_oracle(oracle_mod, stacks):
    from paper_1912_06474_gb300 import sddm
    room = scenes.tiny_room(L=41, seed=6, coated=True)
    first = room.glass_materials()[0]
    mats = list(room.materials)
    mats[first] = _pane(room, stacks[0])
    where = [first]
    for j in stacks[1:]:
        mats.append(_pane(room, j))
        where.append(len(mats) - 1)
    ctx = sddm.Context(0)
    ctx.set_scene(dataclasses.replace(room, materials=mats))
    ctx.build()
    rng = np.random.default_rng(sum(stacks))
    n = 300
    for j, g in zip(stacks, where):
        m = mats[g]
        c, s = rng.uniform(0, 1, n).astype(np.float32), rng.uniform(0, 1, n).astype(np.float32)
        b, d = rng.integers(0, 41, n).astype(np.int32), rng.uniform(0.002, 0.01, n).astype(np.float32)
        R, T = (v.cpu().numpy() for v in ctx.glass_eval(g, *(torch.from_numpy(a).cuda() for a in (c, b, s, d))))
        for q in range(n):
            i = b[q]
            films = [(float(f["n"][i]), float(np.float32(f["k"][i]) + np.float32(s[q]) * np.float32(f["dk"][i])),
                      float(np.float32(f["t_nm"]))) for f in (m.layers or [])]
            alpha = float(np.float32(m.alpha_clear[i]) + np.float32(s[q]) * np.float32(m.dalpha[i]))
            r, t = oracle_mod.coated_slab(c[q], room.lam[i], m.n[i], alpha, d[q], films) if films else \
                oracle_mod.slab(c[q], room.lam[i], m.n[i], alpha, d[q])
            assert abs(R[q] - r) < 1e-4 and abs(T[q] - t) < 1e-4, (j, q)
    ctx.close()
