"""Learned glass over explicit rows on both sides of the sizes at which the passes
change: up to 2^18 rows the network runs over every row and a warp per batch checks
it, above that probes come first; up to 2^22 raw rows a CTA carries one tile, above
that four.

The network's rows are equal bit for bit (the same operations on the same row
whatever carries it); exact rows come from two instantiations of the slab formula
and are equal up to float contraction (1e-5 relative, 1e-6 absolute); decisions
closer than 1e-6 to the threshold are left out."""
import numpy as np
import pytest

from paper_1912_06474_gb300 import scenes

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]

LINE = 1 << 18


@pytest.fixture(scope="module", params=[False, True], ids=["bare", "coated"])
def ctx_mat(request):
    from paper_1912_06474_gb300 import sddm
    sc = scenes.tiny_room(L=41, seed=2, coated=request.param)
    ctx = sddm.Context(0)
    ctx.set_scene(sc)
    ctx.build()
    g = sc.glass_materials()[0]
    ctx.mlp_train(g, seed=7)
    yield ctx, g
    ctx.close()


def _rows(n, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    c, s = torch.rand(n, generator=gen, device="cuda"), torch.rand(n, generator=gen, device="cuda")
    b = torch.randint(0, 41, (n,), generator=gen, device="cuda", dtype=torch.int32)
    d = torch.rand(n, generator=gen, device="cuda") * 0.007 + 0.0025
    out = torch.randperm(n, generator=gen, device="cuda")[:max(1, n // 500)]   # rows outside the trained box
    d[out[::2]] = 0.02
    s[out[1::2]] = 1.5
    return c, b, s, d


@pytest.mark.parametrize("n", [1, 31, 33, 1000, LINE - 33, LINE - 1, LINE, LINE + 1, LINE + 31, LINE + 32, LINE + 33,
                               LINE + 127, LINE + 4097])
def test_probe_and_fallback(ctx_mat, n):
    ctx, g = ctx_mat
    rows = _rows(n, n)
    raw, exact, got = (np.stack([v.cpu().numpy() for v in ctx.glass_eval(g, *rows, mode=m)], 1)
                       for m in ("mlp_raw", "exact", "mlp"))
    nb = (n + 31) // 32
    ctr = torch.zeros(nb, 4, dtype=torch.int32, device="cuda")
    ctr[:, 0] = torch.arange(nb, dtype=torch.int32, device="cuda")
    ctr[:, 3] = 0x10004
    word = ctx.philox(ctr, 0x5EED, 0x50524F42).cpu().numpy().view(np.uint32)[:, 0]
    length = np.minimum(32, n - 32 * np.arange(nb))
    probe = 32 * np.arange(nb) + word % length.astype(np.uint32)
    batch = np.arange(n) // 32
    s, d = rows[2].cpu().numpy(), rows[3].cpu().numpy()
    outside = np.zeros(nb, bool)
    outside[batch[(s > 1) | (d < 0.002) | (d > np.float32(0.010))]] = True
    err = np.abs(raw[probe] - exact[probe]).max(1)
    clear = outside | (np.abs(err - 1e-3) >= 1e-6)
    serve = (~outside & (err <= 1e-3))[batch]
    clear = clear[batch]
    assert np.array_equal(got[clear & serve], raw[clear & serve])
    assert np.allclose(got[clear & ~serve], exact[clear & ~serve], rtol=1e-5, atol=1e-6)
    print(f"{serve.mean():.2f} of the rows served by the network")


@pytest.mark.parametrize("n", [(1 << 22) - 1, 1 << 22, (1 << 22) + 1, (1 << 22) + 129])
def test_raw_rows_do_not_depend_on_the_call(ctx_mat, n):
    ctx, g = ctx_mat
    rows = _rows(n, 1)
    whole = ctx.glass_eval(g, *rows, mode="mlp_raw")
    for at, end in ((0, 1000), (n // 2 + 7, n // 2 + 100_000), (n - 300, n)):
        part = ctx.glass_eval(g, *(v[at:end].clone() for v in rows), mode="mlp_raw")
        for w, p in zip(whole, part):
            assert torch.equal(w[at:end], p)
