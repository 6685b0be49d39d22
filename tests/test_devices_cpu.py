"""Contexts on two devices of one process: every call works on the second device
as on the first, in whatever order they are made. The library's own objects are
linked with tests/host/fake_cudart.cpp, a runtime that keeps kernel attributes
and memory per device and runs nothing; what the calls return are zeros, what is
tested are their error codes."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
OUT = os.path.join(ROOT, "paper_1912_06474_gb300", "_build")

CALLS = r"""
import ctypes, sys, tempfile, os
from types import SimpleNamespace
import numpy as np, torch
real = ctypes.CDLL
ctypes.CDLL = lambda path, *a, **k: real(sys.argv[1])
torch.cuda.current_stream = lambda device=None: SimpleNamespace(cuda_stream=0)
from paper_1912_06474_gb300 import scenes, sddm
ctypes.CDLL = real
lib = real(sys.argv[1])
what = sys.argv[2]


def context(device, L):
    sc = scenes.tiny_room(L=L, seed=1, coated=True)
    ctx = sddm.Context(device)
    ctx.set_scene(sc)
    ctx.build(grid=(2, 2, 1))
    return sc, ctx


def render(sc, ctx, **k):
    spec = scenes.RenderSpec(16, 8, 1, 3, seed=1, camera=sc.camera)
    ctx.render_host([spec], [np.zeros((8, 16, 3), np.float32)], **k)


def photons(sc, ctx, method="ddm"):
    spec = scenes.RenderSpec(16, 8, 1, 4, seed=1, camera=sc.camera)
    arr, keep = ctx._descs([spec], method, "exact", [np.zeros((8, 16, 3), np.float32).ctypes.data], None, None)
    sddm._check(sddm.lib.sddm_render_photon_map(ctx._h, arr, 1000, 0.1, 0.05, ctypes.byref(sddm.Stats()),
                                                ctypes.byref(sddm.PhotonStats())))


def learned(sc, ctx):
    g = sc.glass_materials()[0]
    n = 100
    rows = [torch.rand(n), torch.zeros(n, dtype=torch.int32), torch.rand(n), torch.full((n,), 0.004)]
    for mode in ("mlp", "mlp_raw"):
        ctx.glass_eval(g, *rows, mode=mode)
    render(sc, ctx, method="ddm", bsdf="mlp")


first, second = context(0, 41), context(1, 256)
both = (first, second, first, second)
if what == "renders":
    for sc, ctx in both:
        render(sc, ctx, method="megakernel")
        render(sc, ctx, method="ddm")
    # no memory for the throughput rows of 256 bins: they stay in shared memory
    lib.fake_limit_alloc(ctypes.c_size_t(1 << 20))
    for device in (0, 1):
        render(*context(device, 256), method="megakernel")
elif what == "photons":
    for sc, ctx in both + (context(0, 64), context(0, 8), first):
        photons(sc, ctx)
        photons(sc, ctx, "megakernel")
elif what == "weights":
    for sc, ctx in both:
        ctx.mlp_set_weights(sc.glass_materials()[0], np.zeros(sddm.MLP_PARAMS, np.float32))
    for sc, ctx in both:
        learned(sc, ctx)
    with tempfile.TemporaryDirectory() as tmp:
        for k, (sc, ctx) in enumerate(both):
            other = both[1 - k % 2][1]
            path = os.path.join(tmp, str(k))
            render(*both[1 - k % 2])           # the other device is current
            ctx.mlp_save(sc.glass_materials()[0], path)
            render(*both[1 - k % 2])
            ctx.mlp_load(sc.glass_materials()[0], path)
            render(*both[1 - k % 2])
            ctx.mlp_get_weights(sc.glass_materials()[0])
            learned(sc, ctx)
elif what == "no memory":
    sc, ctx = context(0, 8)
    ctx.mlp_set_weights(sc.glass_materials()[0], np.zeros(sddm.MLP_PARAMS, np.float32))
    learned(sc, ctx)
    spec = scenes.RenderSpec(2, 1, 1, 1, seed=1, camera=sc.camera)
    lib.fake_limit_alloc(ctypes.c_size_t(1 << 16))
    try:
        out = np.zeros((1, 2, 3), np.float32)
        arr, keep = ctx._descs([spec] * 2000, "megakernel", "exact", [out.ctypes.data] * 2000, None, None)
        sddm._check(sddm.lib.sddm_render(ctx._h, arr, 2000, ctypes.byref(sddm.Stats())))
        sys.exit("the table of 2000 renders fits?")
    except sddm.SddmError:
        pass
    n = 100
    rows = [torch.rand(n), torch.zeros(n, dtype=torch.int32), torch.rand(n), torch.full((n,), 0.004)]
    ctx.glass_eval(sc.glass_materials()[0], *rows, mode="mlp")     # what fits still works
    ctx.render_host([spec], [np.zeros((1, 2, 3), np.float32)], method="megakernel")
elif what == "training":
    for sc, ctx in both:
        ctx.mlp_train(sc.glass_materials()[0], samples=256, steps=2, batch=64)
        learned(sc, ctx)
    for sc, ctx in (context(0, 16), context(1, 16)):   # a gradient is a context's first learned call
        ctx.mlp_grad(torch.zeros(100, 4), torch.zeros(100, 2), torch.zeros(sddm.MLP_PARAMS))
assert lib.fake_launches() > 20
assert lib.fake_optin_launches() > 0, "no launch above 48 KiB"
"""


@pytest.fixture(scope="module")
def fake_library(tmp_path_factory):
    import torch
    if torch.cuda.is_available():
        pytest.skip("the real runtime is here")
    from paper_1912_06474_gb300 import build
    build.build()
    lib = str(tmp_path_factory.mktemp("fake") / "libsddm_fake.so")
    objs = sorted(os.path.join(OUT, f) for f in os.listdir(OUT) if f.endswith(".o"))
    r = subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I", "/usr/local/cuda/include", "-o", lib,
                        os.path.join(ROOT, "tests", "host", "fake_cudart.cpp"), *objs, "-lpthread"],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return lib


@pytest.mark.parametrize("what", ["renders", "photons", "weights", "no memory", "training"])
def test_second_device(fake_library, what):
    r = subprocess.run([sys.executable, "-c", CALLS, fake_library, what], cwd=ROOT, capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
