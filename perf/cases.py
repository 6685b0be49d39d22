"""What a user of this framework has it compute, as measurable cases.

A case is one pass through the package's Python binding: a render call (plain
megakernel or domain decomposition, exact or learned glass), a batched render
call, a photon-mapped render, a table of glass evaluations, one gradient of the
learned glass model, or a short training run of it. The scenes are the
repository's seeded synthetic rooms; sizes are those of its workloads, tests and
benchmark, or smaller and ragged ones.

Every state holds a context of its own with its scene set and built, as a
program that opens a scene has it; the seed changes the geometry, the
materials' curves, the camera, the coloration states and the random stream.
"""
import math

import numpy as np
import torch

from paper_1912_06474_gb300 import scenes, sddm

DEV = "cuda"


# --------------------------------------------------------------------- cases
def _render(scene, L, width, height, spp, depth, method, grid="1x1x1", handoff=0, bsdf="exact", coated=False, n=1,
            tris=0, aov=False, entry="render"):
    return dict(op="render", scene=scene, L=L, width=width, height=height, spp=spp, depth=depth, method=method,
                grid=grid, handoff=handoff, bsdf=bsdf, coated=coated, n=n, tris=tris, aov=aov, entry=entry)


def listed():
    return [
        # the smallest call: the FP64-checkable tiny room, plain method, with the per-sample outputs
        # a denoiser or a checker takes
        dict(_render("tiny", 16, 64, 64, 1, 2, "megakernel", aov=True), name="tiny_plain_64"),
        # an interactive preview of a coated (electrochromic) pane, ragged size, result read back on the host
        dict(_render("tiny", 41, 201, 143, 3, 5, "ddm", "2x2x2", coated=True, entry="host"),
             name="tiny_ddm_coated_host"),
        # many small renders of one room in different glass states, one call (learned glass)
        dict(_render("tiny", 41, 256, 256, 4, 5, "ddm", "1x1x1", bsdf="mlp", n=6), name="tiny_batch_mlp"),
        # the hotel room as benchmarked: domain decomposition, exact glass / learned glass
        dict(_render("hotel", 41, 512, 512, 16, 5, "ddm", "4x4x2", 1), name="hotel_ddm_exact"),
        dict(_render("hotel", 41, 512, 512, 16, 5, "ddm", "4x4x2", 1, "mlp"), name="hotel_ddm_mlp"),
        # the same room by the plain global-BVH method
        dict(_render("hotel", 41, 512, 512, 4, 5, "megakernel"), name="hotel_plain"),
        # a final frame of the facade room at a tenth of its triangles: deep paths, 81 bins, 256 subdomains
        dict(_render("facade", 81, 960, 540, 4, 8, "ddm", "8x8x4", 1, "mlp", tris=500_000), name="facade_ddm_mlp"),
        # global illumination by photon mapping through the subdomain queues, global and caustic maps
        dict(op="photon", scene="hotel", L=41, width=256, height=256, spp=4, depth=5, method="ddm", grid="4x4x2",
             photons=1 << 18, radius=0.1, caustic=0.05, passes=1, name="hotel_photon_map"),
        # a dense table of the learned glass model (angle, wavelength, state, thickness) with its probe and fallback
        dict(op="glass", L=41, n=1 << 22, mode="mlp", coated=False, name="glass_table_mlp"),
        # the exact coated pane at an odd number of angles, as a designer of a film stack samples it
        dict(op="glass", L=81, n=262_147, mode="exact", coated=True, name="glass_table_coated"),
        # one forward and backward pass of the learned glass model on a batch of the default size
        dict(op="grad", n=8192, name="surrogate_grad"),
        # the start of training the learned glass model at the default batch
        dict(op="train", steps=300, batch=8192, samples=1 << 18, L=41, name="surrogate_train"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["tiny", "tiny", "hotel", "hotel", "facade", "photon", "glass", "grad", "train"])
    if op == "glass":
        mode = rng.choice(["exact", "mlp", "mlp_raw"])
        coated = rng.random() < 0.4
        return dict(op="glass", L=rng.choice([16, 41, 81]), n=_log(rng, 100, 1 << (20 if coated else 22)), mode=mode,
                    coated=coated)
    if op == "grad":
        return dict(op="grad", n=_log(rng, 64, 1 << 16))
    if op == "train":
        return dict(op="train", steps=_log(rng, 20, 400), batch=64 * _log(rng, 4, 128), samples=_log(rng, 4096, 1 << 18),
                    L=rng.choice([16, 41, 81]))
    if op == "photon":
        return dict(op="photon", scene=rng.choice(["tiny", "hotel"]), L=rng.choice([16, 41]),
                    width=_log(rng, 32, 256), height=_log(rng, 32, 256), spp=rng.randint(1, 4), depth=rng.randint(2, 5),
                    method=rng.choice(["ddm", "megakernel"]), grid=rng.choice(["1x1x1", "2x2x2", "4x4x2"]),
                    photons=_log(rng, 2000, 1 << 18), radius=0.1, caustic=rng.choice([0.0, 0.05]),
                    passes=rng.choice([1, 1, 3]))
    method = rng.choice(["ddm", "ddm", "megakernel"])
    bsdf = rng.choice(["exact", "mlp"]) if method == "ddm" else "exact"
    if op == "tiny":
        entry = rng.choice(["render", "host", "noalloc"] if method == "megakernel" else ["render", "host"])
        coated = rng.random() < 0.3
        return _render("tiny", rng.choice([8, 16, 41]), _log(rng, 32, 400), _log(rng, 32, 400), rng.randint(1, 6),
                       rng.randint(1, 6), method, rng.choice(["1x1x1", "2x2x2", "4x4x2"]), rng.choice([0, 1]), bsdf,
                       coated, 1 if entry == "noalloc" else rng.randint(1, 4), entry=entry,
                       aov=entry == "render" and rng.random() < 0.5)
    if op == "hotel":
        side = _log(rng, 48, 512)
        return _render("hotel", rng.choice([16, 31, 41]), side, rng.randint(32, 512), rng.randint(1, 8),
                       rng.randint(2, 6), method, rng.choice(["1x1x1", "2x2x2", "4x4x2"]), rng.choice([0, 1, 2]), bsdf,
                       n=1)
    return _render("facade", rng.choice([41, 81]), _log(rng, 64, 640), _log(rng, 36, 360), rng.randint(1, 4),
                   rng.randint(3, 8), "ddm", rng.choice(["4x4x2", "8x8x4"]), 1, bsdf, tris=_log(rng, 50_000, 500_000))


# -------------------------------------------------------------------- states
def _scene_of(case, seed):
    if case.get("scene") == "hotel":
        return scenes.hotel_room(L=case["L"], seed=seed % 1000)
    if case.get("scene") == "facade":
        return scenes.facade_room(L=case["L"], seed=seed % 1000, target_tris=case["tris"])
    return scenes.tiny_room(L=case["L"], seed=seed % 1000, coated=case.get("coated", False))


def _grid(case):
    return tuple(int(x) for x in case.get("grid", "1x1x1").split("x"))


def _specs(case, scene, seed):
    """The renders of a call: each with a camera near the room's own and glass states of its own; in a batch the
    sizes differ from render to render."""
    rng = np.random.default_rng(seed + 17)
    out = []
    for r in range(case.get("n", 1)):
        base = scene.camera
        look = [float(x + rng.uniform(-0.2, 0.2)) for x in base.look]
        cam = scenes.Camera(pos=tuple(base.pos), look=tuple(look), up=tuple(base.up), vfov_deg=base.vfov_deg)
        w, h, spp = case["width"], case["height"], case["spp"]
        if r % 3 == 1:
            w, h = max(1, w // 2), max(1, h // 2)
        elif r % 3 == 2:
            w, h, spp = max(1, (3 * w) // 4), h, spp + 1
        out.append(scenes.RenderSpec(w, h, spp, case["depth"], seed=seed & 0xFFFF, render_id=r, camera=cam,
                                     glass_s={g: float(rng.uniform(0, 1)) for g in scene.glass_materials()}))
    return out


def _context(case, seed):
    scene = _scene_of(case, seed)
    ctx = sddm.Context(0)
    ctx.set_scene(scene)
    ctx.build(grid=_grid(case), handoff_waves=case.get("handoff", 0))
    if case.get("bsdf") == "mlp" or case.get("mode") in ("mlp", "mlp_raw"):
        ctx.mlp_train(scene.glass_materials()[0], seed=7)     # every pane of a scene shares its glass curves
    return scene, ctx


def _xavier(gen):
    p = torch.zeros(sddm.MLP_PARAMS, device=DEV)
    for lo, hi, fan in ((0, 256, 68), (320, 4416, 128), (4480, 8576, 128), (8640, 8768, 66)):
        b = math.sqrt(6.0 / fan)
        p[lo:hi] = (torch.rand(hi - lo, generator=gen, device=DEV) * 2 - 1) * b
    for lo, hi in ((256, 320), (4416, 4480), (8576, 8640), (8768, 8770)):
        p[lo:hi] = (torch.rand(hi - lo, generator=gen, device=DEV) * 2 - 1) * 0.1
    return p


def prepare(case, seed):
    op = case["op"]
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    if op == "grad":
        scene, ctx = _context(dict(scene="tiny", L=16), seed)
        n = case["n"]
        X = torch.rand(n, 4, generator=gen, device=DEV) * 2 - 1
        # targets as in training: log(R + 1e-3), log(T + 1e-3)
        Y = torch.log(torch.rand(n, 2, generator=gen, device=DEV) + 1e-3)
        return dict(case=case, ctx=ctx, X=X, Y=Y, p=_xavier(gen))
    scene, ctx = _context(case, seed)
    st = dict(case=case, ctx=ctx, scene=scene)
    if op == "glass":
        n = case["n"]
        st["cos"] = torch.rand(n, generator=gen, device=DEV)
        st["bin"] = torch.randint(0, case["L"], (n,), generator=gen, device=DEV, dtype=torch.int32)
        st["s"] = torch.rand(n, generator=gen, device=DEV)
        st["d"] = torch.rand(n, generator=gen, device=DEV) * 0.008 + 0.002
        st["mat"] = scene.glass_materials()[0]
    elif op == "train":
        st["mat"] = scene.glass_materials()[0]
        st["seed"] = seed & 0xFFFF
    else:
        st["specs"] = _specs(case, scene, seed)
        if case.get("entry") == "host":
            st["outs"] = [torch.empty((s.height, s.width, 3), pin_memory=True) for s in st["specs"]]
        elif case.get("entry") == "noalloc":
            st["outs"] = [torch.empty((s.height, s.width, 3), device=DEV) for s in st["specs"]]
    return st


def run(state):
    case, ctx = state["case"], state["ctx"]
    op = case["op"]
    if op == "grad":
        grad, loss = ctx.mlp_grad(state["X"], state["Y"], state["p"])
        return dict(grad=grad, loss=loss)
    if op == "train":
        rep = ctx.mlp_train(state["mat"], samples=case["samples"], steps=case["steps"], batch=case["batch"],
                            seed=state["seed"])
        return dict(weights=ctx.mlp_get_weights(state["mat"]), loss=rep["final_loss"])
    if op == "glass":
        R, T = ctx.glass_eval(state["mat"], state["cos"], state["bin"], state["s"], state["d"], mode=case["mode"])
        return dict(R=R, T=T)
    if op == "photon":
        spec = state["specs"][0]
        if case["passes"] > 1:
            img, _, _ = ctx.render_progressive_photon_map(spec, case["passes"], case["photons"], case["radius"],
                                                          method=case["method"], caustic_radius=case["caustic"])
        else:
            img, _, _ = ctx.render_photon_map(spec, case["photons"], case["radius"], method=case["method"],
                                              caustic_radius=case["caustic"])
        return dict(image=img)
    if case["entry"] == "host":
        ctx.render_host(state["specs"], state["outs"], method=case["method"], bsdf=case["bsdf"])
        return dict(images=state["outs"])
    if case["entry"] == "noalloc":
        ctx.render_noalloc(state["specs"][0], state["outs"][0])
        return dict(images=state["outs"])
    if case["aov"]:
        imgs, _, (sx, prim) = ctx.render(state["specs"], method=case["method"], bsdf=case["bsdf"], aov=True)
        return dict(images=imgs, samples=sx, prims=prim)
    imgs, _ = ctx.render(state["specs"], method=case["method"], bsdf=case["bsdf"])
    return dict(images=imgs)


# ---------------------------------------------------------------------- work
def _paths(case):
    total = 0
    for r in range(case.get("n", 1)):
        w, h, spp = case["width"], case["height"], case["spp"]
        if r % 3 == 1:
            w, h = max(1, w // 2), max(1, h // 2)
        elif r % 3 == 2:
            w, spp = max(1, (3 * w) // 4), spp + 1
        total += w * h * spp
    return total


_MLP_FLOP = 2 * (4 * 64 + 64 * 64 + 64 * 64 + 64 * 2)


def work(case):
    """What a pass cannot do without. A render reads its scene once (48 B a triangle, 32 B a child box for half as
    many leaves) and writes its pixels, and works through its paths: about 2 segments a vertex (extension and shadow
    ray), each of some 8 levels of two boxes (36 flop) and 4 triangles (60 flop), and some 12 flop a bin and vertex."""
    op = case["op"]
    if op == "grad":
        return dict(bytes=case["n"] * 24 + 2 * 4 * sddm.MLP_PARAMS, flops=3 * _MLP_FLOP * case["n"])
    if op == "train":
        rows = case["steps"] * case["batch"]
        return dict(bytes=rows * 24 + case["steps"] * 6 * 4 * sddm.MLP_PARAMS, flops=3 * _MLP_FLOP * rows)
    if op == "glass":
        films = 3 * 250 if case["coated"] else 0
        net = _MLP_FLOP if case["mode"] != "exact" else 0
        return dict(bytes=case["n"] * 24, flops=case["n"] * (100 + films + net))
    tris = {"tiny": 38, "hotel": 200_522, "facade": case.get("tris", 0)}[case["scene"]]
    levels = 1 + max(1, math.ceil(math.log2(max(tris, 2) / 4)) // 2)
    paths = _paths(case) * case.get("passes", 1)
    vertices = paths * (1 + 0.7 * (case["depth"] - 1))
    flops = vertices * (2 * (levels * 36 + 4 * 60) + 12 * case["L"])
    byts = 80 * tris + 12 * _paths(case) / case["spp"]
    if op == "photon":
        ph = case["photons"] * case["passes"]
        hits = ph * (1 + 0.7 * (case["depth"] - 2))
        flops += hits * (levels * 36 + 4 * 60 + 4 * case["L"])
        byts += hits * (32 + 4 * case["L"]) * 2
    elif case.get("aov"):
        byts += 16 * paths
    return dict(bytes=byts, flops=flops)


# -------------------------------------------------------- values in 64 bits
def _f64(a):
    return torch.as_tensor(np.asarray(a, np.float64), device=DEV)


def _slab(c, n, alpha, lam, d):
    """R, T of an absorbing plane-parallel slab in air (multiple reflections, incoherent)."""
    c = c.clamp(1e-8, 1.0)
    s2 = 1.0 - c * c
    m = torch.complex(n, alpha * lam * 1e-9 / (4 * math.pi))
    ct = torch.sqrt(1.0 - s2 / (m * m))
    rho = (((c - m * ct) / (c + m * ct)).abs() ** 2, ((m * c - ct) / (m * c + ct)).abs() ** 2)
    tau = torch.exp(-alpha * d / torch.sqrt(1.0 - s2 / (n * n)))
    R = T = 0.0
    for r in rho:
        den = 1.0 / (1.0 - (r * tau) ** 2)
        R = R + 0.5 * (r + (1 - r) ** 2 * r * tau ** 2 * den)
        T = T + 0.5 * (1 - r) ** 2 * tau * den
    return R, T


def _coated(c, n, alpha, lam, d, films):
    """R, T of a slab coated on both faces: films = [(complex index, thickness in nm), ...], outermost first."""
    c = c.clamp(1e-8, 1.0)
    s2 = 1.0 - c * c
    cs = torch.sqrt(1.0 - s2 / (n * n))
    tau = torch.exp(-alpha * d / cs)
    R = T = 0.0
    for pol in (0, 1):
        e0 = c if pol == 0 else 1.0 / c
        es = n * cs if pol == 0 else n / cs
        one, zero = torch.ones_like(n).to(torch.complex128), torch.zeros_like(n).to(torch.complex128)
        fwd, bwd = (one, zero, zero, one), (one, zero, zero, one)
        for m, t in films:
            ct = torch.sqrt(1.0 - s2 / (m * m))
            ct = torch.where((m * ct).imag < 0, -ct, ct)
            eta = m * ct if pol == 0 else m / ct
            delta = 2 * math.pi * t / lam * m * ct
            a, b, g = torch.cos(delta), -1j * torch.sin(delta) / eta, -1j * eta * torch.sin(delta)
            p, q, r, s = fwd
            fwd = (p * a + q * g, p * b + q * a, r * a + s * g, r * b + s * a)
            p, q, r, s = bwd
            bwd = (a * p + b * r, a * q + b * s, g * p + a * r, g * q + a * s)

        def face(M, ei, et):
            B, C = M[0] + et * M[1], M[2] + et * M[3]
            den = (ei * B + C).abs() ** 2
            return (ei * B - C).abs() ** 2 / den, 4 * ei * et / den
        Ra, Ta = face(fwd, e0, es)
        Rg, Tg = face(bwd, es, e0)
        den = 1.0 / (1.0 - (Rg * tau) ** 2)
        R = R + 0.5 * (Ra + Ta * Tg * Rg * tau ** 2 * den)
        T = T + 0.5 * Ta * Tg * tau * den
    return R, T


def _pane_rt(scene, mat, bins, c, s, d):
    """R, T of glass material `mat` at wavelength bins `bins` (tensors that broadcast)."""
    m = scene.materials[mat]
    lam = _f64(scene.lam)[bins]
    n, alpha = _f64(m.n)[bins], _f64(m.alpha_clear)[bins] + s * _f64(m.dalpha)[bins]
    if not m.layers:
        return _slab(c, n, alpha, lam, d)
    films = [(torch.complex(*torch.broadcast_tensors(_f64(f["n"])[bins], _f64(f["k"])[bins] + s * _f64(f["dk"])[bins])),
              float(np.float32(f["t_nm"]))) for f in m.layers]
    return _coated(c, n, alpha, lam, d, films)


def _philox(ctr, k0, k1):
    """Philox4x32-10 of four int64 counter words."""
    M32 = 0xFFFFFFFF
    c = list(ctr)
    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32

        def mul(a, b):      # 32 x 32 -> (hi, lo), without overflowing a signed 64-bit product
            lo = a * (b & 0xFFFF)
            hi = a * (b >> 16) + (lo >> 16)
            return (hi >> 16) & M32, ((hi << 16) | (lo & 0xFFFF)) & M32
        h0, l0 = mul(c[0], 0xD2511F53)
        h1, l1 = mul(c[2], 0xCD9E8D57)
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
    return [(x >> 8).double() / 16777216.0 for x in c]


def _unit(v):
    return v / v.norm(dim=-1, keepdim=True)


def _tiny_samples(scene, spec, first, count):
    """XYZ of the samples [first, first + count) of a render of a room of a few dozen triangles with Lambertian
    walls, one pane and emitters: path tracing with next-event estimation, every triangle tested for every ray."""
    V, F = _f64(scene.V), torch.as_tensor(np.asarray(scene.F, np.int64), device=DEV)
    mat = torch.as_tensor(np.asarray(scene.mat_id, np.int64), device=DEV)
    obj = torch.as_tensor(np.asarray(scene.obj_id, np.int64), device=DEV)
    kind = torch.as_tensor([m.kind for m in scene.materials], device=DEV)
    p0, e1, e2 = V[F[:, 0]], V[F[:, 1]] - V[F[:, 0]], V[F[:, 2]] - V[F[:, 0]]
    cr = torch.linalg.cross(e1, e2)
    N = _unit(cr)
    lights = torch.nonzero(kind[mat] == scenes.EMITTER).flatten()
    area = 0.5 * cr[lights].norm(dim=1)
    cdf = torch.cumsum(area, 0) / area.sum()
    pane = scene.glass_materials()[0]
    pane_s = float(np.float32(spec.glass_s[pane]))
    pane_d = float(np.float32(scene.materials[pane].thickness_m))
    bins = torch.arange(scene.L, device=DEV)
    rho = torch.stack([_f64(m.rho if m.rho is not None else np.zeros(scene.L)) for m in scene.materials])
    Le = torch.stack([_f64(m.Le if m.Le is not None else np.zeros(scene.L)) for m in scene.materials])
    wcmf = _f64(scene.quad_w)[:, None] * _f64(scene.cmf)
    inf = float("inf")

    def hits(o, d):
        """Distance to every triangle along every ray, inf where it is not met."""
        out = torch.empty(o.shape[0], F.shape[0], device=DEV, dtype=torch.float64)
        for t in range(F.shape[0]):
            h = torch.linalg.cross(d, e2[t].expand_as(d))
            a = h @ e1[t]
            s = o - p0[t]
            u = (s * h).sum(1) / a
            q = torch.linalg.cross(s, e1[t].expand_as(s))
            v = (d * q).sum(1) / a
            dist = (q @ e2[t]) / a
            ok = (a != 0) & (u >= 0) & (v >= 0) & (u + v <= 1) & (dist > 0)
            out[:, t] = torch.where(ok, dist, torch.full_like(dist, inf))
        return out

    k = torch.arange(first, first + count, device=DEV)
    p, j = k // spec.spp, k % spec.spp

    def rand(b, slot):
        z = torch.zeros_like(p)
        return _philox([p, j, z + b, z + slot], spec.seed, spec.render_id)

    f32 = lambda v: torch.tensor([float(np.float32(x)) for x in v], device=DEV, dtype=torch.float64)  # noqa: E731
    cam = spec.camera
    fwd = _unit(f32(cam.look) - f32(cam.pos))
    right = _unit(torch.linalg.cross(fwd, f32(cam.up)))
    up = torch.linalg.cross(right, fwd)
    ty = math.tan(0.5 * math.radians(cam.vfov_deg))
    u = rand(0, 0x10000)
    nx = 2 * ((p % spec.width) + u[0]) / spec.width - 1
    ny = 1 - 2 * ((p // spec.width) + u[1]) / spec.height
    d = _unit(fwd + nx[:, None] * ty * spec.width / spec.height * right + ny[:, None] * ty * up)
    o = f32(cam.pos).expand_as(d)
    T = torch.ones(count, scene.L, device=DEV, dtype=torch.float64)
    xyz = torch.zeros(count, 3, device=DEV, dtype=torch.float64)
    prim_x = torch.full((count,), -1, device=DEV)
    obj_x = torch.full((count,), -1, device=DEV)
    spec_prev = torch.ones(count, dtype=torch.bool, device=DEV)
    live = torch.arange(count, device=DEV)
    ar = torch.arange(F.shape[0], device=DEV)
    off = float(np.float32(1e-4))
    for b in range(1, spec.max_depth + 1):
        if not live.numel():
            break
        h = hits(o, d)
        h[(ar[None] == prim_x[:, None]) | (obj[None] == obj_x[:, None])] = inf
        dist, prim = h.min(dim=1)
        keep = torch.isfinite(dist)
        m, ng = mat[prim], N[prim]
        cd = (d * ng).sum(1)
        kd = kind[m]
        seen = keep & (kd == scenes.EMITTER) & (cd < 0) & (spec_prev | (b == 1))
        xyz[live[seen]] += (T[seen] * Le[m[seen]]) @ wcmf
        keep &= kd != scenes.EMITTER
        x = o + torch.where(keep, dist, torch.zeros_like(dist))[:, None] * d
        ns = torch.where((cd < 0)[:, None], ng, -ng)

        def r_of(slot):
            z = torch.zeros_like(live)
            return _philox([p[live], j[live], z + b, z + slot], spec.seed, spec.render_id)
        # next-event light at diffuse vertices
        dif = keep & (kd == scenes.LAMBERT)
        ul = r_of(0x10002)
        li = torch.searchsorted(cdf, ul[0].contiguous(), right=True).clamp(max=lights.numel() - 1)
        lt = lights[li]
        su = torch.sqrt(ul[1])
        b0, b1 = 1 - su, ul[2] * su
        y = p0[lt] + b1[:, None] * e1[lt] + (1 - b0 - b1)[:, None] * e2[lt]
        xo = x + off * ns
        w = y - xo
        far = w.norm(dim=1)
        w = w / far[:, None]
        cx, cy = (ns * w).sum(1), -(N[lt] * w).sum(1)
        lit = torch.nonzero(dif & (cx > 0) & (cy > 0)).flatten()
        if lit.numel():
            hs = hits(xo[lit], w[lit])
            met = (hs <= ((1 - 1e-4) * far[lit])[:, None]) & (ar[None] != prim[lit][:, None])
            glass = kind[mat][None] == scenes.GLASS
            clear = ~(met & ~glass).any(1)
            through = met & glass & ((w[lit] @ N.T) < 0)
            tr = torch.ones(lit.numel(), scene.L, device=DEV, dtype=torch.float64)
            cross = torch.nonzero(through.any(1)).flatten()
            if cross.numel():
                tri = through[cross].float().argmax(1)
                cc = -(w[lit[cross]] * N[tri]).sum(1)
                tr[cross] = _pane_rt(scene, pane, bins[None], cc[:, None], pane_s, pane_d)[1]
            G = cx[lit] * cy[lit] / far[lit] ** 2 * area.sum() / math.pi * clear
            xyz[live[lit]] += (T[lit] * rho[m[lit]] * Le[mat[lt[lit]]] * G[:, None] * tr) @ wcmf
        # the next direction
        if b == spec.max_depth:
            break
        ub = r_of(0x10001)
        A, B = 2 * ub[0] - 1, 2 * ub[1] - 1
        wide = A.abs() > B.abs()
        rr = torch.where(wide, A, B)
        phi = torch.where(wide, math.pi / 4 * (B / A), math.pi / 2 - math.pi / 4 * (A / B))
        dx, dy = rr * torch.cos(phi), rr * torch.sin(phi)
        dz = torch.sqrt((1 - dx * dx - dy * dy).clamp(min=0))
        sg = torch.where(ns[:, 2] >= 0, 1.0, -1.0).double()
        aa = -1 / (sg + ns[:, 2])
        bb = ns[:, 0] * ns[:, 1] * aa
        t1 = torch.stack([1 + sg * ns[:, 0] ** 2 * aa, sg * bb, -sg * ns[:, 0]], 1)
        t2 = torch.stack([bb, sg + ns[:, 1] ** 2 * aa, -ns[:, 1]], 1)
        diffuse_d = dx[:, None] * t1 + dy[:, None] * t2 + dz[:, None] * ns
        gl = keep & (kd == scenes.GLASS)
        mirror = d - 2 * cd[:, None] * ng
        refl = torch.zeros_like(gl)
        gi = torch.nonzero(gl).flatten()
        W = rho[m]
        if gi.numel():
            c = cd[gi].abs()[:, None]
            n = _f64(scene.materials[pane].n)[None]
            ct = torch.sqrt(1 - (1 - c * c) / (n * n))
            rs, rp = ((c - n * ct) / (c + n * ct)) ** 2, ((n * c - ct) / (n * c + ct)) ** 2
            pr = (0.5 * (2 * rs / (1 + rs) + 2 * rp / (1 + rp))).mean(1).clamp(0.05, 0.95)
            refl[gi] = r_of(0x10003)[0][gi] < pr
            R, Tt = _pane_rt(scene, pane, bins[None], c, pane_s, pane_d)
            back = refl[gi][:, None]
            W[gi] = torch.where(back, R, Tt) / torch.where(back, pr[:, None], 1 - pr[:, None])
        thru = gl & ~refl
        d = torch.where(dif[:, None], diffuse_d, torch.where(refl[:, None], mirror, d))
        o = torch.where(thru[:, None], x - off * ns, x + off * ns)
        prim_x = prim
        obj_x = torch.where(thru, obj[prim], torch.full_like(prim, -1))
        T = T * W
        spec_prev = gl
        keep = torch.nonzero(keep).flatten()
        live, o, d, T = live[keep], o[keep], d[keep], T[keep]
        prim_x, obj_x, spec_prev = prim_x[keep], obj_x[keep], spec_prev[keep]
    return xyz


def exact(case, seed):
    op = case["op"]
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    if op == "grad":
        n = case["n"]
        X = (torch.rand(n, 4, generator=gen, device=DEV) * 2 - 1).double()
        Y = torch.log(torch.rand(n, 2, generator=gen, device=DEV) + 1e-3).double()
        p = _xavier(gen).double().requires_grad_(True)
        h, at = X, 0
        for o, i in ((64, 4), (64, 64), (64, 64), (2, 64)):
            W, b = p[at:at + o * i].view(o, i), p[at + o * i:at + o * i + o]
            h = h @ W.T + b
            at += o * i + o
            if o == 64:
                h = torch.nn.functional.silu(h)
        loss = ((h - Y) ** 2).mean()
        loss.backward()
        return dict(grad=p.grad, loss=loss.detach().reshape(1))
    if op == "glass":
        scene, n = _scene_of(case, seed), case["n"]
        c = torch.rand(n, generator=gen, device=DEV).double()
        bins = torch.randint(0, case["L"], (n,), generator=gen, device=DEV, dtype=torch.int32).long()
        s = torch.rand(n, generator=gen, device=DEV).double()
        d = (torch.rand(n, generator=gen, device=DEV) * 0.008 + 0.002).double()
        R, T = _pane_rt(scene, scene.glass_materials()[0], bins, c, s, d)
        return dict(R=R, T=T)
    if op == "render" and case["scene"] == "tiny" and _paths(case) * case["depth"] <= 1 << 23:
        scene = _scene_of(case, seed)
        imgs, samples = [], []
        for spec in _specs(case, scene, seed):
            parts = [_tiny_samples(scene, spec, a, min(1 << 17, spec.n_paths - a))
                     for a in range(0, spec.n_paths, 1 << 17)]
            xyz = torch.cat(parts)
            samples.append(xyz)
            imgs.append(xyz.view(spec.height, spec.width, spec.spp, 3).mean(2))
        if case["aov"]:
            return dict(images=imgs, samples=samples, prims=[None] * len(imgs))
        return dict(images=imgs)
    # rooms of hundreds of thousands of triangles, photon maps: over 20 s in plain 64-bit torch; training: the weights
    # after some hundred steps of Adam are no function that 64 bits follow to float accuracy
    return None
