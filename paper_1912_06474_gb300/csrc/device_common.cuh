// Device building blocks of the path tracer: random stream, ray/box and
// ray/triangle tests, BVH traversal, spectral optics, sampling, compensated sums.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "sddm_internal.h"

namespace sddm {

// ------------------------------------------------- overlapped kernel launches
// First statement of a kernel launched by launch_after: let the kernel after it be
// launched, and wait until the kernel before it is done and its writes are seen.
__device__ __forceinline__ void grid_entry() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}
// Launch a kernel that may be brought in while the stream's kernel before it
// drains: its blocks wait for that kernel themselves (grid_entry, before they read
// anything it wrote), so that launch latency and start-up overlap. After anything
// but a kernel (a memset, an event), or with early = false, it is an ordinary launch.
template <typename... P, typename... A>
inline cudaError_t launch_after(bool early, void (*kernel)(P...), unsigned blocks, unsigned threads, size_t smem,
                                cudaStream_t stream, A &&...args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = early ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

// ----------------------------------------------------------- vector helpers
struct V3 {
    float x, y, z;
};
__device__ __forceinline__ V3 v3(float x, float y, float z) { return V3{x, y, z}; }
__device__ __forceinline__ V3 operator+(V3 a, V3 b) { return v3(a.x + b.x, a.y + b.y, a.z + b.z); }
__device__ __forceinline__ V3 operator-(V3 a, V3 b) { return v3(a.x - b.x, a.y - b.y, a.z - b.z); }
__device__ __forceinline__ V3 operator*(float s, V3 a) { return v3(s * a.x, s * a.y, s * a.z); }
__device__ __forceinline__ float dot(V3 a, V3 b) { return a.x * b.x + a.y * b.y + a.z * b.z; }
__device__ __forceinline__ V3 cross(V3 a, V3 b) {
    return v3(a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x);
}
__device__ __forceinline__ V3 normalize(V3 a) {
    float inv = 1.0f / sqrtf(dot(a, a));
    return inv * a;
}
__device__ __forceinline__ V3 xyz(float4 f) { return v3(f.x, f.y, f.z); }

// ------------------------------------------------------------- Philox4x32-10
// Counter-based generator of Salmon et al. (SC'11): ten rounds of two
// 32x32->64 products whose high halves are xored with the other counter words
// and the round key; the key advances by the Weyl constants between rounds.
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint32_t k0, uint32_t k1) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        if (r > 0) {
            k0 += 0x9E3779B9u;
            k1 += 0xBB67AE85u;
        }
        uint32_t lo0 = 0xD2511F53u * c.x, hi0 = __umulhi(0xD2511F53u, c.x);
        uint32_t lo1 = 0xCD9E8D57u * c.z, hi1 = __umulhi(0xCD9E8D57u, c.z);
        c = make_uint4(hi1 ^ c.y ^ k0, lo1, hi0 ^ c.w ^ k1, lo0);
    }
    return c;
}
// Top 24 bits as a uniform in [0, 1): exact in float.
__device__ __forceinline__ float u01(uint32_t x) { return (float)(x >> 8) * (1.0f / 16777216.0f); }

// ---------------------------------------------------------------- BVH nodes
// Node = 4 float4: (c0.lo.x, c0.hi.x, c0.lo.y, c0.hi.y) (c1 same) (c0.lo.z, c0.hi.z,
// c1.lo.z, c1.hi.z) (child0, child1 as int bits). child >= 0: node index;
// child < 0: leaf, ~child = (first triangle << 4) | count.
// Triangle = 3 float4, one per axis: (v0, v1, v2 along x, key) (along y, key)
// (along z, key), key = id, with bit 30 set on glass: the vertices themselves,
// so that triangles sharing an edge see bit-identical endpoints. A ray reads
// the rows in the order of its own axes (below).
constexpr int kTriIdMask = (1 << 30) - 1;
constexpr int kTriGlassBit = 1 << 30;
struct TriRows {
    float4 x, y, z;   // along the ray's kx, ky, kz
    __device__ __forceinline__ int key() const { return __float_as_int(x.w); }
};

// A ray with what its box and triangle tests need: reciprocal direction and
// origin times it (boxes), and the set-up of the watertight triangle test of
// Woop, Benthin and Wald (JCGT 2013): the axis kz along which the direction is
// largest, the next two kx, ky in cyclic order, the shear (sx, sy) = (d[kx],
// d[ky]) / d[kz] that maps the ray onto the z axis of a frame centred on its
// origin, the scale sz = 1 / d[kz] (|d[kz]| >= 1/sqrt(3) for a unit direction,
// never clamped) and the origin in that axis order. For d[kz] < 0 the method
// swaps kx and ky to keep the winding; exchanging them only negates U, V, W,
// their sum and the scaled distance, each exactly, and the test looks at neither
// sign, so the swap is left out.
struct Ray {
    V3 inv, oi;         // oi = o * inv
    float sx, sy, sz;
    V3 po;              // o along kx, ky, kz
    int k;              // kx | ky << 2 | kz << 4
};
__device__ __forceinline__ float safe_inv(float d) {
    return 1.0f / (fabsf(d) > 1e-20f ? d : copysignf(1e-20f, d));
}
__device__ __forceinline__ float comp(V3 v, int k) { return k == 0 ? v.x : (k == 1 ? v.y : v.z); }
__device__ __forceinline__ Ray make_ray(V3 o, V3 d) {
    Ray r;
    r.inv = v3(safe_inv(d.x), safe_inv(d.y), safe_inv(d.z));
    r.oi = v3(o.x * r.inv.x, o.y * r.inv.y, o.z * r.inv.z);
    const float ax = fabsf(d.x), ay = fabsf(d.y), az = fabsf(d.z);
    const int kz = ax >= ay ? (ax >= az ? 0 : 2) : (ay >= az ? 1 : 2);
    const int kx = kz == 2 ? 0 : kz + 1, ky = kx == 2 ? 0 : kx + 1;
    const float dz = comp(d, kz);
    r.sx = comp(d, kx) / dz;
    r.sy = comp(d, ky) / dz;
    r.sz = comp(r.inv, kz);
    r.po = v3(comp(o, kx), comp(o, ky), comp(o, kz));
    r.k = kx | (ky << 2) | (kz << 4);
    return r;
}
// Triangle record i in the ray's axis order: the permutation is in the
// addresses, not in selects of the nine coordinates.
__device__ __forceinline__ TriRows load_tri(const float4 *__restrict__ tris, int i, const Ray &r) {
    const float4 *tp = tris + 3 * i;
    return TriRows{__ldg(tp + (r.k & 3)), __ldg(tp + ((r.k >> 2) & 3)), __ldg(tp + (r.k >> 4))};
}
// Whether a ray of direction d leaves the (glass) triangle's front side.
__device__ __forceinline__ bool tri_leaving(const float4 *__restrict__ tris, int i, V3 d) {
    const float4 *tp = tris + 3 * i;
    const float4 x = __ldg(tp), y = __ldg(tp + 1), z = __ldg(tp + 2);
    const V3 a = v3(x.x, y.x, z.x);
    return dot(d, cross(v3(x.y, y.y, z.y) - a, v3(x.z, y.z, z.z) - a)) >= 0.0f;
}

// Watertight ray/triangle test (Woop, Benthin, Wald 2013), double sided:
// the vertices are taken relative to the ray origin and sheared so that the
// ray runs along z; the signed edge functions U, V, W of the projected
// triangle decide inside/outside. Each is a difference of two correctly
// rounded products, so a shared edge gives its two triangles edge functions
// of exactly opposite sign and a ray through it cannot slip between them;
// an exact zero is re-evaluated in double precision. Returns the hit
// distance, or +inf.
__device__ __forceinline__ float wt_intersect(const Ray &r, const TriRows &p) {
    const float Az = p.z.x - r.po.z, Bz = p.z.y - r.po.z, Cz = p.z.z - r.po.z;
    const float Ax = fmaf(-r.sx, Az, p.x.x - r.po.x), Ay = fmaf(-r.sy, Az, p.y.x - r.po.y);
    const float Bx = fmaf(-r.sx, Bz, p.x.y - r.po.x), By = fmaf(-r.sy, Bz, p.y.y - r.po.y);
    const float Cx = fmaf(-r.sx, Cz, p.x.z - r.po.x), Cy = fmaf(-r.sy, Cz, p.y.z - r.po.y);
    float U = __fsub_rn(__fmul_rn(Cx, By), __fmul_rn(Cy, Bx));
    float V = __fsub_rn(__fmul_rn(Ax, Cy), __fmul_rn(Ay, Cx));
    float W = __fsub_rn(__fmul_rn(Bx, Ay), __fmul_rn(By, Ax));
    if (U == 0.0f || V == 0.0f || W == 0.0f) {
        U = (float)((double)Cx * (double)By - (double)Cy * (double)Bx);
        V = (float)((double)Ax * (double)Cy - (double)Ay * (double)Cx);
        W = (float)((double)Bx * (double)Ay - (double)By * (double)Ax);
    }
    if (fminf(U, fminf(V, W)) < 0.0f && fmaxf(U, fmaxf(V, W)) > 0.0f) return __int_as_float(0x7f800000);
    const float det = U + V + W;
    if (det == 0.0f) return __int_as_float(0x7f800000);
    const float T = fmaf(U, r.sz * Az, fmaf(V, r.sz * Bz, W * (r.sz * Cz)));
    return T / det;
}

// Three-operand minimum and maximum (one instruction on sm_100 and later, at the
// rate of the two-operand form; a NaN operand is ignored as by fminf / fmaxf).
__device__ __forceinline__ float fmin3(float a, float b, float c) {
    float d;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}
__device__ __forceinline__ float fmax3(float a, float b, float c) {
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

// Slab test of both children of a node against [tmin, tmax]: hit flags and entry distances.
__device__ __forceinline__ void child_boxes(const Ray &r, float4 n0, float4 n1, float4 n2, float tmin, float tmax,
                                            float &t0, float &t1, bool &h0, bool &h1) {
    float ax0 = fmaf(n0.x, r.inv.x, -r.oi.x), ax1 = fmaf(n0.y, r.inv.x, -r.oi.x);
    float ay0 = fmaf(n0.z, r.inv.y, -r.oi.y), ay1 = fmaf(n0.w, r.inv.y, -r.oi.y);
    float az0 = fmaf(n2.x, r.inv.z, -r.oi.z), az1 = fmaf(n2.y, r.inv.z, -r.oi.z);
    float bx0 = fmaf(n1.x, r.inv.x, -r.oi.x), bx1 = fmaf(n1.y, r.inv.x, -r.oi.x);
    float by0 = fmaf(n1.z, r.inv.y, -r.oi.y), by1 = fmaf(n1.w, r.inv.y, -r.oi.y);
    float bz0 = fmaf(n2.z, r.inv.z, -r.oi.z), bz1 = fmaf(n2.w, r.inv.z, -r.oi.z);
    const float alo = fmax3(fminf(ax0, ax1), fminf(ay0, ay1), fmaxf(fminf(az0, az1), tmin));
    const float ahi = fmin3(fmaxf(ax0, ax1), fmaxf(ay0, ay1), fminf(fmaxf(az0, az1), tmax));
    const float blo = fmax3(fminf(bx0, bx1), fminf(by0, by1), fmaxf(fminf(bz0, bz1), tmin));
    const float bhi = fmin3(fmaxf(bx0, bx1), fmaxf(by0, by1), fminf(fmaxf(bz0, bz1), tmax));
    h0 = alo <= ahi;
    h1 = blo <= bhi;
    t0 = alo;
    t1 = blo;
}

struct Hit {
    float t;
    int prim;   // original triangle id, -1 = none
};

// Closest hit with t in (tmin, tmax); ties on t go to the lower triangle id. A
// triangle the ray misses has t = +inf, which is no hit for tmax = +inf either.
// excl_prim: triangle skipped; excl_obj >= 0: every triangle of that object skipped.
// The hierarchy starts at node `root` (0 for the global one).
// With COUNT, interior nodes visited and triangles tested are added to *cnt.
struct TravCount {
    unsigned long long nodes = 0, tris = 0;
};
template <bool COUNT = false>
__device__ __forceinline__ Hit trace_closest(const float4 *__restrict__ nodes, const float4 *__restrict__ tris,
                                             const int *__restrict__ tri_obj, int root, const Ray &r, float tmin,
                                             float tmax, int excl_prim, int excl_obj, TravCount *cnt = nullptr) {
    Hit h;
    h.t = tmax;
    h.prim = -1;
    int stack[kStackSize];
    int sp = 0;
    int node = root;
    for (;;) {
        if (node >= 0) {
            if (COUNT) ++cnt->nodes;
            float4 n0 = __ldg(nodes + 4 * node + 0);
            float4 n1 = __ldg(nodes + 4 * node + 1);
            float4 n2 = __ldg(nodes + 4 * node + 2);
            float4 n3 = __ldg(nodes + 4 * node + 3);
            float ta, tb;
            bool ha, hb;
            child_boxes(r, n0, n1, n2, tmin, h.t, ta, tb, ha, hb);
            int ca = __float_as_int(n3.x), cb = __float_as_int(n3.y);
            if (ha && hb) {
                int near = ta <= tb ? ca : cb, far = ta <= tb ? cb : ca;
                if (sp < kStackSize) stack[sp++] = far;
                node = near;
                continue;
            }
            if (ha) { node = ca; continue; }
            if (hb) { node = cb; continue; }
        } else {
            int v = ~node;
            int first = v >> kLeafBits, count = v & ((1 << kLeafBits) - 1);
            for (int i = 0; i < count; ++i) {
                const TriRows tr = load_tri(tris, first + i, r);
                const int id = tr.key() & kTriIdMask;
                if (id == excl_prim || (excl_obj >= 0 && __ldg(tri_obj + id) == excl_obj)) continue;
                if (COUNT) ++cnt->tris;
                const float t = wt_intersect(r, tr);
                if (t > tmin && (t < h.t || (t == h.t && id < h.prim))) {
                    h.t = t;
                    h.prim = id;
                }
            }
        }
        if (sp == 0) break;
        node = stack[--sp];
    }
    return h;
}

// Shadow query over (tmin, tmax]. Returns true if occluded. Glass triangles
// hit from their front (the ray enters the convex slab) are recorded once per
// slab object in cross_obj/cross_tri (up to kMaxCross; one more occludes);
// glass leaving faces are ignored; any other triangle occludes.
struct Crossings {
    int n;
    int obj[kMaxCross];
    int tri[kMaxCross];
};
template <bool COUNT = false>
__device__ __forceinline__ bool trace_shadow(const float4 *__restrict__ nodes, const float4 *__restrict__ tris,
                                             const int *__restrict__ tri_obj, int root, const Ray &r, V3 d, float tmin,
                                             float tmax, int excl_prim, Crossings &cr, TravCount *cnt = nullptr) {
    int stack[kStackSize];
    int sp = 0;
    int node = root;
    for (;;) {
        if (node >= 0) {
            if (COUNT) ++cnt->nodes;
            float4 n0 = __ldg(nodes + 4 * node + 0);
            float4 n1 = __ldg(nodes + 4 * node + 1);
            float4 n2 = __ldg(nodes + 4 * node + 2);
            float4 n3 = __ldg(nodes + 4 * node + 3);
            float ta, tb;
            bool ha, hb;
            child_boxes(r, n0, n1, n2, tmin, tmax, ta, tb, ha, hb);
            int ca = __float_as_int(n3.x), cb = __float_as_int(n3.y);
            if (ha && hb) {
                if (sp < kStackSize) stack[sp++] = cb;
                node = ca;
                continue;
            }
            if (ha) { node = ca; continue; }
            if (hb) { node = cb; continue; }
        } else {
            int v = ~node;
            int first = v >> kLeafBits, count = v & ((1 << kLeafBits) - 1);
            for (int i = 0; i < count; ++i) {
                const TriRows tr = load_tri(tris, first + i, r);
                const int id = tr.key() & kTriIdMask;
                if (id == excl_prim) continue;
                if (COUNT) ++cnt->tris;
                const float t = wt_intersect(r, tr);
                if (!(t > tmin && t <= tmax)) continue;
                if (!(tr.key() & kTriGlassBit)) return true;
                if (tri_leaving(tris, first + i, d)) continue;
                const int ob = __ldg(tri_obj + id);
                bool seen = false;
                for (int q = 0; q < cr.n; ++q) seen |= cr.obj[q] == ob;
                if (seen) continue;
                if (cr.n >= kMaxCross) return true;
                cr.obj[cr.n] = ob;
                cr.tri[cr.n] = id;
                ++cr.n;
            }
        }
        if (sp == 0) break;
        node = stack[--sp];
    }
    return false;
}

// First device check to fail records its code and two details in the error word.
__device__ __forceinline__ void trace_check_fail(int *err, int code, int x, int y) {
    if (atomicCAS(err, 0, code) == 0) {
        err[1] = x;
        err[2] = y;
    }
}

// A lane's query in a persistent warp: a closest hit in (tmin, tw] (ties on t to
// the lower triangle id) or a shadow query, resumable between rounds.
struct LaneTrav {
    Ray ray;
    float tmin, tw;     // tw shrinks to the closest hit so far
    int node, sp;       // node < 0: standing at a leaf
    int best, ep, eo;   // closest triangle so far; triangle and object to skip (-1 = none)
    bool occ, fin;      // shadow ray blocked; query answered
};

// One while-while round of a warp's queries: an interior phase in which the lanes
// descend until at most 1 / QUORUM of the live ones still do (at most STEPS
// steps), then a leaf phase in which the lanes at a leaf test its triangles.
// All lanes call it; dir() gives a lane's ray direction (glass in front of a
// shadow ray only). CHECKED: every child and leaf index is checked against the
// records there are before it is read (codes 9, 10).
template <bool COUNT, bool CHECKED, int STEPS, int QUORUM, typename DirF>
__device__ __forceinline__ void trav_round(const float4 *__restrict__ nodes, const float4 *__restrict__ tris,
                                           const int *__restrict__ tri_obj, LaneTrav &s, Crossings &cr,
                                           int (&stack)[kStackSize], bool live, bool shadow, DirF &&dir, TravCount &tc, int *err,
                                           int64_t node_cap, int64_t tri_cap) {
    const unsigned full = 0xffffffffu;
    const int n_live = __popc(__ballot_sync(full, live));
#pragma unroll 1
    for (int it = 0; it < STEPS; ++it) {
        const bool act = live && !s.fin && s.node >= 0;
        if (__popc(__ballot_sync(full, act)) * QUORUM <= n_live) break;
        if (act) {
            if (COUNT) ++tc.nodes;
            const float4 n0 = __ldg(nodes + 4 * s.node + 0), n1 = __ldg(nodes + 4 * s.node + 1),
                         n2 = __ldg(nodes + 4 * s.node + 2), n3 = __ldg(nodes + 4 * s.node + 3);
            float ta, tb;
            bool ha, hb;
            child_boxes(s.ray, n0, n1, n2, s.tmin, s.tw, ta, tb, ha, hb);
            int ca = __float_as_int(n3.x), cb = __float_as_int(n3.y);
            if (CHECKED) {
                if (ca >= node_cap) {
                    trace_check_fail(err, 9, s.node, ca);
                    ca = ~0;
                }
                if (cb >= node_cap) {
                    trace_check_fail(err, 9, s.node, cb);
                    cb = ~0;
                }
            }
            if (ha && hb) {
                const bool a_first = shadow || ta <= tb;
                if (s.sp < kStackSize) {
                    stack[s.sp++] = a_first ? cb : ca;
                } else {
                    atomicCAS(err, 0, 5);   // deeper than the builder allows
                }
                s.node = a_first ? ca : cb;
            } else if (ha) {
                s.node = ca;
            } else if (hb) {
                s.node = cb;
            } else if (s.sp == 0) {
                s.fin = true;
            } else {
                s.node = stack[--s.sp];
            }
        }
    }
    if (live && !s.fin && s.node < 0) {
        const int v = ~s.node;
        const int first = v >> kLeafBits;
        int count = v & ((1 << kLeafBits) - 1);
        if (CHECKED && (int64_t)first + count > tri_cap) {
            trace_check_fail(err, 10, first, count);
            count = 0;
        }
#pragma unroll 1
        for (int i = first; i < first + count; ++i) {
            const TriRows tri = load_tri(tris, i, s.ray);
            const int id = tri.key() & kTriIdMask;
            if (id == s.ep || (!shadow && s.eo >= 0 && __ldg(tri_obj + id) == s.eo)) continue;
            if (COUNT) ++tc.tris;
            const float t = wt_intersect(s.ray, tri);
            if (!(t > s.tmin && t <= s.tw)) continue;
            if (!shadow) {
                if (t < s.tw || s.best < 0 || id < s.best) {
                    s.tw = t;
                    s.best = id;
                }
                continue;
            }
            if (!(tri.key() & kTriGlassBit)) {
                s.occ = true;
                break;
            }
            if (tri_leaving(tris, i, dir())) continue;
            const int ob = __ldg(tri_obj + id);
            bool seen = false;
#pragma unroll 1
            for (int k = 0; k < cr.n; ++k) seen |= cr.obj[k] == ob;
            if (seen) continue;
            if (cr.n >= kMaxCross) {
                s.occ = true;
                break;
            }
            cr.obj[cr.n] = ob;
            cr.tri[cr.n] = id;
            ++cr.n;
        }
        if (s.occ || s.sp == 0) {
            s.fin = true;
        } else {
            s.node = stack[--s.sp];
        }
    }
}

// ------------------------------------------------------------------- optics
// Fresnel reflectances |r_s|^2, |r_p|^2 for light arriving from vacuum onto a
// medium of complex index n + ik (Eq. 1), cos_i = c in (0, 1], in real
// arithmetic: with a + ib = n~ cos_t, (a + ib)^2 = n^2 - k^2 - sin^2 + 2ink, so
// a b = n k, and
//   Rs = ((a - c)^2 + b^2) / ((a + c)^2 + b^2),
//   Rp = Rs ((a - q)^2 + b^2) / ((a + q)^2 + b^2),  q = sin^2 / cos.
// a or b is taken from the larger-magnitude side of the square root so that
// neither suffers cancellation (k is ~1e-5 for glass, ~1..8 for metals).
__device__ __forceinline__ void fresnel_rs_rp(float c, float n, float k, float &Rs, float &Rp) {
    const float s2 = fmaf(-c, c, 1.0f);
    const float t0 = fmaf(n, n, -fmaf(k, k, s2));
    const float nk = n * k;
    const float r = sqrtf(fmaf(t0, t0, 4.0f * nk * nk));
    float a, b;
    if (t0 >= 0.0f) {
        a = sqrtf(0.5f * (r + t0));
        b = a > 0.0f ? __fdividef(nk, a) : 0.0f;
    } else {
        b = sqrtf(0.5f * (r - t0));
        a = __fdividef(nk, b);
    }
    const float b2 = b * b;
    const float am = a - c, ap = a + c;
    Rs = __fdividef(fmaf(am, am, b2), fmaf(ap, ap, b2));
    const float q = __fdividef(s2, c);
    const float qm = a - q, qp = a + q;
    Rp = Rs * __fdividef(fmaf(qm, qm, b2), fmaf(qp, qp, b2));
}

__device__ __forceinline__ float conductor_F(float c, float n, float k) {
    if (c <= 0.0f) return 1.0f;
    c = fminf(fmaxf(c, 1e-8f), 1.0f);
    float Rs, Rp;
    fresnel_rs_rp(c, n, k, Rs, Rp);
    return 0.5f * (Rs + Rp);
}

// Absorbing plane-parallel slab (Sec. 6 evaluates glass with the Fresnel
// equations; Eq. 1 with k = alpha lambda / 4 pi): interface reflectance rho_j per
// polarisation, internal transmittance tau = exp(-alpha d / cos_t) with the
// real-index refraction angle, and the multiple-reflection sums
//   R_j = rho_j + (1 - rho_j)^2 rho_j tau^2 / (1 - rho_j^2 tau^2)
//   T_j = (1 - rho_j)^2 tau / (1 - rho_j^2 tau^2),   R, T = mean over j.
__device__ __forceinline__ void slab_RT(float c, float lam_nm, float n, float alpha, float thick, float &R,
                                        float &T) {
    if (c <= 0.0f) {
        R = 1.0f;
        T = 0.0f;
        return;
    }
    c = fminf(fmaxf(c, 1e-8f), 1.0f);
    const float k = alpha * lam_nm * (1e-9f / (4.0f * 3.14159265358979f));
    float Rs, Rp;
    fresnel_rs_rp(c, n, k, Rs, Rp);
    const float s2 = fmaf(-c, c, 1.0f);
    const float ctr = __fdividef(sqrtf(fmaf(n, n, -s2)), n);
    const float tau = __expf(-__fdividef(alpha * thick, ctr));
    const float t2 = tau * tau;
    const float ds = __frcp_rn(fmaf(-Rs * Rs, t2, 1.0f)), dp = __frcp_rn(fmaf(-Rp * Rp, t2, 1.0f));
    const float qs = (1.0f - Rs) * (1.0f - Rs), qp = (1.0f - Rp) * (1.0f - Rp);
    R = 0.5f * (fmaf(qs * Rs * t2, ds, Rs) + fmaf(qp * Rp * t2, dp, Rp));
    T = 0.5f * tau * (qs * ds + qp * dp);
}

// ---------------------------------------------------- coated glass (thin films)
// Complex numbers for the thin-film characteristic matrices.
struct Cx {
    float r, i;
};
__device__ __forceinline__ Cx cx(float r, float i = 0.0f) { return Cx{r, i}; }
__device__ __forceinline__ Cx operator+(Cx a, Cx b) { return Cx{a.r + b.r, a.i + b.i}; }
__device__ __forceinline__ Cx operator-(Cx a, Cx b) { return Cx{a.r - b.r, a.i - b.i}; }
__device__ __forceinline__ Cx operator*(Cx a, Cx b) { return Cx{fmaf(a.r, b.r, -a.i * b.i), fmaf(a.r, b.i, a.i * b.r)}; }
__device__ __forceinline__ Cx operator*(float s, Cx a) { return Cx{s * a.r, s * a.i}; }
__device__ __forceinline__ float cx_abs2(Cx a) { return fmaf(a.r, a.r, a.i * a.i); }
__device__ __forceinline__ Cx cx_div(Cx a, Cx b) {
    const float d = __frcp_rn(cx_abs2(b));
    return Cx{d * fmaf(a.r, b.r, a.i * b.i), d * fmaf(a.i, b.r, -a.r * b.i)};
}
__device__ __forceinline__ Cx cx_sqrt(Cx z) {   // principal root
    const float m = sqrtf(sqrtf(cx_abs2(z)));
    const float h = 0.5f * atan2f(z.i, z.r);
    float sh, ch;
    sincosf(h, &sh, &ch);
    return Cx{m * ch, m * sh};
}

// Up to kMaxFilms films per face.
constexpr int kMaxFilms = SDDM_MAX_FILMS;
constexpr int kDenseFilms = 3;   // films of a stack held in registers (glass_rt, DENSE)

// Glass coated on both faces with the same stack of J thin films (outermost
// first): each face is a coherent stack evaluated by its characteristic
// matrix (per film: complex index n + i k, cos theta = sqrt(1 - sin^2 / n^2)
// on the decaying branch, tilted admittance n cos (s) or n / cos (p), phase
// delta = 2 pi n t cos / lambda, M = [[cos d, -i sin d / eta], [-i eta sin d, cos d]]),
// from air onto the glass and from the glass out to air (films reversed);
// the thick substrate (real index, tau = exp(-alpha d / cos_t)) combines the
// faces incoherently:
//   R = R_a + T_a T_g R_g tau^2 / (1 - R_g^2 tau^2),  T = T_a T_g tau / (1 - R_g^2 tau^2),
// per polarisation, averaged.
// JT > 0: that many films, known to the compiler.
template <int JT>
__device__ __forceinline__ void coated_RT_films(float c, float lam_nm, float n_sub, float alpha, float thick, int Jn,
                                                const float *nf, const float *kf, const float *tf_nm, float &R,
                                                float &T) {
    const int J = JT > 0 ? JT : Jn;
    constexpr int kN = JT > 0 ? JT : kMaxFilms;
    if (c <= 0.0f) {
        R = 1.0f;
        T = 0.0f;
        return;
    }
    c = fminf(fmaxf(c, 1e-8f), 1.0f);
    const float s2 = fmaf(-c, c, 1.0f);
    const float ct_sub = sqrtf(fmaf(-s2, __frcp_rn(n_sub * n_sub), 1.0f));
    const float tau = expf(-alpha * thick / ct_sub), t2 = tau * tau;
    Cx N[kN], CT[kN], CD[kN], SD[kN];
    for (int j = 0; j < J; ++j) {
        N[j] = cx(nf[j], kf[j]);
        const Cx n2 = N[j] * N[j];
        Cx ct = cx_sqrt(cx(1.0f) - cx_div(cx(s2), n2));
        if ((N[j] * ct).i < 0.0f) ct = (-1.0f) * ct;
        CT[j] = ct;
        const Cx delta = (6.283185307179586f * tf_nm[j] / lam_nm) * (N[j] * ct);
        float sa, ca;
        sincosf(delta.r, &sa, &ca);
        const float ep = expf(delta.i), em = expf(-delta.i);
        const float chb = 0.5f * (ep + em), shb = 0.5f * (ep - em);
        CD[j] = cx(ca * chb, -sa * shb);   // cos(a + ib)
        SD[j] = cx(sa * chb, ca * shb);    // sin(a + ib)
    }
    float Rsum = 0.0f, Tsum = 0.0f;
    for (int pol = 0; pol < 2; ++pol) {
        const float eta0 = pol == 0 ? c : __frcp_rn(c);
        const float etas = pol == 0 ? n_sub * ct_sub : n_sub / ct_sub;
        Cx m00 = cx(1.0f), m01 = cx(0.0f), m10 = cx(0.0f), m11 = cx(1.0f);   // M_1 ... M_J
        Cx g00 = cx(1.0f), g01 = cx(0.0f), g10 = cx(0.0f), g11 = cx(1.0f);   // M_J ... M_1
        for (int j = 0; j < J; ++j) {
            const Cx eta = pol == 0 ? N[j] * CT[j] : cx_div(N[j], CT[j]);
            const Cx a = CD[j];
            const Cx b = cx_div(cx(SD[j].i, -SD[j].r), eta);   // -i sin / eta
            const Cx d = eta * cx(SD[j].i, -SD[j].r);          // -i eta sin
            Cx t00 = m00 * a + m01 * d, t01 = m00 * b + m01 * a, t10 = m10 * a + m11 * d, t11 = m10 * b + m11 * a;
            m00 = t00;
            m01 = t01;
            m10 = t10;
            m11 = t11;
            t00 = a * g00 + b * g10;
            t01 = a * g01 + b * g11;
            t10 = d * g00 + a * g10;
            t11 = d * g01 + a * g11;
            g00 = t00;
            g01 = t01;
            g10 = t10;
            g11 = t11;
        }
        const Cx B = m00 + etas * m01, C = m10 + etas * m11;
        const Cx dn = eta0 * B + C, nu = eta0 * B - C;
        const float id = __frcp_rn(cx_abs2(dn));
        const float Ra = cx_abs2(nu) * id, Ta = 4.0f * eta0 * etas * id;
        const Cx B2 = g00 + eta0 * g01, C2 = g10 + eta0 * g11;
        const Cx dn2 = etas * B2 + C2, nu2 = etas * B2 - C2;
        const float id2 = __frcp_rn(cx_abs2(dn2));
        const float Rg = cx_abs2(nu2) * id2, Tg = 4.0f * etas * eta0 * id2;
        const float den = __frcp_rn(fmaf(-Rg * Rg, t2, 1.0f));
        Rsum += fmaf(Ta * Tg * Rg * t2, den, Ra);
        Tsum += Ta * Tg * tau * den;
    }
    R = 0.5f * Rsum;
    T = 0.5f * Tsum;
}
static __device__ __noinline__ void coated_RT(float c, float lam_nm, float n_sub, float alpha, float thick, int J,
                                       const float *nf, const float *kf, const float *tf_nm, float &R, float &T) {
    coated_RT_films<0>(c, lam_nm, n_sub, alpha, thick, J, nf, kf, tf_nm, R, T);
}
// A stack of J films of material m at bin i in state s, all of it in registers.
template <int J>
static __device__ __noinline__ float2 coated_few(const DevScene &sc, int m, int i, float c, float s, float alpha,
                                                 float thick) {
    float nf[J], kf[J], tf[J], R, T;
#pragma unroll
    for (int j = 0; j < J; ++j) {
        const size_t f = ((size_t)m * kMaxFilms + j) * sc.L + i;
        nf[j] = __ldg(sc.film_n + f);
        kf[j] = __ldg(sc.film_k + f) + s * __ldg(sc.film_dk + f);
        tf[j] = __ldg(sc.film_t + (size_t)m * kMaxFilms + j);
    }
    coated_RT_films<J>(c, __ldg(sc.lam + i), __ldg(sc.mat_a + (size_t)m * sc.L + i), alpha, thick, J, nf, kf, tf, R, T);
    return make_float2(R, T);
}

// R, T of glass material m at wavelength bin i: the bare absorbing slab, or
// the coated slab when the material carries films (film k = k + s dk).
// Kernels are instantiated with FILMS = false for scenes without coated glass,
// which keeps the film code (and its call) out of them entirely. DENSE: for the dense
// exact passes (k_glass_eval, k_slab_rows) over scenes whose stacks have at most
// kDenseFilms films, which keep their matrices in registers instead of indexed local
// arrays (the same bits). 2^22 rows of 1 / 2 / 3 films 140 / 197 / 257 -> 134 / 183 / 241 us;
// a call of 262,147 rows, mostly launch and wait, 40 / 45 / 49 -> 37 / 41 / 45. Deeper
// stacks have kernels of their own: sharing one with the register variants takes it
// from 48 to 80 registers, 4 / 6 / 10 films 320 / 440 / 681 us but 356 / 496 / 789.
// Three is what the electrochromic panes here have; more in registers was not tried.
template <bool FILMS = true, bool DENSE = false>
__device__ __forceinline__ void glass_rt(const DevScene &sc, int m, int i, float c, float s, float thick, float &R,
                                         float &T) {
    const size_t k = (size_t)m * sc.L + i;
    const float alpha = __ldg(sc.mat_b + k) + s * __ldg(sc.mat_c + k);
    if constexpr (!FILMS) {
        slab_RT(c, __ldg(sc.lam + i), __ldg(sc.mat_a + k), alpha, thick, R, T);
    } else {
        const int J = sc.mat_nfilm ? __ldg(sc.mat_nfilm + m) : 0;
        if (J == 0) {
            slab_RT(c, __ldg(sc.lam + i), __ldg(sc.mat_a + k), alpha, thick, R, T);
            return;
        }
        if constexpr (DENSE) {
            const float2 rt = J == 1   ? coated_few<1>(sc, m, i, c, s, alpha, thick)
                              : J == 2 ? coated_few<2>(sc, m, i, c, s, alpha, thick)
                                       : coated_few<kDenseFilms>(sc, m, i, c, s, alpha, thick);
            R = rt.x;
            T = rt.y;
        } else {
            float nf[kMaxFilms], kf[kMaxFilms], tf[kMaxFilms];
            for (int j = 0; j < J; ++j) {
                const size_t f = ((size_t)m * kMaxFilms + j) * sc.L + i;
                nf[j] = __ldg(sc.film_n + f);
                kf[j] = __ldg(sc.film_k + f) + s * __ldg(sc.film_dk + f);
                tf[j] = __ldg(sc.film_t + (size_t)m * kMaxFilms + j);
            }
            coated_RT(c, __ldg(sc.lam + i), __ldg(sc.mat_a + k), alpha, thick, J, nf, kf, tf, R, T);
        }
    }
}

// Glass branch probability: clamp(mean over bins of the lossless slab
// reflectance 2 rho / (1 + rho), averaged over polarisations, 0.05, 0.95).
// It decides an integer, so it is evaluated with explicitly rounded
// operations in a fixed order (no contraction), matching a plain float
// evaluation of the same formula.
__device__ __forceinline__ float branch_term(float c, float ni) {
    const float s2 = __fsub_rn(1.0f, __fmul_rn(c, c));
    const float x = __fsub_rn(1.0f, __fdiv_rn(s2, __fmul_rn(ni, ni)));
    float rs2, rp2;
    if (x <= 0.0f) {
        rs2 = 1.0f;
        rp2 = 1.0f;
    } else {
        const float ct = __fsqrt_rn(x);
        const float a = __fsub_rn(c, __fmul_rn(ni, ct)), b = __fadd_rn(c, __fmul_rn(ni, ct));
        const float e = __fsub_rn(__fmul_rn(ni, c), ct), f = __fadd_rn(__fmul_rn(ni, c), ct);
        const float rs = __fdiv_rn(a, b), rp = __fdiv_rn(e, f);
        rs2 = __fmul_rn(rs, rs);
        rp2 = __fmul_rn(rp, rp);
    }
    const float ps = __fdiv_rn(__fadd_rn(rs2, rs2), __fadd_rn(1.0f, rs2));
    const float pp = __fdiv_rn(__fadd_rn(rp2, rp2), __fadd_rn(1.0f, rp2));
    return __fmul_rn(0.5f, __fadd_rn(ps, pp));
}
__device__ __forceinline__ float branch_clamp(float acc, int L) {
    return fminf(fmaxf(__fdiv_rn(acc, (float)L), 0.05f), 0.95f);
}
static __device__ __noinline__ float branch_proxy(float c, int L, const float *__restrict__ n) {
    float acc = 0.0f;
    for (int i = 0; i < L; ++i) acc = __fadd_rn(acc, branch_term(c, __ldg(n + i)));
    return branch_clamp(acc, L);
}

// The same for the lanes of a warp with `want`, all 32 lanes calling: some 100
// instructions a bin ran in the one or two lanes of a warp that stood on glass
// while the others waited. Here the warp computes a lane's terms side by side and
// the lane adds them in bin order, so the value is the same bit for bit. Facade
// room (480 x 270 x 4 spp, 81 bins): continuation pass 0.92 -> 0.57 ms over its bounces.
// terms: kBranchTerms floats of shared memory of this warp.
constexpr int kBranchTerms = kMaxL;
__device__ __forceinline__ float warp_branch_proxy(bool want, float c, int L, const float *__restrict__ n, float *terms) {
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    float pr = 0.0f;
    unsigned left = __ballot_sync(full, want);
    while (left) {
        int mine = -1, k = 0;
#pragma unroll 1
        for (; left && (k + 1) * L <= kBranchTerms; ++k, left &= left - 1) {
            const int src = __ffs(left) - 1;
            if (lane == src) mine = k;
            const float cs = __shfl_sync(full, c, src);
            const float *ns = reinterpret_cast<const float *>(__shfl_sync(full, reinterpret_cast<unsigned long long>(n), src));
#pragma unroll 1
            for (int i = lane; i < L; i += 32) terms[k * L + i] = branch_term(cs, __ldg(ns + i));
        }
        __syncwarp();
        if (mine >= 0) {
            float acc = 0.0f;
#pragma unroll 4
            for (int i = 0; i < L; ++i) acc = __fadd_rn(acc, terms[mine * L + i]);
            pr = branch_clamp(acc, L);
        }
        __syncwarp();   // the next lanes' terms take their place
    }
    return pr;
}

// -------------------------------------------------------------- sampling
// Cosine-distributed direction about unit ns: Malley's method on the
// Shirley-Chiu concentric disk; tangent frame of Duff et al. (JCGT 2017).
__device__ __forceinline__ V3 cosine_dir(V3 ns, float u0, float u1) {
    float a = 2.0f * u0 - 1.0f, b = 2.0f * u1 - 1.0f;
    float dx = 0.0f, dy = 0.0f;
    if (a != 0.0f || b != 0.0f) {
        float r, phi;
        if (fabsf(a) > fabsf(b)) {
            r = a;
            phi = 0.78539816339744831f * (b / a);
        } else {
            r = b;
            phi = 1.57079632679489662f - 0.78539816339744831f * (a / b);
        }
        float sp, cp;
        sincosf(phi, &sp, &cp);
        dx = r * cp;
        dy = r * sp;
    }
    float dz = sqrtf(fmaxf(0.0f, 1.0f - dx * dx - dy * dy));
    float sgn = ns.z >= 0.0f ? 1.0f : -1.0f;
    float aa = -1.0f / (sgn + ns.z);
    float bb = ns.x * ns.y * aa;
    V3 t = v3(1.0f + sgn * ns.x * ns.x * aa, sgn * bb, -sgn * ns.x);
    V3 bt = v3(bb, sgn + ns.y * ns.y * aa, -ns.y);
    return dx * t + dy * bt + dz * ns;
}

// ----------------------------------------------------- compensated sums
struct Kahan {
    float s = 0.0f, c = 0.0f;
    __device__ __forceinline__ void add(float x) {
        float y = x - c;
        float t = s + y;
        c = (t - s) - y;
        s = t;
    }
};
struct Kahan3 {
    Kahan x, y, z;
    __device__ __forceinline__ void add(float a, float b, float c) {
        x.add(a);
        y.add(b);
        z.add(c);
    }
};
// k + (s2 - c2), the rounding error of the addition kept in k.c (true sum k.s - k.c)
// whichever term is the larger.
__device__ __forceinline__ void two_sum(Kahan &k, float s2, float c2) {
    const float t = k.s + s2, b = t - k.s;
    const float e = (k.s - (t - b)) + (s2 - b);
    k.c = (k.c + c2) - e;
    k.s = t;
}

// Four bins of a padded row.
struct Float4 {
    float v[4];
};
__device__ __forceinline__ Float4 ld4(const float4 *p) {
    const float4 x = __ldg(p);
    return Float4{{x.x, x.y, x.z, x.w}};
}
// XYZ of a chunk of four bins, with what its additions rounded off handed on, so that
// a sum over bins rounds its products and its result and nothing between. Root mean
// square error against 64 bits, 8 / 16 / 41 / 81 bins, of sums that differ in this alone:
// 4.28 / 3.62 / 3.18 / 2.70e-8 with plain sums inside the chunk and compensated ones
// between chunks, 3.08 / 2.59 / 2.18 / 2.16e-8 so (3.09 / 2.57 / 2.23 / 2.14e-8 is what
// one rounding of products and result makes). It costs 1 % of a hotel or facade room
// render, up to 3 % of a tiny room's by the DDM and 7 % by the plain method, whose time is
// mostly this.
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.0f, -1.0f), a); }
__device__ __forceinline__ Kahan weigh4(const Float4 &e, const Float4 &w) {
    // bins 0, 2 and 1, 3 side by side (two operations an instruction); what adding the
    // second pair rounds off, again with a fused product; then the two sums
    const float2 e2 = make_float2(e.v[2], e.v[3]), w2 = make_float2(w.v[2], w.v[3]);
    const float2 p = __fmul2_rn(make_float2(e.v[0], e.v[1]), make_float2(w.v[0], w.v[1]));
    const float2 t = __ffma2_rn(e2, w2, p), r = __ffma2_rn(e2, w2, sub2(p, t));
    const float s = t.x + t.y, b = s - t.x;
    Kahan k;
    k.s = s;
    k.c = -(((t.x - (s - b)) + (t.y - b)) + (r.x + r.y));
    return k;
}
// A chunk's sums of x, y, z and what x lost go to *s, what y and z lost to *c (true sums
// s - c). UNROLL 1 keeps the code short where the instruction cache bounds the kernel.
template <int UNROLL>
__device__ __forceinline__ void chunk_xyz(const Float4 &e, const float4 *w, int n_chunk, float4 *s, float2 *c) {
    float *ps = reinterpret_cast<float *>(s), *pc = ps + 3;
#pragma unroll UNROLL
    for (int k = 0; k < 3; ++k, w += n_chunk) {
        const Kahan v = weigh4(e, ld4(w));
        ps[k] = v.s;
        *pc = v.c;
        pc = reinterpret_cast<float *>(c) + k;
    }
}
// Component k of the sum of n chunks, in bin order.
template <int UNROLL>
__device__ __forceinline__ Kahan sum_chunks(const float4 *s, const float2 *c, int n, int k) {
    const float *ps = reinterpret_cast<const float *>(s) + k;
    const float *pc = k == 0 ? reinterpret_cast<const float *>(s) + 3 : reinterpret_cast<const float *>(c) + (k - 1);
    const int step = k == 0 ? 4 : 2;
    Kahan sum;
#pragma unroll UNROLL
    for (int i = 0; i < n; ++i) two_sum(sum, ps[4 * i], pc[step * i]);
    return sum;
}

// ------------------------------------------------------------------ camera
__device__ __forceinline__ void camera_ray(const RenderInfo &ri, float px, float py, V3 &o, V3 &d) {
    float nx = 2.0f * px / (float)ri.width - 1.0f;
    float ny = 1.0f - 2.0f * py / (float)ri.height;
    V3 f = v3(ri.cam_f[0], ri.cam_f[1], ri.cam_f[2]);
    V3 X = v3(ri.cam_x[0], ri.cam_x[1], ri.cam_x[2]);
    V3 Y = v3(ri.cam_y[0], ri.cam_y[1], ri.cam_y[2]);
    V3 c = v3(ri.cam_o[0], ri.cam_o[1], ri.cam_o[2]);
    if (ri.ortho) {
        o = c + nx * X + ny * Y;
        d = f;
    } else {
        o = c;
        d = normalize(f + nx * X + ny * Y);
    }
}

// Pixel and sample of a path of a render: local = pixel * spp + sample. Nearly
// every render has fewer than 2^32 paths and is divided in 32 bits.
__device__ __forceinline__ void pixel_sample(int64_t local, int spp, uint32_t &p, uint32_t &j) {
    if ((local >> 32) == 0) {
        p = (uint32_t)local / (uint32_t)spp;
        j = (uint32_t)local - p * (uint32_t)spp;
    } else {
        p = (uint32_t)(local / spp);
        j = (uint32_t)(local - (int64_t)p * spp);
    }
}

// Render of a global path index (binary search over the batch table).
__device__ __forceinline__ int find_render(const RenderBatch &rb, int64_t g) {
    int lo = 0, hi = rb.n - 1;
#pragma unroll 1
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (rb.info[mid].path_begin <= g) lo = mid; else hi = mid - 1;
    }
    return lo;
}
__device__ __forceinline__ int find_render_pixel(const RenderBatch &rb, int64_t gp) {
    int lo = 0, hi = rb.n - 1;
#pragma unroll 1
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (rb.info[mid].pixel_begin <= gp) lo = mid; else hi = mid - 1;
    }
    return lo;
}

}  // namespace sddm
