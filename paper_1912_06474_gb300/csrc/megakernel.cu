// Plain baseline: a lane per camera path over the global BVH -- the
// classical parallelisation of Sec. 5 (split the pixels, every worker sees
// the whole scene) -- computing the same estimator as the DDM path.
//
// Per path (pixel p, sample j, render r), following Sec. 4's algorithm and
// Eq. 2-3: a primary ray per pixel; at each of at most D vertices the closest
// surface; emission seen directly or through specular vertices; at Lambertian
// vertices one shadow ray toward a point on the area lights (Eq. 3's light
// sum), through glass slabs weighted by their transmittance; continuation by
// the reflection/refraction laws (cosine-distributed diffuse, Fresnel-weighted
// mirror for metals, R- or T-weighted mirror/straight branch for glass).
// Spectral values over the L bins are turned into XYZ with a compensated sum.
// With a photon map (PM) the path ends at its first diffuse vertex, after the
// emission and the next-event light there, with the photons' radiance estimate
// (Sec. 4's photon mapping for global illumination): rho / pi times the power
// of the photons within radius r that arrived on the visible side, over pi r^2.
#include <cuda_runtime.h>

#include <type_traits>

#include "device_common.cuh"
#include "photon.cuh"

namespace sddm {

// Spectral throughput storage: registers for a compile-time L, local memory otherwise.
template <int LT>
struct Spectrum {
    float v[LT > 0 ? LT : kMaxL];
};

__device__ __forceinline__ float state_of(const RenderBatch &rb, int r, int mat, int n_mat) {
    return __ldg(rb.state_s + (size_t)r * n_mat + mat);
}

// Loop over the L bins: unrolled (throughput in registers) for a small
// compile-time L, a plain loop over local memory otherwise.
template <int LT, typename F>
__device__ __forceinline__ void for_bins(int L, F &&f) {
    if constexpr (LT > 0) {
#pragma unroll
        for (int i = 0; i < LT; ++i) f(i);
    } else {
#pragma unroll 1
        for (int i = 0; i < L; ++i) f(i);
    }
}

// Add sum_i wcmf_i * f(i) to acc (compensated over i).
template <int LT, typename F>
__device__ __forceinline__ void add_xyz(const DevScene &sc, int L, Kahan3 &acc, F &&f) {
    Kahan X, Y, Z;
    for_bins<LT>(L, [&](int i) {
        float e = f(i);
        const float4 w4 = __ldg(sc.wcmf + i);
        X.add(e * w4.x);
        Y.add(e * w4.y);
        Z.add(e * w4.z);
    });
    acc.add(X.s, Y.s, Z.s);
}

// The photon-mapped camera pass: a thread per path, which ends at its first
// diffuse vertex, where it gathers the map.
template <int LT, bool FILMS>
__global__ void __launch_bounds__(128) k_megakernel_pm(MegaArgs a) {
    const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= a.path_count) return;
    const DevScene &sc = a.sc;
    const int L = LT > 0 ? LT : sc.L;
    const int64_t gp = a.path_begin + g;
    const int r = find_render(a.rb, gp);
    const RenderInfo &ri = a.rb.info[r];
    const int64_t local = gp - ri.path_begin;
    uint32_t p, j;
    pixel_sample(local, ri.spp, p, j);
    const int px = (int)(p % (uint32_t)ri.width), py = (int)(p / (uint32_t)ri.width);
    const uint32_t k0 = ri.seed, k1 = ri.render_id;

    uint4 x = philox4x32_10(make_uint4(p, j, 0u, kSlotCamera), k0, k1);
    V3 o, d;
    camera_ray(ri, (float)px + u01(x.x), (float)py + u01(x.y), o, d);

    Spectrum<LT> T;
    for_bins<LT>(L, [&](int i) {
        T.v[i] = 1.0f;
    });
    Kahan3 acc;
    int excl_prim = -1, excl_obj = -1;
    bool prev_specular = true;
    unsigned long long n_ext = 0, n_sh = 0, n_glass = 0;
    int first = -1;

    for (int b = 1; b <= ri.max_depth; ++b) {
        Ray ray = make_ray(o, d);
        ++n_ext;
        Hit h = trace_closest<false>(sc.g_nodes, sc.g_tris, sc.tri_obj, 0, ray, 0.0f, __int_as_float(0x7f800000), excl_prim,
                                    excl_obj);
        if (b == 1) first = h.prim;
        if (h.prim < 0) break;
        const float4 tn = __ldg(sc.tri_n + h.prim);
        const V3 ng = xyz(tn);
        const int mat = __float_as_int(tn.w);
        const int kind = __ldg(sc.mat_kind + mat);
        const V3 xh = o + h.t * d;
        const float cd = dot(d, ng);
        const V3 ns = cd < 0.0f ? ng : (-1.0f) * ng;
        const float *mA = sc.mat_a + (size_t)mat * L;
        const float *mB = sc.mat_b + (size_t)mat * L;

        if ((kind == kEmitter || kind == kDiffuseEmitter) && cd < 0.0f && (!ri.nee || b == 1 || prev_specular))
            add_xyz<LT>(sc, L, acc, [&](int i) { return T.v[i] * __ldg(mA + i); });
        if (kind == kEmitter) break;

        if (kind == kLambert || kind == kDiffuseEmitter) {
            const float *rho = kind == kLambert ? mA : mB;
            if (ri.nee && sc.n_light > 0) {
                uint4 xl = philox4x32_10(make_uint4(p, j, (uint32_t)b, kSlotLight), k0, k1);
                float ua = u01(xl.x), su = sqrtf(u01(xl.y)), u2 = u01(xl.z);
                int li = sc.n_light - 1;
                for (int q = 0; q < sc.n_light; ++q)
                    if (ua < __ldg(sc.light_cdf + q)) { li = q; break; }
                const float4 lv0 = __ldg(sc.light_v + 3 * li), lv1 = __ldg(sc.light_v + 3 * li + 1),
                             lv2 = __ldg(sc.light_v + 3 * li + 2);
                const float b0 = 1.0f - su, b1 = u2 * su, b2 = 1.0f - b0 - b1;
                const V3 y = b0 * xyz(lv0) + b1 * xyz(lv1) + b2 * xyz(lv2);
                const V3 xo = xh + kRayOffset * ns;
                V3 w = y - xo;
                const float dist = sqrtf(dot(w, w));
                w = (1.0f / dist) * w;
                const int lt = __float_as_int(lv0.w);
                const float4 ln = __ldg(sc.tri_n + lt);
                const float cx = dot(ns, w), cy = -dot(xyz(ln), w);
                if (cx > 0.0f && cy > 0.0f) {
                    ++n_sh;
                    Crossings cr;
                    cr.n = 0;
                    Ray sray = make_ray(xo, w);
                    bool occ = trace_shadow<false>(sc.g_nodes, sc.g_tris, sc.tri_obj, 0, sray, w, 0.0f,
                                                   (1.0f - kShadowShorten) * dist, h.prim, cr);
                    if (!occ) {
                        const float G = cx * cy / (dist * dist) * sc.light_area * (1.0f / 3.14159265358979f);
                        const float *Le = sc.mat_a + (size_t)__float_as_int(ln.w) * L;
                        float ccos[kMaxCross];
                        int cmat[kMaxCross];
                        for (int q = 0; q < cr.n; ++q) {
                            const float4 cn = __ldg(sc.tri_n + cr.tri[q]);
                            ccos[q] = -dot(w, xyz(cn));
                            cmat[q] = __float_as_int(cn.w);
                        }
                        n_glass += cr.n;
                        add_xyz<LT>(sc, L, acc, [&](int i) {
                            float tr = 1.0f;
                            for (int q = 0; q < cr.n; ++q) {
                                const int m = cmat[q];
                                float R_, T_;
                                glass_rt<FILMS>(sc, m, i, ccos[q], state_of(a.rb, r, m, sc.n_mat), __ldg(sc.mat_thick + m), R_,
                                         T_);
                                tr *= T_;
                            }
                            return T.v[i] * __ldg(rho + i) * __ldg(Le + i) * G * tr;
                        });
                    }
                }
            }
            pm_radiance_xyz(a.pm, a.pmc, xh, ns, L, rho, sc.wcmf, [&](int i) { return T.v[i]; }, acc);
            break;
        } else if (kind == kConductor) {
            if (b == ri.max_depth) break;
            const float c = fabsf(cd);
            for_bins<LT>(L, [&](int i) {
                T.v[i] *= conductor_F(c, __ldg(mA + i), __ldg(mB + i));
            });
            d = d - (2.0f * cd) * ng;
            o = xh + kRayOffset * ns;
            excl_prim = h.prim;
            excl_obj = -1;
            prev_specular = true;
        } else {  // glass slab
            if (b == ri.max_depth) break;
            const float c = fabsf(cd);
            const float pr = branch_proxy(c, L, mA);
            uint4 xg = philox4x32_10(make_uint4(p, j, (uint32_t)b, kSlotGlass), k0, k1);
            const bool reflect = u01(xg.x) < pr;
            const float s = state_of(a.rb, r, mat, sc.n_mat);
            const float th = __ldg(sc.mat_thick + mat);
            const float wsel = reflect ? 1.0f / pr : 1.0f / (1.0f - pr);
            ++n_glass;
            for_bins<LT>(L, [&](int i) {
                float R_, T_;
                glass_rt<FILMS>(sc, mat, i, c, s, th, R_, T_);
                T.v[i] *= (reflect ? R_ : T_) * wsel;
            });
            if (reflect) {
                d = d - (2.0f * cd) * ng;
                o = xh + kRayOffset * ns;
                excl_obj = -1;
            } else {
                o = xh - kRayOffset * ns;
                excl_obj = __ldg(sc.tri_obj + h.prim);
            }
            excl_prim = h.prim;
            prev_specular = true;
        }
    }
    a.sample_xyz[3 * g + 0] = acc.x.s;
    a.sample_xyz[3 * g + 1] = acc.y.s;
    a.sample_xyz[3 * g + 2] = acc.z.s;
    if (a.first_prim) a.first_prim[g] = first;
    // counters: warp-aggregated when the whole warp is here, per thread otherwise
    if (!a.counters) return;
    unsigned long long v[3] = {n_ext, n_sh, n_glass};
    if (__activemask() == 0xffffffffu) {
        for (int k = 0; k < 3; ++k)
            for (int off = 16; off > 0; off >>= 1) v[k] += __shfl_down_sync(0xffffffffu, v[k], off);
        if ((threadIdx.x & 31) != 0) return;
    }
    atomicAdd(a.counters + 0, v[0]);
    atomicAdd(a.counters + 1, v[1]);
    atomicAdd(a.counters + 2, v[2]);
}

// ---------------------------------------------------------- plain renders
// Persistent warps, a path per lane. A thread per path left most of its warp
// idle: 4.8 of 32 lanes per instruction (hotel room), since paths differ in
// length, vertex kind and traversal and each walked its own bins. Here
//  * a lane is a state machine of queries (trav_round, as in the DDM trace): an
//    extension or shadow query runs in rounds with the other lanes', and once
//    kMegaBatch lanes wait the warp stops to shade them, start their next
//    queries and give lanes without a path the next one;
//  * the spectral part of shading is done by the whole warp: each waiting lane
//    leaves a record (emission, resolved shadow ray, weight), the rows of bins
//    are dealt out to the lanes in chunks of four, as in the DDM's spectral pass,
//    with a throughput row per lane, in shared memory while there are few bins.
// Hotel room, 512 x 512 x 4 spp, 41 bins: 10.2 -> 5.9 ms; tiny room, 400 x 400 x 6
// spp, depth 6: 4.4 -> 3.7 ms; with a coated pane, 200 x 200 x 3 spp: 2.1 -> 1.04.
// The loop holds all that a path meets, some 4000 instructions, and the
// instruction cache bounds it on small scenes (2.7 of 9 stall cycles per
// instruction): not unrolling its loops took the tiny room from 4.4 to 3.5 ms,
// 32-bit path indices and one triangle test for both query kinds from 5.0 to 4.4
// (pixel_sample, trav_round), the glass branch by the whole warp from 6.8 to 5.0
// (warp_branch_proxy). Waiting lanes that stop the warp, 12 / 16 / 20 / 24 (hotel):
// 8.0 (early version) / 6.04 / 6.06 / 6.25 ms, tiny room - / 3.54 / 3.41 / 3.35;
// resident blocks 8 / 9 / 10 / 12: 6.0 / 6.3 / 5.9 / 6.4, tiny room 3.5 / 3.9 /
// 3.9 / 4.7. (These choices were measured while the sums inside a chunk were plain ones.)
struct __align__(16) MegaRec {
    float G, pcos, pw;             // shadow ray's geometry factor; |cos| and branch weight at this vertex
    int flags;                     // kMr* bits, 0 = nothing to do
    int r_le, r_rho;               // table rows: light of the shadow ray; reflectance here (its weight too)
    int r_w, r_w2;                 // table rows of a specular weight (n, k of a conductor; the glass)
    int r_emit, ncr, r, pad;       // table row of the emitter hit; slabs crossed; render
    int cmat[kMaxCross];           // their materials and cosines
    float ccos[kMaxCross];
};
constexpr int kMrEmit = 1, kMrResolve = 2, kMrDiffuse = 4, kMrConductor = 8, kMrGlass = 16, kMrFirst = 32;
#ifndef SDDM_MEGA_BATCH
#define SDDM_MEGA_BATCH 20
#endif
#ifndef SDDM_MEGA_MIN_BLOCKS
#define SDDM_MEGA_MIN_BLOCKS 8
#endif
constexpr int kMegaBatch = SDDM_MEGA_BATCH;
constexpr int kMegaMinLanes = 2;   // lanes of a warp that take paths, at least
constexpr int kMegaWarps = 2;      // warps of a block: small images spread over more SMs
constexpr int kMegaItems = 64;     // chunks worked through between two sums (a record of 256 bins)
static_assert(4 * kMegaItems >= kBranchTerms, "the two share their place");
// What a lane needs only when the warp shades: the path's sums, and the
// continuation ray while its vertex's shadow ray is under way.
struct MegaWarp {
    float acc[6][32];
    float on[3][32], dn[3][32];
    int xprim[32], xobj[32];
    MegaRec rec[32];
    float4 part[kMegaItems];   // also the glass branch's terms
    float2 lost[kMegaItems];
    int order[32];
};
// Shared memory of a warp whose throughput rows are there, too.
__host__ __device__ constexpr size_t mega_warp_bytes(int Lp) { return sizeof(MegaWarp) + sizeof(float) * 32 * (size_t)Lp; }
// Padded bins up to which the rows lie in shared memory. Above them they lie in global
// memory (a.rows): a warp's rows push eight blocks out of an SM from some 56 bins on (at
// 256 there are two), and take the L1 from the nodes and stacks before that. Rows in
// shared / global memory, hotel room 512 x 512 x 4 spp at 41 / 48 / 64 / 81 / 128 / 256 bins:
// 6.03 / 6.36 / 7.12 / 8.40 / 10.1 / 24.0 against 5.95 / 5.88 / 5.93 / 6.32 / 6.41 / 7.74 ms;
// tiny room, 400 x 400 x 4 spp: 2.23 / 2.25 / 2.48 / 3.00 / 4.03 / 17.3 against 2.24 / 2.25 /
// 2.35 / 2.75 / 3.14 / 5.93, coated, 16 bins: 0.85 against 0.89. (A thread per path with its
// row in local memory, before this kernel: 21.5 and 12.2 ms at 256 bins.)
constexpr int kMegaRowBins = 44;
size_t mega_row_bytes(int sm_count, int Lp) {
    return Lp > kMegaRowBins ? (size_t)sm_count * SDDM_MEGA_MIN_BLOCKS * kMegaWarps * 32 * Lp * sizeof(float) : 0;
}

// One chunk of a lane's record: the XYZ it adds, to *s and *c; its four throughput bins updated.
template <bool FILMS>
__device__ __forceinline__ void mega_chunk(const MegaArgs &a, const MegaRec &m, float4 *row, int ch, float4 *s, float2 *c) {
    const DevScene &sc = a.sc;
    const int n_chunk = sc.Lp >> 2, xf = m.flags;
    const float4 *const tab = reinterpret_cast<const float4 *>(sc.tab) + ch;
    Float4 t{{1.f, 1.f, 1.f, 1.f}}, e{{0.f, 0.f, 0.f, 0.f}};
    if (!(xf & kMrFirst)) {
        const float4 v = row[ch];
        t = Float4{{v.x, v.y, v.z, v.w}};
    }
    if (xf & kMrEmit) {
        const Float4 le = ld4(tab + m.r_emit * n_chunk);
#pragma unroll
        for (int u = 0; u < 4; ++u) e.v[u] = t.v[u] * le.v[u];
    }
    if (xf & (kMrResolve | kMrDiffuse)) {
        const Float4 rho = ld4(tab + m.r_rho * n_chunk);
        if (xf & kMrResolve) {
            const Float4 le = ld4(tab + m.r_le * n_chunk);
            Float4 tr{{1.f, 1.f, 1.f, 1.f}};
#pragma unroll 1
            for (int k = 0; k < m.ncr; ++k) {
                const int cm = m.cmat[k];
                const float st = __ldg(a.rb.state_s + (size_t)m.r * sc.n_mat + cm), th = __ldg(sc.mat_thick + cm);
#pragma unroll 1
                for (int u = 0; u < 4; ++u) {
                    float R_, T_;
                    glass_rt<FILMS>(sc, cm, min(4 * ch + u, sc.L - 1), m.ccos[k], st, th, R_, T_);
#pragma unroll
                    for (int x = 0; x < 4; ++x) tr.v[x] *= x == u ? T_ : 1.0f;
                }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) e.v[u] += t.v[u] * rho.v[u] * le.v[u] * m.G * tr.v[u];
        }
        if (xf & kMrDiffuse) {
#pragma unroll
            for (int u = 0; u < 4; ++u) t.v[u] *= rho.v[u];
        }
    }
    if (xf & kMrConductor) {
        const Float4 n = ld4(tab + m.r_w * n_chunk), k = ld4(tab + m.r_w2 * n_chunk);
#pragma unroll
        for (int u = 0; u < 4; ++u) t.v[u] *= conductor_F(m.pcos, n.v[u], k.v[u]);
    } else if (xf & kMrGlass) {
        const float st = __ldg(a.rb.state_s + (size_t)m.r * sc.n_mat + m.r_w), th = __ldg(sc.mat_thick + m.r_w);
        const bool refl = m.pw < 0.0f;
#pragma unroll 1
        for (int u = 0; u < 4; ++u) {
            float R_, T_;
            glass_rt<FILMS>(sc, m.r_w, min(4 * ch + u, sc.L - 1), m.pcos, st, th, R_, T_);
            const float w = (refl ? R_ : T_) * fabsf(m.pw);
#pragma unroll
            for (int x = 0; x < 4; ++x) t.v[x] *= x == u ? w : 1.0f;
        }
    }
    if (xf & (kMrDiffuse | kMrConductor | kMrGlass)) row[ch] = make_float4(t.v[0], t.v[1], t.v[2], t.v[3]);
    if (xf & (kMrEmit | kMrResolve)) {
        chunk_xyz<1>(e, tab + 2 * sc.n_mat * n_chunk, n_chunk, s, c);
    }
}

template <bool COUNT, bool FILMS, bool ROWS>
__global__ void __launch_bounds__(32 * kMegaWarps, SDDM_MEGA_MIN_BLOCKS) k_megakernel(const __grid_constant__ MegaArgs a,
                                                                                           int lanes, int batch) {
    extern __shared__ __align__(16) unsigned char s_mega[];
    const DevScene &sc = a.sc;
    const int L = sc.L, Lp = sc.Lp, n_chunk = Lp >> 2, M = sc.n_mat;
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const unsigned lt_mask = (1u << lane) - 1u;
    const int warp = threadIdx.x >> 5;
    unsigned char *const mem = s_mega + (ROWS ? sizeof(MegaWarp) : mega_warp_bytes(Lp)) * warp;
    float4 *const rows = ROWS ? a.rows + ((size_t)blockIdx.x * kMegaWarps + warp) * 32 * n_chunk : reinterpret_cast<float4 *>(mem);
    MegaWarp &w = *reinterpret_cast<MegaWarp *>(ROWS ? mem : mem + sizeof(float) * 32 * (size_t)Lp);
    const int per_pass = min(32, kMegaItems / n_chunk);           // records summed at a time (n_chunk <= 64)
    const unsigned inv_chunk = 65536u / (unsigned)n_chunk + 1u;   // i / n_chunk = i inv >> 16 for i < kMegaItems

    enum { kIdle, kExt, kShadow };
    int mode = kIdle, b = 0;
    int64_t g = 0;                // the lane's path
    bool dry = lane >= lanes;     // no path left for this lane
    bool prev_specular = true, t_set = false;   // t_set: the lane's row holds the throughput (1 until a weight)
    V3 rd = v3(0.f, 0.f, 0.f);    // direction of the query under way
    V3 ro = rd;
    LaneTrav t;
    t.tmin = t.tw = 0.f;
    t.node = t.sp = 0;
    t.best = t.ep = t.eo = -1;
    t.occ = t.fin = false;
    Crossings cr;
    cr.n = 0;
    int stack[kStackSize];
    unsigned n_ext = 0, n_sh = 0, n_glass = 0;
    TravCount tc;

    for (;;) {
        const unsigned m_wait = __ballot_sync(full, t.fin || (mode == kIdle && !dry));
        const unsigned m_busy = __ballot_sync(full, mode != kIdle && !t.fin);
        if (m_busy == 0 || __popc(m_wait) >= batch) {
            if (m_wait == 0) break;
            int next_mode = kIdle;        // the lane's next query, where it has one
            V3 no = ro, nd = rd;
            float n_tmax = 3.402823466e38f;   // below +inf: a missed triangle's distance is no hit
            int n_ep = -1, n_eo = -1;
            bool ended = false;
            int flags = 0;
            float u_glass = 0.0f;
            V3 thru = ro;
            MegaRec &me = w.rec[lane];
            if (t.fin && mode == kShadow) {
                flags = me.flags;         // the diffuse weight, where the path goes on
                if (!t.occ) {
                    flags |= kMrResolve;
                    me.ncr = cr.n;
#pragma unroll 1
                    for (int k = 0; k < cr.n; ++k) {
                        const float4 cn = __ldg(sc.tri_n + cr.tri[k]);
                        me.ccos[k] = -dot(rd, xyz(cn));
                        me.cmat[k] = __float_as_int(cn.w);
                    }
                    n_glass += cr.n;
                }
                if (flags & kMrDiffuse) {
                    next_mode = kExt;
                    no = v3(w.on[0][lane], w.on[1][lane], w.on[2][lane]);
                    nd = v3(w.dn[0][lane], w.dn[1][lane], w.dn[2][lane]);
                    n_ep = w.xprim[lane];
                    n_eo = -1;
                } else {
                    ended = true;
                }
            } else if (t.fin) {
                const int prim = t.best;
                if (b == 1 && a.first_prim) a.first_prim[g] = prim;
                if (prim < 0) {
                    ended = true;
                } else {
                    const int64_t gp = a.path_begin + g;
                    const int r = find_render(a.rb, gp);
                    const RenderInfo &ri = a.rb.info[r];
                    const int64_t local = gp - ri.path_begin;
                    uint32_t p, j;
                    pixel_sample(local, ri.spp, p, j);
                    const uint32_t k0 = ri.seed, k1 = ri.render_id;
                    const float4 tn = __ldg(sc.tri_n + prim);
                    const V3 ng = xyz(tn);
                    const int mat = __float_as_int(tn.w);
                    const int kind = __ldg(sc.mat_kind + mat);
                    const V3 xh = ro + t.tw * rd;
                    const float cd = dot(rd, ng);
                    const V3 ns = cd < 0.0f ? ng : (-1.0f) * ng;
                    const bool last = b == ri.max_depth;
                    me.r = r;
                    if ((kind == kEmitter || kind == kDiffuseEmitter) && cd < 0.0f &&
                        (!ri.nee || b == 1 || prev_specular)) {
                        flags |= kMrEmit;
                        me.r_emit = mat;
                    }
                    if (kind == kLambert || kind == kDiffuseEmitter) {
                        me.r_rho = kind == kLambert ? mat : M + mat;
                        if (!last) {
                            uint4 xb = philox4x32_10(make_uint4(p, j, (uint32_t)b, kSlotBsdf), k0, k1);
                            nd = cosine_dir(ns, u01(xb.x), u01(xb.y));
                            no = xh + kRayOffset * ns;
                            n_ep = prim;
                            next_mode = kExt;
                        }
                        bool shadow = false;
                        if (ri.nee && sc.n_light > 0) {
                            uint4 xl = philox4x32_10(make_uint4(p, j, (uint32_t)b, kSlotLight), k0, k1);
                            float ua = u01(xl.x), su = sqrtf(u01(xl.y)), u2 = u01(xl.z);
                            int li = sc.n_light - 1;
#pragma unroll 1
                            for (int q = 0; q < sc.n_light; ++q)
                                if (ua < __ldg(sc.light_cdf + q)) { li = q; break; }
                            const float4 lv0 = __ldg(sc.light_v + 3 * li), lv1 = __ldg(sc.light_v + 3 * li + 1),
                                         lv2 = __ldg(sc.light_v + 3 * li + 2);
                            const float b0 = 1.0f - su, b1 = u2 * su, b2 = 1.0f - b0 - b1;
                            const V3 y = b0 * xyz(lv0) + b1 * xyz(lv1) + b2 * xyz(lv2);
                            const V3 xo = xh + kRayOffset * ns;
                            V3 wl = y - xo;
                            const float dist = sqrtf(dot(wl, wl));
                            wl = (1.0f / dist) * wl;
                            const int lt = __float_as_int(lv0.w);
                            const float4 ln = __ldg(sc.tri_n + lt);
                            const float cx = dot(ns, wl), cy = -dot(xyz(ln), wl);
                            if (cx > 0.0f && cy > 0.0f) {
                                ++n_sh;
                                shadow = true;
                                me.G = cx * cy / (dist * dist) * sc.light_area * (1.0f / 3.14159265358979f);
                                me.r_le = __float_as_int(ln.w);
                                w.on[0][lane] = no.x;
                                w.on[1][lane] = no.y;
                                w.on[2][lane] = no.z;
                                w.dn[0][lane] = nd.x;
                                w.dn[1][lane] = nd.y;
                                w.dn[2][lane] = nd.z;
                                w.xprim[lane] = prim;
                                no = xo;
                                nd = wl;
                                n_tmax = (1.0f - kShadowShorten) * dist;
                                n_ep = prim;
                            }
                        }
                        prev_specular = false;
                        if (shadow) {
                            me.flags = last ? 0 : kMrDiffuse;   // taken up when the shadow ray is answered
                            next_mode = kShadow;
                        } else if (last) {
                            ended = true;
                        } else {
                            flags |= kMrDiffuse;
                        }
                    } else if (kind == kEmitter || last) {
                        ended = true;
                    } else {
                        const float c = fabsf(cd);
                        me.pcos = c;
                        me.r_w = mat;
                        me.r_w2 = M + mat;
                        nd = rd - (2.0f * cd) * ng;
                        no = xh + kRayOffset * ns;
                        n_ep = prim;
                        if (kind == kConductor) {
                            flags |= kMrConductor;
                        } else {
                            flags |= kMrGlass;
                            ++n_glass;
                            n_eo = __ldg(sc.tri_obj + prim);   // for the branch that transmits
                            const uint4 xg = philox4x32_10(make_uint4(p, j, (uint32_t)b, kSlotGlass), k0, k1);
                            u_glass = u01(xg.x);
                            thru = xh - kRayOffset * ns;
                        }
                        next_mode = kExt;
                        prev_specular = true;
                    }
                }
            }
            if (__any_sync(full, flags & kMrGlass)) {
                const float pr = warp_branch_proxy((flags & kMrGlass) != 0, me.pcos, L,
                                                   sc.mat_a + (size_t)((flags & kMrGlass) ? me.r_w : 0) * L,
                                                   reinterpret_cast<float *>(w.part));
                if (flags & kMrGlass) {
                    if (u_glass < pr) {
                        me.pw = -1.0f / pr;
                        n_eo = -1;
                    } else {
                        me.pw = 1.0f / (1.0f - pr);
                        nd = rd;
                        no = thru;
                    }
                }
            }
            // the warp works through the records' bins
            if (flags && !t_set) flags |= kMrFirst;
            const int held = me.flags;     // a shadow ray now under way keeps its flags
            const unsigned work = __ballot_sync(full, flags != 0);
            const int n_rec = __popc(work), mine = __popc(work & lt_mask);
            if (flags) {
                me.flags = flags;
                w.order[mine] = lane;
            }
            __syncwarp();
#pragma unroll 1
            for (int r0 = 0; r0 < n_rec; r0 += per_pass) {
                const int nr = min(per_pass, n_rec - r0), n_item = nr * n_chunk;
#pragma unroll 1
                for (int i = lane; i < n_item; i += 32) {
                    const int jr = (int)((unsigned)i * inv_chunk >> 16), from = w.order[r0 + jr];
                    mega_chunk<FILMS>(a, w.rec[from], rows + from * n_chunk, i - jr * n_chunk, w.part + i, w.lost + i);
                }
                __syncwarp();
#pragma unroll 1
                for (int i = lane; i < 3 * nr; i += 32) {
                    const int jr = i / 3, k = i - 3 * jr, from = w.order[r0 + jr];
                    if (!(w.rec[from].flags & (kMrEmit | kMrResolve))) continue;
                    const Kahan sum = sum_chunks<1>(w.part + jr * n_chunk, w.lost + jr * n_chunk, n_chunk, k);
                    Kahan to;
                    to.s = w.acc[k][from];
                    to.c = w.acc[3 + k][from] + sum.c;   // what the chunk sums lost goes on to the path's sum
                    to.add(sum.s);
                    w.acc[k][from] = to.s;
                    w.acc[3 + k][from] = to.c;
                }
                __syncwarp();
            }
            if (flags & (kMrDiffuse | kMrConductor | kMrGlass)) t_set = true;
            if (next_mode == kShadow) me.flags = held;
            if (ended) {
                a.sample_xyz[3 * g + 0] = w.acc[0][lane];
                a.sample_xyz[3 * g + 1] = w.acc[1][lane];
                a.sample_xyz[3 * g + 2] = w.acc[2][lane];
                mode = kIdle;
                t.fin = false;
            }
            // lanes without a path take the next ones
            const bool need = mode == kIdle && !dry;
            const unsigned m = __ballot_sync(full, need);
            if (m) {
                unsigned long long c0 = 0;
                if (lane == 0) c0 = atomicAdd(a.cursor, (unsigned long long)__popc(m));
                c0 = __shfl_sync(full, c0, 0);
                if (need) {
                    g = (int64_t)(c0 + (unsigned long long)__popc(m & lt_mask));
                    dry = g >= a.path_count;
                    if (!dry) {
                        const int64_t gp = a.path_begin + g;
                        const RenderInfo &ri = a.rb.info[find_render(a.rb, gp)];
                        const int64_t local = gp - ri.path_begin;
                        uint32_t p, j;
                        pixel_sample(local, ri.spp, p, j);
                        const int px = (int)(p % (uint32_t)ri.width), py = (int)(p / (uint32_t)ri.width);
                        uint4 x = philox4x32_10(make_uint4(p, j, 0u, kSlotCamera), ri.seed, ri.render_id);
                        camera_ray(ri, (float)px + u01(x.x), (float)py + u01(x.y), no, nd);
                        next_mode = kExt;
                        n_ep = n_eo = -1;
                        n_tmax = 3.402823466e38f;
                        b = 0;
                        prev_specular = true;
                        t_set = false;
                        mode = kExt;
#pragma unroll
                        for (int k = 0; k < 6; ++k) w.acc[k][lane] = 0.0f;
                    }
                }
            }
            if (next_mode != kIdle) {
                if (next_mode == kExt) {
                    ++b;
                    ++n_ext;
                }
                mode = next_mode;
                ro = no;
                rd = nd;
                t.ray = make_ray(ro, rd);
                t.tmin = 0.0f;
                t.tw = n_tmax;
                t.node = t.sp = 0;
                t.best = -1;
                t.ep = n_ep;
                t.eo = n_eo;
                t.occ = t.fin = false;
                cr.n = 0;
            }
        }
        trav_round<COUNT, false, 64, 6>(sc.g_nodes, sc.g_tris, sc.tri_obj, t, cr, stack, mode != kIdle && !t.fin,
                                        mode == kShadow, [&]() { return rd; }, tc, a.error_flag, 0, 0);
    }
    if (!a.counters) return;
    unsigned long long v[6] = {n_ext, n_sh, n_glass, tc.nodes, tc.tris, (unsigned long long)n_ext + n_sh};
    const int nv = COUNT ? 6 : 3;
    for (int k = 0; k < nv; ++k)
        for (int off = 16; off > 0; off >>= 1) v[k] += __shfl_down_sync(full, v[k], off);
    if (lane != 0) return;
    atomicAdd(a.counters + 0, v[0]);
    atomicAdd(a.counters + 1, v[1]);
    atomicAdd(a.counters + 2, v[2]);
    if (COUNT) {
        atomicAdd(a.counters + 5, v[3]);
        atomicAdd(a.counters + 6, v[4]);
        atomicAdd(a.counters + 7, v[5]);
    }
}

template <bool FILMS>
static void launch_pm(const MegaArgs &a, cudaStream_t stream) {
    const unsigned nb = (unsigned)((a.path_count + 127) / 128);
    switch (a.sc.L) {
        case 8: k_megakernel_pm<8, FILMS><<<nb, 128, 0, stream>>>(a); break;
        case 16: k_megakernel_pm<16, FILMS><<<nb, 128, 0, stream>>>(a); break;
        default: k_megakernel_pm<0, FILMS><<<nb, 128, 0, stream>>>(a); break;
    }
}

template <bool COUNT, bool FILMS, bool ROWS>
static cudaError_t launch_plain(const MegaArgs &a, cudaStream_t stream) {
    const size_t smem = (ROWS ? sizeof(MegaWarp) : mega_warp_bytes(a.sc.Lp)) * kMegaWarps;
    cudaError_t e = cudaSuccess;
    if (smem > 48 * 1024)   // more than a block has without asking (over 104 bins); the same for every caller
        e = cudaFuncSetAttribute(k_megakernel<COUNT, FILMS, ROWS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)(mega_warp_bytes(kMaxL) * kMegaWarps));
    if (e == cudaSuccess) e = cudaMemsetAsync(a.cursor, 0, sizeof(unsigned long long), stream);
    if (e != cudaSuccess) return e;
    // One wave of resident blocks. An image with fewer paths than lanes there are
    // spreads over more warps of fewer lanes: a warp's rounds last as long as its
    // longest lane's, so narrow warps answer sooner (at least 32 / 8 / 4 / 2 lanes:
    // tiny room 64 x 64 x 1 spp 70 / 56 / 50 / 49 us, hotel room 654 / 465 / 386 /
    // 330 us, 128 x 128 x 2 spp 759 / 677 / 683 / 692 us).
    constexpr int kWarpsPerSm = kMegaWarps * SDDM_MEGA_MIN_BLOCKS;
    const int64_t warps = (int64_t)a.sm_count * kWarpsPerSm, per_warp = (a.path_count + warps - 1) / warps;
    const int lanes = (int)(per_warp < kMegaMinLanes ? kMegaMinLanes : per_warp < 32 ? per_warp : 32);
    const int batch = lanes * kMegaBatch / 32 > 1 ? lanes * kMegaBatch / 32 : 1;
    const int64_t want = (a.path_count + lanes * kMegaWarps - 1) / (lanes * kMegaWarps);
    int64_t most = want;
    if (lanes == 32) {
        int per_sm = 1;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_megakernel<COUNT, FILMS, ROWS>, 32 * kMegaWarps, smem);
        if (e != cudaSuccess) return e;
        if (ROWS && per_sm > SDDM_MEGA_MIN_BLOCKS) per_sm = SDDM_MEGA_MIN_BLOCKS;   // as many rows as there are
        most = (int64_t)a.sm_count * (per_sm > 0 ? per_sm : 1);
    }
    k_megakernel<COUNT, FILMS, ROWS><<<(unsigned)(want < most ? want : most), 32 * kMegaWarps, smem, stream>>>(a, lanes, batch);
    return cudaGetLastError();
}

cudaError_t launch_megakernel(const MegaArgs &a, cudaStream_t stream) {
    if (a.path_count <= 0) return cudaSuccess;
    const bool films = a.sc.mat_nfilm != nullptr;
    if (a.pm.on) {
        films ? launch_pm<true>(a, stream) : launch_pm<false>(a, stream);
        return cudaGetLastError();
    }
    const bool rows = a.rows && a.sc.Lp > kMegaRowBins;
    auto launch = [&](auto count) {
        constexpr bool C = decltype(count)::value;
        if (rows) return films ? launch_plain<C, true, true>(a, stream) : launch_plain<C, false, true>(a, stream);
        return films ? launch_plain<C, true, false>(a, stream) : launch_plain<C, false, false>(a, stream);
    };
    return a.count_traversal ? launch(std::true_type()) : launch(std::false_type());
}

}  // namespace sddm
