// Photon mapping through the domain decomposition (Sec. 4 photon mapping,
// Sec. 5 sub-domains). Included by ddm.cu: it reuses the ray queues, the
// scatter and the trace kernel unchanged.
//
// Photon pass: k_photon_emit starts photon i at a point of the area lights
// (triangle by area, uniform point, cosine direction about the front face,
// power pi Le A / N) and stages its ray in the queue of the subdomain where it
// enters the grid; every hit b = 1 .. D-1 runs the subdomain waves, then
// k_photon_shade stores the photon at a diffuse hit once a bounce or a
// reflection has changed its direction and continues it like a camera path
// (diffuse bounce times rho, conductor mirror times Fresnel, glass branch with
// R/P, T/(1-P)). The photon's power lives in the path state's throughput rows.
// Philox counter (photon, 0xffffffff, hit, slot), key (seed, render id).
//
// Camera pass: k_ddm_gather adds, at a path's diffuse vertex, the power of
// the photons within radius r on the visible side times rho / pi / (pi r^2);
// k_shade_continue then issues the shadow ray but no continuation.

constexpr int kFlPhotonTurned = 16;   // the photon's direction has changed (bounce or reflection)
constexpr int kFlPhotonDiffuse = 32;  // ... by a diffuse bounce (else it is a caustic photon)

struct PhotonPass {
    int64_t begin, n_total;
    int max_depth;
    uint32_t seed, render_id;
    float scale;                // pi * total light area / n_total
    const float *state_s;
    float4 *pos, *dir;
    float *pow;
};

__global__ void __launch_bounds__(256) k_photon_emit(KArgs a, PhotonPass pp) {
    const int64_t np = a.ps.np;
    const DevScene &sc = a.sc;
    const int L = sc.L;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    unsigned long long n_ext = 0;
    __shared__ PushSmem psm;
    int *bins = block_bins_init(a.g.n_bins);
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < np; base += stride) {   // block-uniform trips
        const int64_t q = base + threadIdx.x;
        bool want = false;
        int cell = 0;
        float4 r0 = make_float4(0, 0, 0, 0), r1 = r0;
        int4 r2 = make_int4(0, 0, 0, 0);
        if (q < np) {
            a.ps.flags[q] = 0;
            if (sc.n_light > 0) {
                const uint32_t pi = (uint32_t)(pp.begin + q), pj = 0xffffffffu;
                uint4 xl = philox4x32_10(make_uint4(pi, pj, 0u, kSlotLight), pp.seed, pp.render_id);
                const float ua = u01(xl.x), su = sqrtf(u01(xl.y)), u2 = u01(xl.z);
                int li = sc.n_light - 1;
                for (int k = 0; k < sc.n_light; ++k)
                    if (ua < __ldg(sc.light_cdf + k)) { li = k; break; }
                const float4 lv0 = __ldg(sc.light_v + 3 * li), lv1 = __ldg(sc.light_v + 3 * li + 1),
                             lv2 = __ldg(sc.light_v + 3 * li + 2);
                const int lt = __float_as_int(lv0.w);
                const float4 ln = __ldg(sc.tri_n + lt);
                const V3 nl = xyz(ln);
                const float b0 = 1.0f - su, b1 = u2 * su, b2 = 1.0f - b0 - b1;
                const V3 o = b0 * xyz(lv0) + b1 * xyz(lv1) + b2 * xyz(lv2) + kRayOffset * nl;
                uint4 xd = philox4x32_10(make_uint4(pi, pj, 0u, kSlotBsdf), pp.seed, pp.render_id);
                const V3 d = cosine_dir(nl, u01(xd.x), u01(xd.y));
                const float *Le = sc.mat_a + (size_t)__float_as_int(ln.w) * L;
                for (int i = 0; i < L; ++i) a.ps.T[(size_t)i * np + q] = __ldg(Le + i) * pp.scale;
                a.ps.flags[q] = kFlExt;
                a.ps.hit0[q] = make_float4(0.f, 0.f, 0.f, __int_as_float(-1));
                ++n_ext;
                float t0;
                if (grid_enter(a.g, o, d, __int_as_float(0x7f800000), t0, cell)) {
                    want = true;
                    r0 = make_float4(o.x, o.y, o.z, t0);
                    r1 = make_float4(d.x, d.y, d.z, __int_as_float(0x7f800000));
                    r2 = make_int4((int)q, lt, 0, cell);
                }
            }
        }
        block_stage_push2(a.Q, a.g, psm, bins, want, cell, r0, r1, r2, false, 0, r0, r1, r2, a.err);
    }
    block_bins_flush(a.Q, bins, a.g.n_bins);
    block_count3(a.counters + 0, n_ext, nullptr, 0, nullptr, 0);
}

// Power rows of the photons a warp stores are written row by row by the whole
// warp (coalesced) through a [L][33] shared-memory tile per warp, for L up to
// kStageMaxL; one lane per row otherwise.
constexpr int kStageMaxL = 64;
__host__ __device__ constexpr size_t photon_stage_bytes(int L) {
    return L <= kStageMaxL ? (size_t)8 * L * 33 * sizeof(float) : 0;
}

template <bool FILMS>
__global__ void __launch_bounds__(256) k_photon_shade(KArgs a, PhotonPass pp) {
    const int64_t np = a.ps.np;
    const DevScene &sc = a.sc;
    const int L = sc.L, b = a.b, D = pp.max_depth;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    unsigned long long n_ext = 0;
    __shared__ PushSmem psm;
    int *bins = block_bins_init(a.g.n_bins);
    __shared__ float s_terms[8][kBranchTerms];
    const bool staged = L <= kStageMaxL;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    float *stage = reinterpret_cast<float *>(bins + ((a.g.n_bins + 3) & ~3)) + (size_t)w * L * 33;
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < np; base += stride) {   // block-uniform trips
        const int64_t q = base + threadIdx.x;
        bool want = false;
        int cell = 0;
        float4 e0 = make_float4(0, 0, 0, 0), e1 = e0;
        int4 e2 = make_int4(0, 0, 0, 0);
        const int fl = q < np ? a.ps.flags[q] : 0;
        if (staged) {
            bool store = false;
            if ((fl & kFlExt) && (fl & kFlPhotonTurned)) {
                const int prim = __float_as_int(a.ps.hit0[q].w);
                if (prim >= 0) {
                    const int kind = __ldg(sc.mat_kind + __float_as_int(__ldg(sc.tri_n + prim).w));
                    store = kind == kLambert || kind == kDiffuseEmitter;
                }
            }
            const unsigned sm = __ballot_sync(0xffffffffu, store);
            if (sm) {
                if (store)
                    for (int i = 0; i < L; ++i) stage[i * 33 + lane] = a.ps.T[(size_t)i * np + q];
                __syncwarp();
                for (unsigned m = sm; m; m &= m - 1) {
                    const int src = __ffs(m) - 1;
                    const size_t slot = (size_t)(pp.begin + base + 32 * w + src) * (D - 1) + (b - 1);
                    for (int i = lane; i < L; i += 32) pp.pow[slot * L + i] = stage[i * 33 + src];
                }
                __syncwarp();
            }
        }
        // the glass branch of the warp's photons that stand on glass
        float pr = 0.f;
        {
            bool glass = false;
            float c = 0.f;
            int mat = 0;
            if ((fl & kFlExt) && b < D - 1) {
                const int prim = __float_as_int(a.ps.hit0[q].w);
                if (prim >= 0) {
                    const float4 tn = __ldg(sc.tri_n + prim);
                    mat = __float_as_int(tn.w);
                    glass = __ldg(sc.mat_kind + mat) == kGlass;
                    if (glass) c = fabsf(dot(xyz(a.ps.hit1[q]), xyz(tn)));
                }
            }
            pr = warp_branch_proxy(glass, c, L, sc.mat_a + (size_t)mat * L, s_terms[w]);
        }
        if (fl & kFlExt) {
            int nfl = 0;
            const float4 h0 = a.ps.hit0[q], h1 = a.ps.hit1[q];
            const int prim = __float_as_int(h0.w);
            if (prim >= 0) {
                const uint32_t pi = (uint32_t)(pp.begin + q), pj = 0xffffffffu;
                const float4 tn = __ldg(sc.tri_n + prim);
                const V3 ng = xyz(tn), x = xyz(h0), d = xyz(h1);
                const int mat = __float_as_int(tn.w), kind = __ldg(sc.mat_kind + mat);
                const float cd = dot(d, ng);
                const V3 ns = cd < 0.0f ? ng : (-1.0f) * ng;
                const float *mA = sc.mat_a + (size_t)mat * L, *mB = sc.mat_b + (size_t)mat * L;
                bool go = false, turn = true, diffuse = false;   // a transmitted photon keeps its direction
                V3 on = x, dn = d;
                int excl = prim;
                if (kind == kLambert || kind == kDiffuseEmitter) {
                    if (fl & kFlPhotonTurned) {
                        const size_t slot = (size_t)(pp.begin + q) * (D - 1) + (b - 1);
                        // w: 1 global photon, 2 caustic photon (only reflections turned it)
                        pp.pos[slot] = make_float4(x.x, x.y, x.z, (fl & kFlPhotonDiffuse) ? 1.0f : 2.0f);
                        pp.dir[slot] = make_float4(d.x, d.y, d.z, 0.0f);
                        if (!staged) {
                            float *pw = pp.pow + slot * L;
                            for (int i = 0; i < L; ++i) pw[i] = a.ps.T[(size_t)i * np + q];
                        }
                    }
                    if (b < D - 1) {
                        const float *rho = kind == kLambert ? mA : mB;
                        uint4 xb = philox4x32_10(make_uint4(pi, pj, (uint32_t)b, kSlotBsdf), pp.seed, pp.render_id);
                        dn = cosine_dir(ns, u01(xb.x), u01(xb.y));
                        for (int i = 0; i < L; ++i) a.ps.T[(size_t)i * np + q] *= __ldg(rho + i);
                        on = x + kRayOffset * ns;
                        go = true;
                        diffuse = true;
                    }
                } else if (kind == kConductor) {
                    if (b < D - 1) {
                        const float c = fabsf(cd);
                        for (int i = 0; i < L; ++i)
                            a.ps.T[(size_t)i * np + q] *= conductor_F(c, __ldg(mA + i), __ldg(mB + i));
                        dn = d - (2.0f * cd) * ng;
                        on = x + kRayOffset * ns;
                        go = true;
                    }
                } else if (kind == kGlass) {
                    if (b < D - 1) {
                        const float c = fabsf(cd);
                        uint4 xg = philox4x32_10(make_uint4(pi, pj, (uint32_t)b, kSlotGlass), pp.seed, pp.render_id);
                        const bool refl = u01(xg.x) < pr;
                        const float st = __ldg(pp.state_s + mat), th = __ldg(sc.mat_thick + mat);
                        const float wsel = refl ? 1.0f / pr : 1.0f / (1.0f - pr);
                        for (int i = 0; i < L; ++i) {
                            float R_, T_;
                            glass_rt<FILMS>(sc, mat, i, c, st, th, R_, T_);
                            a.ps.T[(size_t)i * np + q] *= (refl ? R_ : T_) * wsel;
                        }
                        if (refl) {
                            dn = d - (2.0f * cd) * ng;
                            on = x + kRayOffset * ns;
                        } else {
                            on = x - kRayOffset * ns;
                            excl = -__ldg(sc.tri_obj + prim) - 2;
                            turn = false;
                        }
                        go = true;
                    }
                }
                if (go) {
                    nfl = kFlExt | ((turn || (fl & kFlPhotonTurned)) ? kFlPhotonTurned : 0) |
                          ((diffuse || (fl & kFlPhotonDiffuse)) ? kFlPhotonDiffuse : 0);
                    ++n_ext;
                    a.ps.hit0[q] = make_float4(0.f, 0.f, 0.f, __int_as_float(-1));
                    float t0;
                    if (grid_enter(a.g, on, dn, __int_as_float(0x7f800000), t0, cell)) {
                        want = true;
                        e0 = make_float4(on.x, on.y, on.z, t0);
                        e1 = make_float4(dn.x, dn.y, dn.z, __int_as_float(0x7f800000));
                        e2 = make_int4((int)q, excl, 0, cell);
                    }
                }
            }
            a.ps.flags[q] = nfl;
        }
        block_stage_push2(a.Q, a.g, psm, bins, want, cell, e0, e1, e2, false, 0, e0, e1, e2, a.err);
    }
    block_bins_flush(a.Q, bins, a.g.n_bins);
    block_count3(a.counters + 0, n_ext, nullptr, 0, nullptr, 0);
}

// Photon-map radiance at the diffuse vertex of each path of this bounce, in two
// passes: k_gather_list finds the paths that gather and how many photons lie in
// the cells they look at, and sorts them into a light and a heavy list;
// k_ddm_gather works them off dynamically, the heavy ones first with all warps of
// a block on one path, then the light ones with a warp each (pm_warp_gather, a
// lane holding the bins lane + 32 k). The bound is the photons' power rows through
// L1 and L2 (4 L bytes per photon within the radius), and before that the longest
// gather: next to a light thousands of photons lie within the radius, and their
// paths sit side by side. Hotel room, 256 x 256 x 4 spp, 2^18 photons, 41 bins, six
// bounces: a thread per path 4.5 ms (11 % of the warps active on average), a warp
// per 32 slots 3.3 ms, these two passes 0.97 ms.
constexpr int kGatherHeavy = 512;   // candidates from which a block takes the path
struct GatherLists {
    int *light, *heavy;             // [np] path slots
    unsigned *cnt;                  // [4] light, heavy; next light, next heavy to work off (zero before the passes)
};
__global__ void __launch_bounds__(256) k_gather_list(const __grid_constant__ KArgs a, GatherLists gl) {
    const int64_t np = a.ps.np, q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const DevScene &sc = a.sc;
    const PathState &ps = a.ps;
    int n = -1;
    if (q < np && (ps.flags[q] & kFlExt) && a.b <= a.rb.info[find_render(a.rb, a.path_begin + q)].max_depth) {
        const float4 h0 = ps.hit0[q];
        const int prim = __float_as_int(h0.w);
        if (prim >= 0) {
            const int kind = __ldg(sc.mat_kind + __float_as_int(__ldg(sc.tri_n + prim).w));
            if (kind == kLambert || kind == kDiffuseEmitter) {
                n = pm_candidates(a.pm, xyz(h0));
                if (a.pmc.on) n += pm_candidates(a.pmc, xyz(h0));
            }
        }
    }
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        const bool mine = e == 0 ? n > 0 && n < kGatherHeavy : n >= kGatherHeavy;   // no candidates: nothing to add
        const unsigned m = __ballot_sync(0xffffffffu, mine);
        if (m == 0) continue;
        unsigned at = 0;
        if (lane == 0) at = atomicAdd(gl.cnt + e, (unsigned)__popc(m));
        at = __shfl_sync(0xffffffffu, at, 0) + __popc(m & ((1u << lane) - 1u));
        if (mine) (e == 0 ? gl.light : gl.heavy)[at] = (int)q;
    }
}

constexpr int kGatherWarps = 8;
template <int NB>
__global__ void __launch_bounds__(32 * kGatherWarps) k_ddm_gather(const __grid_constant__ KArgs a, GatherLists gl) {
    __shared__ float s_sum[kGatherWarps][NB][32];
    __shared__ unsigned s_next;
    const unsigned full = 0xffffffffu;
    const int64_t np = a.ps.np;
    const DevScene &sc = a.sc;
    const int L = sc.L, b = a.b, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const PathState &ps = a.ps;
    // rho / pi times the power over pi r^2 of each map (global, caustic)
    const float inv_g = 1.0f / (3.14159265358979f * a.pm.radius * a.pm.radius);
    const float inv_c = a.pmc.on ? 1.0f / (3.14159265358979f * a.pmc.radius * a.pmc.radius) : 0.0f;
    const float norm = 1.0f / 3.14159265358979f;
    struct At {
        V3 x, ns;
        int row;
    };
    auto vertex = [&](int q) {
        const float4 h0 = ps.hit0[q];
        const float4 tn = __ldg(sc.tri_n + __float_as_int(h0.w));
        const int mat = __float_as_int(tn.w);
        const V3 ng = xyz(tn);
        return At{xyz(h0), dot(xyz(ps.hit1[q]), ng) < 0.0f ? ng : (-1.0f) * ng,
                  __ldg(sc.mat_kind + mat) == kLambert ? mat : sc.n_mat + mat};
    };
    auto gather = [&](const At &v, int wi, int nw, float(&S)[NB]) {
#pragma unroll
        for (int k = 0; k < NB; ++k) S[k] = 0.0f;
        pm_warp_gather(a.pm, v.x, v.ns, L, 1.0f, wi, nw, S);
#pragma unroll
        for (int k = 0; k < NB; ++k) S[k] *= inv_g;
        if (a.pmc.on) pm_warp_gather(a.pmc, v.x, v.ns, L, inv_c, wi, nw, S);
    };
    auto finish = [&](int q, const At &v, const float(&S)[NB]) {
        const float *rho = sc.tab + (size_t)v.row * sc.Lp, *T = ps.T + (size_t)q * sc.Lp;
        Kahan X, Y, Z;
#pragma unroll
        for (int k = 0; k < NB; ++k) {
            const int i = lane + 32 * k;
            if (i < L) {
                const float t = b >= 2 ? T[i] : 1.0f;   // no weight yet at the first vertex
                const float e = t * __ldg(rho + i) * S[k] * norm;
                const float4 w4 = __ldg(sc.wcmf + i);
                X.add(e * w4.x);
                Y.add(e * w4.y);
                Z.add(e * w4.z);
            }
        }
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            two_sum(X, __shfl_xor_sync(full, X.s, o), __shfl_xor_sync(full, X.c, o));
            two_sum(Y, __shfl_xor_sync(full, Y.s, o), __shfl_xor_sync(full, Y.c, o));
            two_sum(Z, __shfl_xor_sync(full, Z.s, o), __shfl_xor_sync(full, Z.c, o));
        }
        if (lane < 3) {
            Kahan acc, x = lane == 0 ? X : lane == 1 ? Y : Z;
            acc.s = ps.acc[lane * np + q];
            acc.c = ps.acc[(3 + lane) * np + q] + x.c;   // what the sums lost goes on to the path's sum
            acc.add(x.s);
            ps.acc[lane * np + q] = acc.s;
            ps.acc[(3 + lane) * np + q] = acc.c;
        }
    };
    float S[NB];
    for (const unsigned n = gl.cnt[1];;) {   // heavy: a block per path
        if (threadIdx.x == 0) s_next = atomicAdd(gl.cnt + 3, 1u);
        __syncthreads();
        const unsigned k = s_next;
        __syncthreads();
        if (k >= n) break;
        const int q = gl.heavy[k];
        const At v = vertex(q);
        gather(v, w, kGatherWarps, S);
#pragma unroll
        for (int j = 0; j < NB; ++j) s_sum[w][j][lane] = S[j];
        __syncthreads();
        if (w == 0) {
#pragma unroll
            for (int j = 0; j < NB; ++j)
                for (int o = 1; o < kGatherWarps; ++o) S[j] += s_sum[o][j][lane];
            finish(q, v, S);
        }
    }
    for (const unsigned n = gl.cnt[0];;) {   // light: a warp per path, two at a time
        unsigned k = 0;
        if (lane == 0) k = atomicAdd(gl.cnt + 2, 2u);
        k = __shfl_sync(full, k, 0);
        if (k >= n) break;
        for (unsigned e = k; e < min(k + 2, n); ++e) {
            const int q = gl.light[e];
            const At v = vertex(q);
            gather(v, 0, 1, S);
            finish(q, v, S);
        }
    }
}
template <int NB>
static cudaError_t launch_gather_nb(const KArgs &a, const GatherLists &gl, int sm, cudaStream_t s) {
    const int64_t want = (a.ps.np + kGatherWarps - 1) / kGatherWarps;
    int per_sm = 4;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_ddm_gather<NB>, 32 * kGatherWarps, 0) != cudaSuccess ||
        per_sm < 1)
        per_sm = 4;
    k_ddm_gather<NB><<<(unsigned)std::min<int64_t>(want, (int64_t)sm * per_sm), 32 * kGatherWarps, 0, s>>>(a, gl);
    return cudaGetLastError();
}
static cudaError_t launch_gather(const KArgs &a, const GatherLists &gl, int sm, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(gl.cnt, 0, 16, s);
    if (e != cudaSuccess) return e;
    k_gather_list<<<(unsigned)((a.ps.np + 255) / 256), 256, 0, s>>>(a, gl);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    return a.sc.L <= 32   ? launch_gather_nb<1>(a, gl, sm, s)
           : a.sc.L <= 64 ? launch_gather_nb<2>(a, gl, sm, s)
           : a.sc.L <= 96 ? launch_gather_nb<3>(a, gl, sm, s)
                          : launch_gather_nb<kPmBins>(a, gl, sm, s);
}

int ddm_photon_pass(const DDMPhotonRun &run, DDMBuffers &buf, cudaStream_t s) {
    const int64_t np = run.count;
    const int L = run.sc.L;
    const int nb = run.g.n_bins;
    if (run.g.n_cells > kMaxCells || nb > kMaxBins) {
        set_error("sddm_render_photon_map: the DDM method supports at most 2048 subdomains");
        return SDDM_ERR_INVALID_ARG;
    }
    if (np <= 0 || run.max_depth < 2) return SDDM_OK;
    const int64_t cap = np;   // one ray per photon in flight
    size_t off = 0;
    auto take = [&](size_t bytes) {
        size_t o = off;
        off = (off + bytes + 255) & ~(size_t)255;
        return o;
    };
    const size_t oT = take(sizeof(float) * (size_t)L * np), oFl = take(4 * np), oH0 = take(16 * np),
                 oH1 = take(16 * np), oIn = take(48 * cap), oSt = take(48 * cap), oCtl = take(queue_counter_bytes(nb)),
                 oOff = take(4 * ((size_t)nb + 1));
    if (off > buf.bytes) {
        if (buf.mem) cudaFree(buf.mem);
        buf.mem = nullptr;
        buf.bytes = 0;
        cudaError_t e = cudaMalloc(&buf.mem, off);
        if (e != cudaSuccess) {
            buf.mem = nullptr;
            set_error("sddm_render_photon_map: photon-state allocation failed");
            return SDDM_ERR_OOM;
        }
        buf.bytes = off;
    }
    char *m = (char *)buf.mem;
    KArgs a{};
    a.sc = run.sc;
    a.g = run.g;
    a.counters = run.counters;
    a.err = run.error_flag;
    a.ps.np = np;
    a.ps.T = (float *)(m + oT);
    a.ps.flags = (int *)(m + oFl);
    a.ps.hit0 = (float4 *)(m + oH0);
    a.ps.hit1 = (float4 *)(m + oH1);
    Queues &Q = a.Q;
    Q.cap = cap;
    Q.in = (float4 *)(m + oIn);
    Q.stage = (float4 *)(m + oSt);
    queue_counters(Q, m + oCtl, nb);
    Q.off = (int *)(m + oOff);
    PhotonPass pp;
    pp.begin = run.begin;
    pp.n_total = run.n_total;
    pp.max_depth = run.max_depth;
    pp.seed = run.seed;
    pp.render_id = run.render_id;
    pp.scale = 3.14159265358979f * run.sc.light_area / (float)run.n_total;
    pp.state_s = run.state_s;
    pp.pos = run.pos;
    pp.dir = run.dir;
    pp.pow = run.pow;

    const int sm = std::max(1, run.sm_count);
    const unsigned path_blocks = (unsigned)std::min<int64_t>((np + 255) / 256, (int64_t)sm * 16);
    const int trace_blocks = sm * (run.blocks_per_sm > 0 ? run.blocks_per_sm : SDDM_TRACE_MIN_BLOCKS);
    const int scatter_blocks = sm * 4;
    const int waves = ddm_waves(run.g);
    const size_t bins_smem = sizeof(int) * (size_t)nb;
    cudaError_t e;
#define PM_CHECK(x)                                                                \
    do {                                                                           \
        if ((e = (x)) != cudaSuccess) return cuda_fail(e, "sddm_render_photon_map: " #x); \
    } while (0)
    PM_CHECK(cudaMemsetAsync(Q.ctl, 0, queue_counter_bytes(nb), s));
    k_photon_emit<<<path_blocks, 256, bins_smem, s>>>(a, pp);
    PM_CHECK(cudaGetLastError());
    *run.launches += 1;
    for (int b = 1; b <= run.max_depth - 1; ++b) {
        for (int w = 0; w < waves; ++w) {
            PM_CHECK(launch_after(true, k_scatter, scatter_blocks, 256, 0, s, a));
            Q.flip();
            a.last_wave = w == waves - 1;
            a.g.continue_cells = ddm_wave_continues(run.g, w, waves);
            PM_CHECK(launch_after(true, k_trace_wave<false>, trace_blocks, 128, 0, s, a));
            *run.launches += 2;
        }
        a.b = b;
        const size_t shade_smem = sizeof(int) * (size_t)((nb + 3) & ~3) + photon_stage_bytes(L);
        // the same limit from every caller: contexts on several threads cannot lower one another's
        constexpr int kMostSmem = (int)(sizeof(int) * (size_t)kMaxBins + photon_stage_bytes(kStageMaxL));
        if (run.sc.mat_nfilm) {
            PM_CHECK(cudaFuncSetAttribute(k_photon_shade<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMostSmem));
            k_photon_shade<true><<<path_blocks, 256, shade_smem, s>>>(a, pp);
        } else {
            PM_CHECK(cudaFuncSetAttribute(k_photon_shade<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMostSmem));
            k_photon_shade<false><<<path_blocks, 256, shade_smem, s>>>(a, pp);
        }
        PM_CHECK(cudaGetLastError());
        *run.launches += 1;
    }
#undef PM_CHECK
    return SDDM_OK;
}
