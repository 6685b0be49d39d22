// DDM trace kernel: one wave of closest-hit and shadow queries over the
// cell-sorted ray queue (Sec. 5's work inside one subdomain, with the
// interface hand-off to the neighbour). Included by ddm.cu after KArgs and
// the grid helpers; kept in its own file so that its source, which the
// recorded DRAM-traffic measurement belongs to, is identifiable.
#pragma once

// Distance at which the ray leaves `cell`, and the neighbour it enters
// (-1 when it leaves the grid). Ties between faces go x, then y, then z. The
// cell's planes and neighbours come from the per-cell table; distances use
// the ray's reciprocal direction.
__device__ __forceinline__ float cell_exit(const DDMScene &g, int cell, V3 o, V3 d, V3 inv, int &next) {
    const float4 p0 = __ldg(g.cell_planes + 2 * cell), p1 = __ldg(g.cell_planes + 2 * cell + 1);
    const int4 n0 = __ldg(g.cell_next + 2 * cell), n1 = __ldg(g.cell_next + 2 * cell + 1);
    float t = __int_as_float(0x7f800000);
    next = -1;
    if (d.x != 0.0f) {
        const bool pos = d.x > 0.0f;
        const float ta = ((pos ? p0.y : p0.x) - o.x) * inv.x;
        if (ta < t) {
            t = ta;
            next = pos ? n0.y : n0.x;
        }
    }
    if (d.y != 0.0f) {
        const bool pos = d.y > 0.0f;
        const float ta = ((pos ? p0.w : p0.z) - o.y) * inv.y;
        if (ta < t) {
            t = ta;
            next = pos ? n0.w : n0.z;
        }
    }
    if (d.z != 0.0f) {
        const bool pos = d.z > 0.0f;
        const float ta = ((pos ? p1.y : p1.x) - o.z) * inv.z;
        if (ta < t) {
            t = ta;
            next = pos ? n1.y : n1.x;
        }
    }
    return t;
}

// Block-wide sums of up to three statistics counters, one atomic per counter
// and block. All threads of the block call it.
__device__ __forceinline__ void block_count3(unsigned long long *c0, unsigned long long v0, unsigned long long *c1,
                                             unsigned long long v1, unsigned long long *c2, unsigned long long v2) {
    __shared__ unsigned long long s_red[32][3];
    for (int off = 16; off > 0; off >>= 1) {
        v0 += __shfl_down_sync(0xffffffffu, v0, off);
        v1 += __shfl_down_sync(0xffffffffu, v1, off);
        v2 += __shfl_down_sync(0xffffffffu, v2, off);
    }
    const int w = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) {
        s_red[w][0] = v0;
        s_red[w][1] = v1;
        s_red[w][2] = v2;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long t0 = 0, t1 = 0, t2 = 0;
        for (int k = 0; k < (int)(blockDim.x >> 5); ++k) {
            t0 += s_red[k][0];
            t1 += s_red[k][1];
            t2 += s_red[k][2];
        }
        if (c0 && t0) atomicAdd(c0, t0);
        if (c1 && t1) atomicAdd(c1, t1);
        if (c2 && t2) atomicAdd(c2, t2);
    }
}

// ------------------------------------------------------ trace one wave
// Persistent warps whose lanes are refilled from the cell-sorted queue while the
// others carry on, so a warp is not held by its slowest ray. Traversal is a
// resumable state machine; a round takes the warp through interior nodes, then
// through leaves. What bounds it is latency and issue together (DRAM 5 %, L1
// wavefronts half of peak, 59 % of the slots issued at 13.5 of 32 lanes when a
// round ran until the last lane stood at a leaf and stopped for every single
// finished lane). So
//  * results, hand-offs and refills wait until kTraceBatch lanes need one: their
//    some 300 instructions ran for two or three lanes at a time. Hotel room, 12
//    launches (512 x 512 x 16 spp), lanes 1 / 4 / 8 / 12 / 16: 13.5 / 13.1 / 13.0
//    / 12.7 / 12.7 ms (20: no better);
//  * the interior phase ends once at most 1 / kTraceQuorum of the busy lanes still
//    descend (64 i.e. the last lane / 6 / 4 / 3: 13.6 / 12.9 / 13.0 / 13.3 ms);
//  * a lane carries only what the traversal itself uses, and triangle records are
//    read in the ray's axis order (make_ray, load_tri) instead of permuted by
//    selects: 12.7 -> 12.1 ms;
//  * 7 resident blocks of 128 threads (72 registers, no spills): 11.4 ms, against
//    12.1 with 8 (64 registers) and 12.1 with 6 (80);
//  * one triangle test for both query kinds (trav_round): 11.0 ms.
// 13.2 ms before all of it; facade room (480 x 270 x 4 spp, 81 bins) 7.4 -> 6.4 ms.
#ifndef SDDM_TRACE_STEPS
#define SDDM_TRACE_STEPS 64   // interior steps per round at most
#endif
constexpr int kTraceSteps = SDDM_TRACE_STEPS;
#ifndef SDDM_TRACE_BATCH
#define SDDM_TRACE_BATCH 16
#endif
constexpr int kTraceBatch = SDDM_TRACE_BATCH;
#ifndef SDDM_TRACE_QUORUM
#define SDDM_TRACE_QUORUM 6
#endif
constexpr int kTraceQuorum = SDDM_TRACE_QUORUM;
// Narrow warps of small waves: lanes at least, and the nodes a cell has on average from which.
constexpr int kTraceMinLanes = 4, kTraceDeepCell = 64;
// Rays a warp buffers in shared memory before appending them to the staging area.
constexpr int kPushBuf = 32;

// Append a warp's buffered rays to the staging area: one atomic, then the
// warp copies the 3 * n float4 words with consecutive lanes on consecutive words.
__device__ __forceinline__ void flush_push_buf(const Queues &Q, const float4 *buf, int n, int lane, int *err) {
    unsigned long long base = 0;
    if (lane == 0) base = atomicAdd(Q.ctl + 0, (unsigned long long)n);
    base = __shfl_sync(0xffffffffu, base, 0);
    __syncwarp();
    if (base + (unsigned long long)n > (unsigned long long)Q.cap) {
        if (lane == 0) atomicCAS(err, 0, 1);
        return;
    }
    float4 *dst = Q.stage + 3 * base;
    for (int k = lane; k < 3 * n; k += 32) dst[k] = buf[k];
    __syncwarp();
}
// Resident 128-thread blocks per SM the trace kernel is compiled for (register
// budget), and launched with unless the build options say otherwise.
#ifndef SDDM_TRACE_MIN_BLOCKS
#define SDDM_TRACE_MIN_BLOCKS 7
#endif

// CHECKED (the subdomain cache, whose cells move between loads): every root,
// child and leaf index is checked against the records the cache holds before
// it is read; a bad one is recorded (codes 8-10) and the ray is dropped.
template <bool COUNT, bool CHECKED = false>
__global__ void __launch_bounds__(128, SDDM_TRACE_MIN_BLOCKS) k_trace_wave(KArgs a) {
    grid_entry();
    const Queues &Q = a.Q;
    const DDMScene &g = a.g;
    // the rays of this launch: the whole wave, or one group's range of it
    // (the groups of cells resident together in the subdomain cache)
    const int q0 = a.q_end > 0 ? (int)a.q_begin : 0;
    const int total = (a.q_end > 0 ? (int)a.q_end : Q.off[g.n_bins]) - q0;
    if (Q.ctl_next && blockIdx.x == 0)   // the cursors of the next wave's sort
        for (int i = threadIdx.x; i < g.n_bins; i += blockDim.x) Q.fill[i] = 0;
    if (total <= 0) return;
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    // A wave with fewer rays than lanes there are spreads over more warps of fewer
    // lanes: a warp's rounds last as long as its longest lane's, so narrow warps
    // answer sooner. At least 32 / 8 / 4 / 2 lanes: photon-mapped hotel room 6.36 /
    // 6.07 / 5.96 / 5.87 ms, hotel room 100 x 100 x 4 spp 1.47 / 1.37 / 1.35 / 1.37.
    // In cells of a few nodes the claims cost more than the rounds (coated tiny room
    // 926 / 943 / 943 us): these keep whole warps.
    const int n_warps = (int)(gridDim.x * (blockDim.x >> 5)), per_warp = (total + n_warps - 1) / n_warps;
    const bool deep = g.node_cap >= (int64_t)kTraceDeepCell * g.n_cells;
    const int lanes = deep ? min(32, max(kTraceMinLanes, per_warp)) : 32, batch = max(1, lanes * kTraceBatch / 32);
    const unsigned lt_mask = (1u << lane) - 1u;
    const int64_t np = a.ps.np;
    unsigned n_cross = 0, n_vis = 0, n_cont = 0;   // n_cont: crossings carried on by the lane
    TravCount tc;

    __shared__ float4 s_push[128 / 32][3 * kPushBuf];   // per-warp hand-off buffers
    float4 *pbuf = s_push[threadIdx.x >> 5];
    int nbuf = 0;              // rays in the warp's buffer (uniform)
    int idx = -1;              // queue index of this lane's ray, -1 = none
    bool exhausted = lane >= lanes;   // no ray left for this lane
    __shared__ unsigned long long s_run[128 / 32][2];    // per warp: reserved run [begin, end) of queue slots
    unsigned long long *run = s_run[threadIdx.x >> 5];
    if (lane == 0) run[0] = run[1] = 0;
    __syncwarp();
    // what a lane carries through the traversal; the rest of its ray (direction,
    // range, path slot, exclusion) is read again from the queue when it finishes
    LaneTrav t;
    t.tmin = t.tw = 0.f;
    t.node = t.sp = 0;
    t.best = t.ep = t.eo = -1;
    t.occ = t.fin = false;
    Crossings cr;   // slabs a shadow ray has crossed
    cr.n = 0;
    float t_cur = 0.f, t_exit = 0.f;
    int rfl = 0, next = -1;
    int stack[kStackSize];

    for (;;) {
        // 1. results, hand-offs and refills, once enough lanes wait for them
        const unsigned m_fin = __ballot_sync(full, t.fin);
        const unsigned m_need = __ballot_sync(full, idx < 0 && !exhausted);
        const unsigned m_busy = __ballot_sync(full, idx >= 0 && !t.fin);
        if (m_busy == 0 || __popc(m_fin | m_need) >= batch) {
            if ((m_fin | m_need) == 0) break;
            // 1a. finished lanes: final result, or hand-off to the neighbouring cell
            bool want = false;
            float4 o0 = make_float4(0, 0, 0, 0), o1 = o0;
            int4 o2 = make_int4(0, 0, 0, 0);
            if (t.fin) {
                const float4 *src = Q.in + 3 * (size_t)idx;
                const float4 r0 = src[0], r1 = src[1];
                const float2 r2f = *reinterpret_cast<const float2 *>(src + 2);
                const V3 ro = xyz(r0), rd = xyz(r1);
                const float t_max = r1.w;
                int q = __float_as_int(r2f.x);
                if (CHECKED && (q < 0 || q >= np)) q = 0;   // recorded when the ray was taken
                const int excl = __float_as_int(r2f.y);
                bool done = false;
                int rfl_next = rfl;
                if (rfl & kRayShadow) {
                    for (int k = (rfl >> 1) & 7; k < cr.n; ++k) {
                        const float4 cn = __ldg(a.sc.tri_n + cr.tri[k]);
                        a.ps.cross_obj[k * np + q] = cr.obj[k];
                        a.ps.cross_mat[k * np + q] = __float_as_int(cn.w);
                        a.ps.cross_cos[k * np + q] = -dot(rd, xyz(cn));
                    }
                    if (t.occ) {
                        a.ps.sh_status[q] = kShadowOccluded;
                        done = true;
                    } else if (t_exit + g.eps >= t_max || next < 0) {
                        a.ps.sh_status[q] = kShadowClear | (cr.n << 4);
                        done = true;
                    }
                    rfl_next = (rfl & 1) | (cr.n << 1);
                } else {
                    if (t.best >= 0) {
                        const V3 x = ro + t.tw * rd;
                        a.ps.hit0[q] = make_float4(x.x, x.y, x.z, __int_as_float(t.best));
                        a.ps.hit1[q] = make_float4(rd.x, rd.y, rd.z, t.tw);
                        done = true;
                    } else if (next < 0) {
                        a.ps.hit0[q] = make_float4(0.f, 0.f, 0.f, __int_as_float(-1));
                        a.ps.hit1[q] = make_float4(rd.x, rd.y, rd.z, 0.f);
                        done = true;
                    }
                }
                t.fin = false;
                if (!done && a.g.continue_cells) {
                    // the lane carries the ray on into the neighbouring cell's
                    // BVH, with the same record it would have handed over
                    const int cell = next;
                    t_cur = fmaxf(t_cur, t_exit);
                    t_exit = cell_exit(g, cell, ro, rd, t.ray.inv, next);
                    t.tmin = fmaxf(0.0f, t_cur - g.eps);
                    t.node = __ldg(g.root + cell);
                    t.sp = 0;
                    t.best = -1;
                    t.occ = false;
                    rfl = rfl_next;
                    t.tw = (rfl & kRayShadow) ? fminf(t_exit + g.eps, t_max) : t_exit + g.eps;
                    ++n_cross;
                    if (COUNT) ++n_vis;
                    if (COUNT) ++n_cont;
                } else {
                    if (!done) {
                        want = true;
                        o0 = make_float4(ro.x, ro.y, ro.z, fmaxf(t_cur, t_exit));
                        o1 = r1;
                        o2 = make_int4(q, excl, rfl_next, next);
                        ++n_cross;
                    }
                    idx = -1;
                }
            }
            if (want && a.last_wave) {   // cannot happen: each wave moves a ray forward along one axis
                atomicCAS(a.err, 0, 4);
                want = false;
            }
            // hand-off: append to the warp's buffer, flushing it to the staging
            // area (one atomic, coalesced stores) when the new rays do not fit
            const unsigned mw = __ballot_sync(full, want);
            if (mw) {
                const int n = __popc(mw);
                if (nbuf + n > kPushBuf) {
                    flush_push_buf(Q, pbuf, nbuf, lane, a.err);
                    nbuf = 0;
                }
                if (want) {
                    float4 *slot = pbuf + 3 * (nbuf + __popc(mw & lt_mask));
                    slot[0] = o0;
                    slot[1] = o1;
                    slot[2] = make_float4(__int_as_float(o2.x), __int_as_float(o2.y), __int_as_float(o2.z),
                                          __int_as_float(o2.w));
                    const int bin = ray_bin(g, next, o2.z, o0, o1);
                    const unsigned peers = __match_any_sync(mw, bin);
                    if (lane == __ffs(peers) - 1) atomicAdd(Q.cnt + bin, __popc(peers));
                }
                nbuf += n;
                __syncwarp();
            }
            // 1b. idle lanes take the next rays of the queue, from a run of
            //     queue slots the warp reserves at a time, one for each of its
            //     lanes (one atomic per run instead of one per refill)
            const bool need = idx < 0 && !exhausted;
            const unsigned m = __ballot_sync(full, need);
            if (m) {
                const unsigned want_n = __popc(m);
                const unsigned long long cbeg = run[0], cend = run[1];
                const unsigned long long avail = cend - cbeg;
                unsigned long long nb = 0;
                if (avail < want_n) {
                    if (lane == 0) nb = atomicAdd(Q.ctl + 1, (unsigned long long)lanes);
                    nb = __shfl_sync(full, nb, 0);
                }
                const unsigned rank = __popc(m & lt_mask);
                const unsigned long long mine = rank < avail ? cbeg + rank : nb + (rank - avail);
                __syncwarp();
                if (lane == 0) {
                    if (avail >= want_n) {
                        run[0] = cbeg + want_n;
                    } else {
                        run[0] = nb + (want_n - avail);
                        run[1] = nb + lanes;
                    }
                }
                __syncwarp();
                if (need) {
                    const unsigned long long my = mine;
                    if (my < (unsigned long long)total) {
                        idx = q0 + (int)my;
                        const float4 *src = Q.in + 3 * (size_t)idx;
                        const float4 r0 = src[0], r1 = src[1], r2f = src[2];
                        int q = __float_as_int(r2f.x);
                        const int excl = __float_as_int(r2f.y);
                        rfl = __float_as_int(r2f.z);
                        int cell = __float_as_int(r2f.w);
                        if (CHECKED && (q < 0 || q >= np || cell < 0 || cell >= g.n_cells)) {
                            trace_check_fail(a.err, 12, q, cell);
                            q = 0;
                            cell = 0;
                        }
                        t.ray = make_ray(xyz(r0), xyz(r1));
                        t_cur = r0.w;
                        t_exit = cell_exit(g, cell, xyz(r0), xyz(r1), t.ray.inv, next);
                        t.tmin = fmaxf(0.0f, t_cur - g.eps);
                        t.node = __ldg(g.root + cell);
                        if (CHECKED && (t.node < 0 || t.node >= g.node_cap)) {
                            trace_check_fail(a.err, 8, cell, t.node);
                            t.node = ~0;   // an empty leaf: the ray ends here
                        }
                        t.sp = 0;
                        t.best = -1;
                        t.occ = false;
                        if (COUNT) ++n_vis;
                        t.ep = excl >= 0 ? excl : -1;
                        if (rfl & kRayShadow) {
                            t.tw = fminf(t_exit + g.eps, r1.w);
                            cr.n = (rfl >> 1) & 7;
                            for (int k = 0; k < cr.n; ++k) cr.obj[k] = a.ps.cross_obj[k * np + q];
                        } else {
                            t.tw = t_exit + g.eps;
                            t.eo = excl <= -2 ? -excl - 2 : -1;
                        }
                    } else {
                        exhausted = true;
                    }
                }
            }
        }

        // 2. one traversal round
        trav_round<COUNT, CHECKED, kTraceSteps, kTraceQuorum>(
            g.nodes, g.tris, a.sc.tri_obj, t, cr, stack, idx >= 0 && !t.fin, (rfl & kRayShadow) != 0,
            [&]() { return xyz(Q.in[3 * (size_t)idx + 1]); }, tc, a.err, g.node_cap, g.tri_cap);
    }
    if (nbuf > 0) flush_push_buf(Q, pbuf, nbuf, lane, a.err);
    block_count3(a.counters + 3, n_cross, nullptr, 0, nullptr, 0);
    if (COUNT) {
        __syncthreads();
        block_count3(a.counters + 5, tc.nodes, a.counters + 6, tc.tris, a.counters + 7, n_vis);
        __syncthreads();   // the reduction's shared slots are read by thread 0 above
        block_count3(a.counters + 10, n_cont, nullptr, 0, nullptr, 0);
    }
}
