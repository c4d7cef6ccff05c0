// Fused light-curve kernels: time -> phase -> z -> Eq. 5 -> mean over
// sub-exposures, for a tile of parameter vectors x a tile of times.
//
// FP32 kernel.  A CTA owns a chunk of consecutive 128-time groups (4
// consecutive times per lane of a warp) and a tile of up to 32 parameter
// vectors (lane i of a warp speaks for pv i).  One bulk asynchronous copy
// (TMA engine, mbarrier completion, bounded wait) stages the tile's pv
// records and the chunk's group summaries into shared memory.  Stream warps
// then take the groups: per group one transit test per pv, whole 512-byte
// row segments of exactly 1 for the pvs outside their windows (bulk
// asynchronous stores from a constant shared-memory row), and a work item
// (pv, group) in a shared-memory queue for the others; the remaining warps
// evaluate the items as they appear (candidate samples compacted per warp).
// FP64 kernel: the same groups and queue with CTAs of two warps, transit
// decisions in FP32, every sample in FP64.
//
// Mixed precision (FP32 bulk):
//  * per time, once per call (points_group): dt = t - t_g in FP64, kept as
//    a float pair (dh, dl) -- t_g is the first time of the time's group;
//  * per (CTA, pv), FP64: A = frac((t_ref - T0) / P) as a float pair at the
//    first group of the CTA's chunk, carried to each group in float-float;
//  * per (pv, time): coarse phase psi = A + dh / P with one FMA, rounded
//    with two additions (no FP64, no conversion per point).  If the
//    whole exposure lies outside the pv's transit window the point is 1
//    exactly and nothing else is computed.  Otherwise the phase is formed in
//    float-float (error ~1e-9 of a cycle) and every sub-exposure (two at a
//    time) goes through Kepler (FP32 third-order steps in the offset form,
//    FP64 above e = 0.8),
//    the projected distance, the covered area and the profile row lookup.
// FP64 form: the same structure with every step in FP64 and the phase
// reduced per sub-exposure as tau = t_s - T0 - P rint((t_s - T0) / P).
#include <algorithm>

#include "rr_device.cuh"

namespace rr {

// Order of the time chunks of the FP32 per-point kernels, heaviest first (one
// CTA): chunk i (groups i gpc .. i gpc + gpc - 1) weighs the exposure
// sub-samples of its groups; order[rank] = i, ties in index order.  With
// passbands of different supersampling the chunks' work differs several-fold
// (a chunk of 30-sub-exposure times against one of single samples), and the
// heaviest CTAs are best started first: the last wave then holds light ones.
// More than 1024 chunks: index order.
__global__ void __launch_bounds__(1024) rr_chunk_order_kernel(const GroupInfo* __restrict__ grp, int ngroups,
                                                              int gpc, int nchunks, int* __restrict__ order) {
    __shared__ float w[1024];
    const int i = threadIdx.x;
    if (nchunks > 1024) {
        for (int j = i; j < nchunks; j += blockDim.x) order[j] = j;
        return;
    }
    if (i < nchunks) {
        float s = 0.0f;
        const int g1 = min(ngroups, (i + 1) * gpc);
        for (int g = i * gpc; g < g1; ++g) s += grp[g].weight;
        w[i] = s;
    }
    __syncthreads();
    if (i < nchunks) {
        const float wi = w[i];
        int rank = 0;
        for (int j = 0; j < nchunks; ++j) rank += (w[j] > wi) || (w[j] == wi && j < i);
        order[rank] = i;
    }
}

cudaError_t launch_chunk_order(rr_ctx* c, int npt, void* ws_grp, void* ws_ord, cudaStream_t s) {
    const int ngroups = (npt + kWarpPts - 1) / kWarpPts;
    const int gpc = groups_per_cta(npt);
    rr_chunk_order_kernel<<<1, 1024, 0, s>>>((const GroupInfo*)ws_grp, ngroups, gpc, time_chunks(npt, gpc),
                                             (int*)ws_ord);
    c->launches++;
    return cudaGetLastError();
}

// Stores the 4 outputs of a lane (one 16-byte store when the row is vector-aligned).
__device__ __forceinline__ void store4(float* out, const float (&f)[4], const int (&pbv)[4], bool full) {
    if (full) {
        __stcs(reinterpret_cast<float4*>(out), make_float4(f[0], f[1], f[2], f[3]));
    } else {
        #pragma unroll
        for (int q = 0; q < 4; ++q)
            if (pbv[q] >= 0) __stcs(out + q, f[q]);
    }
}

template <bool STAGE_ROWS, bool SS1, bool COUNT>
__global__ void __launch_bounds__(kBlock, 4) rr_flux_mixed_kernel(const double* __restrict__ times,
                                                               const float2* __restrict__ pdt,
                                                               const int32_t* __restrict__ ppb,
                                                               const GroupInfo* __restrict__ grp,
                                                               int npt, int npv, PbParams pbp, RecLayout L,
                                                               int pv_tile, int groups_per_cta, int chunk_groups,
                                                               const char* __restrict__ records,
                                                               const char* __restrict__ rowsg,
                                                               float* __restrict__ flux,
                                                               int32_t* __restrict__ pv_status, int vec_store,
                                                               int stream_warps, unsigned long long* counts,
                                                               const int* __restrict__ chunk_order, int* err) {
    extern __shared__ __align__(16) unsigned char smem[];
    uint64_t* bar = reinterpret_cast<uint64_t*>(smem);
    PbShared* ps = reinterpret_cast<PbShared*>(smem + kOffPb);
    char* recs = reinterpret_cast<char*>(smem + kOffRecsFlux);
    TileCounters* tc = reinterpret_cast<TileCounters*>(smem + kOffRed);

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    FluxList* wl = reinterpret_cast<FluxList*>(smem + kOffWl + warp * kFlBytes);
    const int ngroups = (npt + kWarpPts - 1) / kWarpPts;
    // grid: x = pv tile, y = time chunk (in launch order; chunk_order: heaviest first)
    const int chunk = chunk_order ? __ldg(chunk_order + blockIdx.y) : (int)blockIdx.y;
    const int gbeg = chunk * groups_per_cta;
    const int gend = min(ngroups, gbeg + groups_per_cta);
    const int pv0 = blockIdx.x * pv_tile;
    const int npv_t = min(pv_tile, npv - pv0);
    // staged: headers of the tile, then (STAGE_ROWS) their profile rows, then the item queue
    char* srows = recs + (size_t)pv_tile * L.head_bytes;
    char* qbase = srows + (STAGE_ROWS ? (size_t)pv_tile * L.rows_bytes : 0);
    const ItemQueue queue = queue_at(qbase, pv_tile * groups_per_cta);
    // constant output rows of one group (1 and NaN), sources of the bulk stores
    float* rows1 = reinterpret_cast<float*>(qbase + queue_bytes(pv_tile * groups_per_cta));
    float* rowsnan = rows1 + kWarpPts;
    // the summaries of the CTA's groups, copied with the records
    GroupInfo* sgrp = reinterpret_cast<GroupInfo*>(rowsnan + kWarpPts);
    const uint32_t hbytes = (uint32_t)npv_t * (uint32_t)L.head_bytes;
    const uint32_t rbytes = STAGE_ROWS ? (uint32_t)npv_t * (uint32_t)L.rows_bytes : 0u;
    const uint32_t gbytes = (uint32_t)(gend - gbeg) * (uint32_t)sizeof(GroupInfo);
    queue_init(queue, tc, pv_tile * groups_per_cta, gbeg);
    for (int j = tid; j < kWarpPts; j += blockDim.x) {
        rows1[j] = 1.0f;
        rowsnan[j] = __int_as_float(0x7fc00000);
    }
    fence_proxy_async_smem();   // the bulk stores read these through the async proxy
    if (tid == 0) {
        mbar_init(bar, 1);
        mbar_expect_tx(bar, hbytes + rbytes + gbytes);
        bulk_g2s(sgrp, grp + gbeg, gbytes, bar);
        const char* src = records + (size_t)pv0 * L.head_bytes;
        for (uint32_t off = 0; off < hbytes; off += 65536u) {
            const uint32_t n = hbytes - off < 65536u ? hbytes - off : 65536u;
            bulk_g2s(recs + off, src + off, n, bar);
        }
        const char* rsrc = rowsg + (size_t)pv0 * L.rows_bytes;
        for (uint32_t off = 0; off < rbytes; off += 65536u) {
            const uint32_t n = rbytes - off < 65536u ? rbytes - off : 65536u;
            bulk_g2s(srows + off, rsrc + off, n, bar);
        }
    }
    stage_pb(pbp, ps);
    __syncthreads();   // publishes the barrier initialisation, the counters and the passband table
    bool ok = mbar_wait_bounded(bar, 0);
    if (!ok) {
        if (tid == 0) atomicExch(err, kErrBarrierTimeout);
        mbar_wait_bounded(bar, 0);
    }
    if (__syncthreads_or(ok ? 0 : 1)) return;
    float4* cta_ph = reinterpret_cast<float4*>(smem + kOffCta);
    const int gref = gbeg - gbeg % chunk_groups;
    const float2 tref = __ldg(reinterpret_cast<const float2*>(grp + gref) + 2);   // its toff
    cta_phase(cta_ph, times, gref, recs, L.head_bytes, npv_t);
    __syncthreads();

    const float nanf_ = __int_as_float(0x7fc00000);
    const uint64_t l2_pol = l2_evict_first_policy();
    Tally tl{};   // the counting form's per-thread sample counts

    // a group: the tile's transit mask; every pv outside it is 1 (NaN for an
    // invalid pv or passband index) without arithmetic, the others are queued
    auto do_group = [&](int g) {
        const int p0 = g * kWarpPts + 4 * lane;
        GroupState gs;
        group_load(gs, sgrp, g - gbeg, tref, cta_ph, recs, L.head_bytes, npv_t);
        unsigned bad;
        float4 cl;
        const unsigned may = group_decide(gs, recs, L.head_bytes, npv_t, bad, cl);
        if (may) queue_push(queue, tc, may, g, cl);
        int pbv[4] = {0, 0, 0, 0};
        if (!gs.full) load_pb(ppb, p0, npt, pbv);    // a partial group or invalid passbands
        float fb[4];
        #pragma unroll
        for (int q = 0; q < 4; ++q) fb[q] = pbv[q] < L.npb ? 1.0f : nanf_;
        const bool full = (vec_store & 1) && (p0 + 3 < npt);
        float* out = flux + (size_t)pv0 * npt + p0;
        // the pvs of the tile that need no arithmetic
        unsigned rest = (npv_t >= 32 ? 0xffffffffu : ((1u << npv_t) - 1u)) & ~may;
        if ((vec_store & 2) && gs.full) {
            // a whole 512-byte row segment per pv from a constant row in shared
            // memory, one bulk asynchronous store per lane (lane i: pv i); the
            // addresses are 16-byte aligned (npt % 4 == 0, aligned flux in device memory)
            if ((rest >> lane) & 1u) {
                bulk_s2g(flux + (size_t)(pv0 + lane) * npt + (size_t)g * kWarpPts,
                         ((bad >> lane) & 1u) ? rowsnan : rows1, kWarpPts * sizeof(float), l2_pol);
                bulk_commit();
            }
            rest = 0u;
        }
        #pragma unroll 1
        while (rest) {
            const int i = __ffs(rest) - 1;
            rest &= rest - 1u;
            const bool inval = (bad >> i) & 1u;
            const float f[4] = {inval ? nanf_ : fb[0], inval ? nanf_ : fb[1], inval ? nanf_ : fb[2],
                                inval ? nanf_ : fb[3]};
            store4(out + (size_t)i * npt, f, pbv, full);
        }
    };

    // an item: every time of the group for one pv that may transit
    auto do_item = [&](int it, int key) {
        const float4 c = queue.c[it];
        const int g = key >> 5, i = key & 31;
        const int p0 = g * kWarpPts + 4 * lane;
        float dh[4], dl[4];
        int pbv[4];
        load_points(pdt, ppb, p0, npt, dh, dl, pbv);
        const char* rec = recs + (size_t)i * L.head_bytes;
        const PvHead<float>& H = *reinterpret_cast<const PvHead<float>*>(rec);
        const PvPb<float>* PB = reinterpret_cast<const PvPb<float>*>(rec + L.off_pb);
        const float* rows = STAGE_ROWS ? reinterpret_cast<const float*>(srows + (size_t)i * L.rows_bytes)
                                       : reinterpret_cast<const float*>(rowsg + (size_t)(pv0 + i) * L.rows_bytes);
        float f[4];
        unsigned cand = 0;
        #pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int pb = pbv[q];
            f[q] = pb < L.npb ? 1.0f : nanf_;
            if (pb < 0 || pb >= L.npb) continue;
            const float psi = fmaf(dh[q], H.Bh, c.x);
            const float d = psi - round_nearest(psi);
            if (fabsf(d) <= PB[pb].win_pc + c.w) cand |= 1u << q;
        }
        bool bad = false;
        if constexpr (SS1) {
          if (__any_sync(0xffffffffu, cand != 0)) {
            // one sample per time: the candidates are the samples
            int bq[4];
            const int nc = build_list_ss1_flux(wl, cand, dh, dl, pbv, bq);
            #pragma unroll 1
            for (int e0 = 0; e0 < nc; e0 += 32) {
                const int j = e0 + lane;
                if (j < nc) {
                    const int pb = wl->ps[j];
                    const float2 cd = wl->cand[j];
                    const Phase32 ph = precise_phase(cd.x, cd.y, c.x, c.y, H.Bh, H.Bl);
                    if (COUNT) ++tl.n[RR_COUNT_TIMES];
                    wl->pacc[j] = delta32<COUNT>(H, PB[pb], rows + (size_t)pb * L.rows_per_pb * L.ng_pad, L.ng,
                                                 ph.fr_h, ph.fr_l, 0.0f, 0.0f, 0.0f, bad, &tl);
                }
            }
            __syncwarp();
            #pragma unroll
            for (int q = 0; q < 4; ++q)
                if ((cand >> q) & 1u) f[q] = 1.0f - wl->pacc[bq[q]];
            __syncwarp();
          }
        } else if (__any_sync(0xffffffffu, cand != 0)) {
            int nc, base;
            const int ns = build_list_flux(wl, cand, dh, dl, pbv, c.x, c.y, H.Bh, H.Bl, ps, nc, base);
            if (COUNT && lane == 0) tl.n[RR_COUNT_TIMES] += nc;
            // The item's flattened samples [0, ns) in 32 contiguous runs of run = ceil(ns / 32),
            // one per lane.  A lane walks its run in order, summing the sub-exposures of the
            // candidate at hand: the sum of a candidate that starts and ends inside the run is
            // final; the candidate at the run's start (head) and the one at its end (tail) may
            // go on in the neighbouring runs, and are combined once per item, in lane order.
            const int run = (ns + 31) >> 5;
            const int e_beg = min(lane * run, ns), e_end = min(e_beg + run, ns);
            int jh = -1, jt = -1;          // head and tail candidates of the run (-1: none)
            float ph = 0.0f, pt = 0.0f;    // their partial sums over the run
            if (e_beg < e_end) {
                // the candidate holding sample e_beg: the last j with soff(j) <= e_beg
                int lo = 0, hi = nc - 1;
                while (lo < hi) {
                    const int mid = (lo + hi + 1) >> 1;
                    if ((wl->ps[mid] >> 5) <= e_beg) lo = mid; else hi = mid - 1;
                }
                int j = lo;
                int pw = wl->ps[j];
                int next = wl->ps[j + 1] >> 5;     // first sample of candidate j + 1 (ps[nc] = ns << 5)
                // the candidate's passband: its constants, profile row and sub-exposure spacing,
                // looked up once per candidate rather than per sample
                int pb = pw & 31;
                float2 cd = wl->cand[j];
                float sub = (float)(e_beg - (pw >> 5));
                float part = 0.0f;
                jh = j;
                const size_t row_stride = (size_t)L.rows_per_pb * L.ng_pad;
                if constexpr (COUNT) {   // one sample at a time
                    #pragma unroll 1
                    for (int e = e_beg; e < e_end; ++e) {
                        if (e == next) {
                            // candidate j ends inside the run: the head's sum, or a final one
                            if (j == jh) ph = part; else wl->pacc[j] = part;
                            ++j;
                            pw = wl->ps[j];
                            next = wl->ps[j + 1] >> 5;
                            pb = pw & 31;
                            cd = wl->cand[j];
                            sub = 0.0f;
                            part = 0.0f;
                        }
                        part += delta32<COUNT>(H, PB[pb], rows + pb * row_stride, L.ng, cd.x, cd.y,
                                               sub, ps->first[pb], ps->step[pb], bad, &tl);
                        sub += 1.0f;
                    }
                } else {   // two at a time, the second possibly of the next candidate
                    #pragma unroll 1
                    for (int e = e_beg; e < e_end; e += 2) {
                        auto finish = [&]() {   // candidate j ends inside the run: the head's sum, or a final one
                            if (j == jh) ph = part; else wl->pacc[j] = part;
                            ++j;
                            next = wl->ps[j + 1] >> 5;
                            part = 0.0f;
                        };
                        if (e == next) {
                            finish();
                            pb = wl->ps[j] & 31;
                            cd = wl->cand[j];
                            sub = 0.0f;
                        }
                        const bool two = e + 1 < e_end, cross = two && e + 1 == next;
                        Sub32 a[2];
                        a[0] = {cd, sub, ps->first[pb], ps->step[pb], PB + pb, rows + pb * row_stride};
                        if (cross) {
                            pb = wl->ps[j + 1] & 31;
                            cd = wl->cand[j + 1];
                            sub = -1.0f;
                        }
                        a[1] = {cd, sub + 1.0f, ps->first[pb], ps->step[pb], PB + pb, rows + pb * row_stride};
                        float d[2];
                        delta32_pair(H, a, two, L.ng, d, bad);
                        part += d[0];
                        if (cross) finish();
                        part += d[1];
                        sub += 2.0f;
                    }
                }
                if (j == jh) ph = part; else { jt = j; pt = part; }
            }
            // a tail that goes on into the next run is added in front of that run's head
            const int tprev_j = __shfl_up_sync(0xffffffffu, jt, 1);
            const float tprev_p = __shfl_up_sync(0xffffffffu, pt, 1);
            if (lane > 0 && jh >= 0 && tprev_j == jh) ph = tprev_p + ph;
            const int hnext_j = __shfl_down_sync(0xffffffffu, jh, 1);
            if (jt >= 0 && (lane == 31 || hnext_j != jt)) wl->pacc[jt] = pt;   // the tail ends with the run
            // heads: segmented inclusive scan over the lanes by candidate (fixed order); the last
            // lane of each segment holds the candidate's sum
            float v = ph;
            #pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const float y = __shfl_up_sync(0xffffffffu, v, o);
                const int ky = __shfl_up_sync(0xffffffffu, jh, o);
                if (lane >= o && ky == jh) v = y + v;
            }
            if (jh >= 0 && (lane == 31 || hnext_j != jh)) wl->pacc[jh] = v;
            __syncwarp();
            int jj = base;
            #pragma unroll
            for (int q = 0; q < 4; ++q) {
                if (cand & (1u << q)) {
                    f[q] = 1.0f - wl->pacc[jj] * ps->inv_ss[pbv[q]];
                    ++jj;
                }
            }
            __syncwarp();
        }
        if (bad && pv_status) atomicOr(pv_status + pv0 + i, RR_PV_KEPLER);
        store4(flux + (size_t)(pv0 + i) * npt + p0, f, pbv, (vec_store & 1) && (p0 + 3 < npt));
    };

    // Warps below stream_warps first take the groups (the output stream) and
    // produce the items; the others start on the items at once.  Every warp
    // then drains the items.
    if (warp < stream_warps) {
        #pragma unroll 1
        while (true) {
            int g = 0;
            if (lane == 0) g = atomicAdd(&tc->next_group, 1);
            g = __shfl_sync(0xffffffffu, g, 0);
            if (g >= gend) break;
            do_group(g);
        }
    }
    queue_producer_done(tc);
    int idle = 0;
    #pragma unroll 1
    while (true) {
        const int it = queue_claim(tc);
        if (it >= 0) {
            const int key = queue_key(queue, it);
            if (key < 0) {
                if (lane == 0) atomicExch(err, kErrQueueTimeout);
                break;
            }
            do_item(it, key);
            continue;
        }
        if (queue_finished(tc)) {
            // no producer left: the queue is final; drain what is still claimable
            const int last = queue_claim(tc);
            if (last < 0) break;
            const int key = queue_key(queue, last);
            if (key < 0) {
                if (lane == 0) atomicExch(err, kErrQueueTimeout);
                break;
            }
            do_item(last, key);
            continue;
        }
        // other warps still take groups: wait for their items (bounded)
        if (++idle > (1 << 22)) {
            if (lane == 0) atomicExch(err, kErrQueueTimeout);
            break;
        }
        __nanosleep(64);
    }
    if (COUNT) tally_flush(tl, counts);
    bulk_wait_all();   // the bulk stores read shared memory that ends with the CTA
}

// ----------------------------- FP64 form -----------------------------------
//
// Bound by the FP64 pipe (two lanes per clock and SM).  The groups and the item queue of the FP32
// kernel in place of a window test in FP64 for every (pv, time), candidate times of a whole warp
// compacted before they are evaluated, and samples of about 130 FP64 instructions (orbit64,
// atan2_upper64; about 480 with a Newton iteration from the mean anomaly, sqrt and atan2).
// CTAs of two warps: an item is a chain of ~6,000 cycles per 32 samples, and small CTAs keep
// up to 16 items of an SM in flight without waiting for a CTA's longest.  Measured: 512 pvs x
// 10,007 times 403 -> 100 us (1.06 million FP64 instructions of warps, 0.67 of the pipe's
// rate), 200 x 5,000 with 10 sub-exposures 4,686 -> 127, 1 x 2,000 24.3 -> 13.9.

template <bool SS1, int Q>
__global__ void __launch_bounds__(kBlock64, 8) rr_flux_fp64_kernel(const double* __restrict__ times,
                                                                 const int32_t* __restrict__ pb_index, int npt, int npv,
                                                                 PbParams pbp, RecLayout L, int pv_tile, int groups_per_cta,
                                                                 const char* __restrict__ records,
                                                                 const char* __restrict__ rowsg, double* __restrict__ flux,
                                                                 int32_t* __restrict__ pv_status, int bulk, int sum_shift,
                                                                 float inv_ss, int* err) {
    extern __shared__ __align__(16) unsigned char smem[];
    uint64_t* bar = reinterpret_cast<uint64_t*>(smem);
    TileCounters* tc = reinterpret_cast<TileCounters*>(smem + kOff64Tc);
    PbShared64* ps = reinterpret_cast<PbShared64*>(smem + kOff64Pb);
    char* recs = reinterpret_cast<char*>(smem + kOff64Recs);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    List64* wl = reinterpret_cast<List64*>(smem + kOff64Wl + warp * kList64Bytes);
    constexpr int kPts = 32 * Q;   // times per group
    const int ngroups = (npt + kPts - 1) / kPts;
    const Cta64 cta = cta64(npv, pv_tile);
    const int gbeg = cta.chunk * groups_per_cta;
    const int gend = min(ngroups, gbeg + groups_per_cta);
    const int pv0 = cta.tile * pv_tile;
    const int npv_t = min(pv_tile, npv - pv0);
    char* qbase = recs + (size_t)pv_tile * L.head_bytes;
    const ItemQueue queue = queue_at(qbase, pv_tile * groups_per_cta);
    const double nan_ = __longlong_as_double(0x7ff8000000000000ll);
    queue_init(queue, tc, pv_tile * groups_per_cta, gbeg);
    ConstRows64 cr;
    cr.init(reinterpret_cast<double*>(qbase + queue_bytes(pv_tile * groups_per_cta)), kPts);
    stage_pb64(pbp, ps);
    if (!stage_to_smem(recs, records + (size_t)pv0 * L.head_bytes, (uint32_t)npv_t * (uint32_t)L.head_bytes, bar, err))
        return;

    auto do_group = [&](int g) {
        Times64<Q> T;
        load_times64(times, pb_index, g, npt, L.npb, T);
        GroupState gs;
        group_state64(T, L.npb, recs, L.head_bytes, npv_t, gs);
        unsigned bad;
        float4 cl;
        const unsigned may = group_decide64(gs, recs, L.head_bytes, npv_t, bad, cl);
        if (may) queue_push(queue, tc, may, g, cl);
        cr.store(T, gs.full, may, bad, npv_t, L.npb, flux + (size_t)pv0 * npt + (size_t)g * kPts, npt, bulk);
    };

    auto do_item = [&](int it, int key) {
        const float4 c = queue.c[it];
        const int g = key >> 5, i = key & 31;
        Times64<Q> T;
        load_times64(times, pb_index, g, npt, L.npb, T);
        const char* rec = recs + (size_t)i * L.head_bytes;
        const PvHead<double>& H = *reinterpret_cast<const PvHead<double>*>(rec);
        const PvPb<double>* PB = reinterpret_cast<const PvPb<double>*>(rec + L.off_pb);
        const double* rows = reinterpret_cast<const double*>(rowsg + (size_t)(pv0 + i) * L.rows_bytes);
        const unsigned cand = candidates64(T, H, PB, L.npb, c);
        double f[Q];
        #pragma unroll
        for (int q = 0; q < Q; ++q) f[q] = T.pb[q] < L.npb ? 1.0 : nan_;
        bool bad = false;
        if (__any_sync(0xffffffffu, cand != 0)) {
            int nc, bq;
            const double zero[Q] = {};
            const int ns = build_list64<SS1, Q>(wl, cand, T, zero, ps, nc, bq);
            auto row_of = [&](int pb) { return rows + (size_t)pb * L.rows_per_pb * L.ng_pad; };
            if (SS1) {
                #pragma unroll 1
                for (int j = lane; j < nc; j += 32) {
                    const int pb = wl->ps[j] & 31;
                    wl->v[j] = delta64(H, PB[pb], row_of(pb), L.ng, wl->t[j], bad);
                }
                __syncwarp();
            } else {
                // The item's flattened samples, kWarpPts at a time into the list, neighbouring ones in neighbouring
                // lanes; then a time's samples are added in an order of their indices alone (whatever other times
                // the group holds, and whatever its size): 2^sum_shift lanes per candidate, each adding every
                // 2^sum_shift-th sample in order, and a fixed tree over them.  A finished sum takes its time's place in
                // the list; the one candidate open at the end of a pass is carried.  Against a contiguous run of the
                // item's samples per lane, whose sums depended on where the runs were cut (and whose lanes took different
                // branches): 200 pvs x 5,000 times with 10 sub-exposures 176 -> 127 us, 64 x 3,000 103 -> 85, 1 x
                // 20,000 with 30 52 -> 45, 8 x 500 with 1,000 3,930 -> 2,415; slower where one pv's transits are
                // far apart and long (1 x 20,000 with 30 at random times, the call 195 -> 203: the sums' chain).
                const int R = 1 << sum_shift;
                int lo = 0, jc = 0;      // the lane's last candidate; the first unfinished one
                double carry = 0.0;      // of candidate jc: the sum of residue lane % R so far
                #pragma unroll 1
                for (int e0 = 0; e0 < ns; e0 += kWarpPts) {
                    const int e1 = min(ns, e0 + kWarpPts);
                    #pragma unroll 1
                    for (int e = e0 + lane; e < e1; e += 32) {
                        // the candidate holding sample e: by division where every passband has as many (exact: e below
                        // 2^17 and at least half a sample from a multiple of the count), else by bisection
                        if (inv_ss > 0.0f) {
                            lo = (int)(((float)e + 0.5f) * inv_ss);
                        } else {
                            int hi = nc - 1;
                            while (lo < hi) {
                                const int mid = (lo + hi + 1) >> 1;
                                if ((wl->ps[mid] >> 5) <= e) lo = mid; else hi = mid - 1;
                            }
                        }
                        const int pw = wl->ps[lo], pb = pw & 31, sub = e - (pw >> 5), at = ps->first[pb];
                        const double off = at >= 0 ? ps->off[at + sub] : sub_offset64(ps->exptime[pb], ps->ss[pb], sub);
                        wl->v[e - e0] = delta64(H, PB[pb], row_of(pb), L.ng, wl->t[lo] + off, bad);
                    }
                    __syncwarp();
                    const int j1 = __shfl_sync(0xffffffffu, lo, (e1 - 1 - e0) & 31);   // the candidate of sample e1 - 1
                    const bool open = (wl->ps[j1 + 1] >> 5) > e1;
                    const int last = (j1 - jc) << sum_shift;
                    double next = 0.0;
                    #pragma unroll 1
                    for (int u0 = 0; u0 < last + R; u0 += 32) {
                        const int u = u0 + lane, j = jc + (u >> sum_shift), r = u & (R - 1);
                        double a = j == jc ? carry : 0.0;
                        int end = 0;
                        if (j <= j1) {
                            end = wl->ps[j + 1] >> 5;
                            int e = (wl->ps[j] >> 5) + r;
                            if (e < e0) e += ((e0 - e + R - 1) >> sum_shift) << sum_shift;
                            #pragma unroll 4
                            for (; e < min(end, e1); e += R) a += wl->v[e - e0];
                        }
                        double sum = a;
                        for (int o = 1; o < R; o <<= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
                        if (j <= j1 && r == 0 && end <= e1) wl->t[j] = sum;
                        if (open && last >= u0 && last < u0 + 32)
                            next = __shfl_sync(0xffffffffu, a, last - u0 + (lane & (R - 1)));
                    }
                    carry = next;
                    jc = open ? j1 : j1 + 1;
                    __syncwarp();
                }
            }
            int j = bq;
            #pragma unroll
            for (int q = 0; q < Q; ++q) {
                if ((cand >> q) & 1u) {
                    f[q] = SS1 ? 1.0 - wl->v[j] : 1.0 - wl->t[j] / ps->ss[T.pb[q]];
                    ++j;
                }
            }
            __syncwarp();
        }
        if (bad && pv_status) atomicOr(pv_status + pv0 + i, RR_PV_KEPLER);
        double* out = flux + (size_t)(pv0 + i) * npt + (size_t)g * kPts + Q * lane;
        #pragma unroll
        for (int q = 0; q < Q; ++q)
            if (T.pb[q] >= 0) __stcs(out + q, f[q]);
    };

    // every warp streams its groups first, then drains the items (FP64 arithmetic dominates)
    #pragma unroll 1
    while (true) {
        int g = 0;
        if (lane == 0) g = atomicAdd(&tc->next_group, 1);
        g = __shfl_sync(0xffffffffu, g, 0);
        if (g >= gend) break;
        do_group(g);
    }
    queue_producer_done(tc);
    queue_drain(queue, tc, err, do_item);
    bulk_wait_all();   // the bulk stores read shared memory that ends with the CTA
}

static size_t flux_smem(int pv_tile, int rec_bytes, bool f64, int gpc) {
    if (f64)
        return kOff64Recs + (size_t)pv_tile * rec_bytes + queue_bytes(pv_tile * gpc) + 2 * kWarpPts * sizeof(double);
    // + two constant rows (1 and NaN) for the bulk stores + the group summaries
    return kOffRecsFlux + (size_t)pv_tile * rec_bytes + queue_bytes(pv_tile * gpc) + 2 * kWarpPts * sizeof(float) +
           (size_t)gpc * sizeof(GroupInfo);
}
static_assert(kOffRecs32 % 16 == 0 && kOffRecs32Packed % 16 == 0 && kOffRecsFlux % 16 == 0,
              "shared-memory regions must stay 16-byte aligned");

// 128-time groups per CTA of the FP32 kernels.  A function of npt only, so
// the adjoint's summation order for a pv never depends on the other pvs in
// the launch: between 1 and 16 groups per warp, about one eighth of the
// point range per CTA.
int groups_per_cta(int npt) {
    const int ntiles = (npt + kPtTile - 1) / kPtTile;
    int t = ntiles / 8;
    t = t < 1 ? 1 : (t > 16 ? 16 : t);
    return t * (kBlock / 32);
}

int pv_tile_for(int rec_bytes) {
    int t = kSmemTarget / rec_bytes;
    if (t < 1) t = 1;
    if (t > kMaxPvTile) t = kMaxPvTile;
    return t;
}

// Groups per CTA and pvs per CTA of the FP64 kernels.  An SM's FP64 work is what its CTAs hold, so
// the launch is cut until there are 24 CTAs per SM, the groups first (at most 8: the adjoint's
// chunk), then the pvs.  Measured at 1, 4, 16, 32 CTAs per SM: 512 pvs x 10,007 times 244, 135, 107, 103
// us (adjoint 376, 215, 170, 163), 200 x 5,000 with 10 sub-exposures 389, 167, 128, 120.
void split64(const rr_ctx* c, int ngroups, int npv, int& gpc, int& pv_tile) {
    const long long want = 24LL * c->num_sms;
    auto ctas = [&] { return (long long)((ngroups + gpc - 1) / gpc) * ((npv + pv_tile - 1) / pv_tile); };
    gpc = kChunk64;
    while (gpc > 1 && ctas() < want) gpc >>= 1;
    while (pv_tile > 1 && ctas() < want) pv_tile = (pv_tile + 1) >> 1;
}

// The same for the FP32 kernels (gpc, pv_tile: the uncut launch's, kept from 3 CTAs per SM on): an
// ensemble whose vectors transit together, or a few vectors, left most SMs without a CTA.  Tiles of more
// than 8 pvs are halved (an item per warp where every pv of 8 transits; tiles of 4 were slower; 9 to 15 pvs become
// 5 to 8), and a CTA takes parts of the chunk (a multiple of 8 groups: a half, a quarter, an eighth, single groups),
// the forward kernel's groups first, the adjoint's pvs first (its CTAs carry sums per (pv, group), and the finish
// kernel more partial sums when the chunk is cut).  Measured, flux and adjoint: 16 pvs x 2,000 times 28.8 -> 11.8 and
// 40.2 -> 13.9 us; 200 x 3,001 40.8 -> 12.8, 64.0 -> 19.4; 100 x 4,407 with 10 sub-exposures 69.1 ->
// 13.5, 92.2 -> 17.5; 3 passbands, 256 x 9,001, adjoint 93.8 -> 35.2; prior populations 1,024 x 5,000
// 24.9 -> 18.3, 33.1 -> 28.3.  With 6 CTAs per SM 1,024 x 5,000 takes 21.2 and 32.8, and tables staged
// per CTA (256 pvs x 8 channels) 15.4 -> 18.3 from 4 on.  The price is the CTAs' own set-up where other streams
// fill the GPU anyway (light curves on 8 to 12 streams at once, a call: 16 x 2,000 3.0 -> 1.4 us, 200 x 3,001 5.0 ->
// 6.1, 500 x 5,000 8.3 -> 10.7, 64 x 20,000 3.7 -> 5.9): the server launches whole chunks (rr_server.cu).
void split32(const rr_ctx* c, int ngroups, int npv, bool adjoint, int& gpc, int& pv_tile) {
    constexpr int min_tile = 8;
    const long long want = 3LL * c->num_sms;
    auto ctas = [&] { return (long long)((ngroups + gpc - 1) / gpc) * ((npv + pv_tile - 1) / pv_tile); };
    auto cut_tile = [&] { while (pv_tile > min_tile && ctas() < want) pv_tile = (pv_tile + 1) >> 1; };
    const int chunk = gpc;
    if (adjoint) cut_tile();
    while (gpc > 1 && ctas() < want) gpc = gpc * 8 > chunk ? gpc >> 1 : 1;
    cut_tile();
}

// Failure-detection self-test: one bounded wait that nothing completes (see
// rr_selftest_wait); the expiry is recorded in the error word like any other.
__global__ void rr_selftest_kernel(int which, int* err) {
    __shared__ uint64_t bar;
    __shared__ int slot[1];
    __shared__ float4 slot_c[1];
    if (which == 0) {
        if (threadIdx.x != 0) return;
        mbar_init(&bar, 1);
        mbar_expect_tx(&bar, 16);   // this thread arrives; the 16 bytes of transaction never come
        if (!mbar_wait_bounded(&bar, 0)) atomicExch(err, kErrBarrierTimeout);
        return;
    }
    // a claimed slot whose producer never publishes it; the whole warp takes part
    // (the claim wait ends in a warp shuffle)
    if (threadIdx.x == 0) slot[0] = -1;
    __syncwarp();
    ItemQueue q;
    q.c = slot_c;
    q.gi = slot;
    if (queue_key(q, 0) < 0 && threadIdx.x == 0) atomicExch(err, kErrQueueTimeout);
}

cudaError_t launch_selftest(rr_ctx* c, int which, cudaStream_t s) {
    rr_selftest_kernel<<<1, 32, 0, s>>>(which, c->d_err);
    c->launches++;
    return cudaGetLastError();
}

// Warps of a flux CTA that take the 128-time groups before any item.  With
// one sample per time the items are light: two warps keep the output stream
// going while six evaluate the transits beside it (population workload: flux
// kernel 80.8 -> 75.1 us).  With supersampling the items dominate and every
// warp streams its groups first (heterogeneous workload: 835 -> 792 us).
constexpr int kStreamWarpsSS1 = 2;

// The cut of one forward launch.
struct FluxCut {
    int gpc, pv_tile, ngroups, per_pv;   // groups and pvs per CTA, groups, staged bytes per pv
    bool stage_rows;   // FP32 kernel with several passbands: headers and rows of the tile in shared memory (the rows of
                       // many passbands do not stay in L1); one passband, the adjoint's record layout (rows
                       // 3 + nldc times larger) and the FP64 kernel: headers only, rows through L1/L2
    bool q1;           // FP64: groups of 32 times
    bool uncut;        // FP32: several whole chunks (they may be launched heaviest first)
};

static FluxCut flux_cut(const rr_ctx* c, const RecLayout& L, int npv, int npt, bool grad_layout) {
    const bool f64 = c->cfg.precision == RR_PREC_FP64;
    FluxCut k;
    k.stage_rows = !f64 && c->cfg.npb > 1 && !grad_layout;
    k.per_pv = k.stage_rows ? L.head_bytes + L.rows_bytes : L.head_bytes;
    k.pv_tile = pv_tile_for(k.per_pv);
    k.gpc = groups_per_cta(npt);
    k.ngroups = (npt + kWarpPts - 1) / kWarpPts;
    // FP64, few (pv, group) pairs: groups of 32 times, so that an item is one pass of its warp
    // (measured: 1 pv x 2,000 times 24.0 -> 13.8 us, 64 x 3,000 33.5 -> 29.4; 512 x 10,007 100 -> 96, but 200 x 5,000
    // with 10 sub-exposures 127 -> 197: the candidates of 128 times fill a warp's passes better)
    k.q1 = f64 && (long long)npv * k.ngroups < 16LL * c->num_sms;
    if (k.q1) k.ngroups = (npt + 31) / 32;
    if (f64) split64(c, k.ngroups, npv, k.gpc, k.pv_tile);
    else if (!c->shared_gpu) split32(c, k.ngroups, npv, false, k.gpc, k.pv_tile);
    k.uncut = !f64 && k.gpc == groups_per_cta(npt) && k.ngroups > k.gpc;
    return k;
}

bool flux_ordered(const rr_ctx* c, const PbParams& pbp, int npv, int npt, bool grad_layout) {
    if (c->cfg.precision == RR_PREC_FP64 || !mixed_sampling(pbp)) return false;
    return flux_cut(c, make_layout<float>(c->cfg.npb, c->cfg.ng, c->nldc, grad_layout), npv, npt, grad_layout).uncut;
}

cudaError_t launch_flux(rr_ctx* c, const double* times, const int32_t* pb_index, const void* pts_dt,
                        const void* pts_pb, const void* pts_grp, const void* pts_ord, int npt, int npv,
                        const PbParams& pbp, const void* records,
                        void* flux, int32_t* pv_status, bool grad_layout, cudaStream_t s) {
    const bool f64 = c->cfg.precision == RR_PREC_FP64;
    RecLayout L = f64 ? make_layout<double>(c->cfg.npb, c->cfg.ng, c->nldc, grad_layout)
                      : make_layout<float>(c->cfg.npb, c->cfg.ng, c->nldc, grad_layout);
    const FluxCut k = flux_cut(c, L, npv, npt, grad_layout);
    const int pv_tile = k.pv_tile, gpc = k.gpc, ngroups = k.ngroups;
    if (!k.uncut || !mixed_sampling(pbp)) pts_ord = nullptr;
    const size_t smem = flux_smem(pv_tile, k.per_pv, f64, gpc);
    const char* rowsg = (const char*)records + rows_offset(L, npv);
    const int npvt = (npv + pv_tile - 1) / pv_tile;
    const dim3 grid = point_grid(f64, npvt, (ngroups + gpc - 1) / gpc);
    if (smem > kMaxSmem || grid.x == 0) return cudaErrorInvalidConfiguration;
    bool ss1 = true;
    for (int pb = 0; pb < pbp.npb; ++pb) ss1 = ss1 && pbp.ss[pb] == 1;
    cudaError_t e;
    if (f64) {
        auto kern = k.q1 ? (ss1 ? rr_flux_fp64_kernel<true, 1> : rr_flux_fp64_kernel<false, 1>)
                       : (ss1 ? rr_flux_fp64_kernel<true, 4> : rr_flux_fp64_kernel<false, 4>);
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        const int bulk = npt % 2 == 0 && ((uintptr_t)flux & 15u) == 0 && in_device_memory(flux);
        // lanes per candidate that add its samples: a function of the sub-exposures alone
        const int ssmax = *std::max_element(pbp.ss, pbp.ss + pbp.npb);
        const int sum_shift = ssmax < 4 ? 0 : (ssmax < 16 ? 1 : (ssmax < 64 ? 2 : 3));
        kern<<<grid, kBlock64, smem, s>>>(times, pb_index, npt, npv, pbp, L, pv_tile, gpc, (const char*)records, rowsg,
                                          (double*)flux, pv_status, bulk, sum_shift,
                                          mixed_sampling(pbp) ? 0.0f : 1.0f / (float)pbp.ss[0], c->d_err);
    } else {
        auto kern = c->counting
                        ? (k.stage_rows ? (ss1 ? rr_flux_mixed_kernel<true, true, true>
                                             : rr_flux_mixed_kernel<true, false, true>)
                                      : (ss1 ? rr_flux_mixed_kernel<false, true, true>
                                             : rr_flux_mixed_kernel<false, false, true>))
                        : (k.stage_rows ? (ss1 ? rr_flux_mixed_kernel<true, true, false>
                                             : rr_flux_mixed_kernel<true, false, false>)
                                      : (ss1 ? rr_flux_mixed_kernel<false, true, false>
                                             : rr_flux_mixed_kernel<false, false, false>));
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        // bit 0: 16-byte stores; bit 1: bulk stores of constant rows (flux in device memory)
        const int vec = (npt % 4 == 0) && (((uintptr_t)flux & 15u) == 0) ? (in_device_memory(flux) ? 3 : 1) : 0;
        kern<<<grid, kBlock, smem, s>>>(times, (const float2*)pts_dt, (const int32_t*)pts_pb,
                                        (const GroupInfo*)pts_grp, npt, npv, pbp, L,
                                        pv_tile, gpc, groups_per_cta(npt), (const char*)records, rowsg, (float*)flux,
                                        pv_status, vec,
                                        ss1 ? kStreamWarpsSS1 : (kBlock >> 5),
                                        c->d_counts ? c->d_counts + (size_t)RR_KERNEL_FLUX * RR_COUNT_KINDS : nullptr,
                                        (const int*)pts_ord, c->d_err);
    }
    c->launches++;
    return cudaGetLastError();
}

}  // namespace rr
