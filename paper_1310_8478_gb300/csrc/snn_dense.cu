// snn_dense.cu -- the dense synapse pass of the DPSNN-STDP step on GB300.
//
// In steps where a large part of the network fired, the first bracket of the
// step, [S4(t-1) S5(t-1) S1(t)] (paper Sec. 2, cycle steps 2.1 and 2.3-2.6,
// Table 2 "long term synaptic plasticity"), is done by one pass that streams
// every source row once: per synapse LTP(t-1) -> long-term update at a period
// end -> delivery + LTD(t), in the same per-synapse order as the event-driven
// kernels of snn_step.cu, so both give bit-identical results.
#include "snn_deliver.cuh"

namespace snn {

// ---------------------------------------------------------------------------
size_t ordered_smem_bytes(uint32_t npc, uint32_t block)
{
    return (size_t)kLut * 4 + (size_t)npc * 24 + kItems * 4 + (size_t)(block / 32) * 64 * 4;
}

size_t dense_smem_bytes(uint32_t npc, uint32_t block)
{
    const size_t warps = block / 32;
    return 2 * kLut * 4                       // LTP / LTD tables
           + (size_t)kSlots * npc * 4         // staged input
           + warps * 32 * 4 * 2               // per-warp bucket offsets, LTP amounts
           + (((size_t)kSlots * npc * 2 + 15) & ~size_t(15));  // packed target words
}

// Packed per-target word of the dense pass, one per staged neuron: bit 15 set
// when the neuron fired in the previous step (its incoming synapses owe LTP),
// bits 0..14 the depression an arrival now applies (LTD table at the lag since
// its last spike; 0 without STDP).  The host enables the dense pass only when
// every LTD amount fits 15 bits.
constexpr uint32_t kFiredLast = 0x8000u;
constexpr uint32_t kDepMask = 0x7fffu;

// One row of the dense pass: the lane takes 8 consecutive synapses per pass,
// with one 16-byte target load and two 16-byte weight and derivative loads.
// A chunk of 8 lies in one or two delay buckets almost always (buckets hold
// M / D synapses); the deliver flags (bit d of fbits: the source fired at
// t - d) and LTP amounts of its positions come from bit masks, and only a
// chunk spread over three or more buckets walks them position by position.
// kDeriv: the step closes a plasticity period (the long-term update runs
// between LTP and delivery) -- excitatory rows only.
constexpr int kPrefetchAhead = 1;   // segments of 256 synapses between a warp's loads and its prefetches

template <bool kExc, bool kDeriv>
__device__ __forceinline__ void dense_row_walk(const DevNet &n, int64_t base, int m, int D, float scale, uint32_t fbits,
                                               bool stdp, bool ltp_on, const int32_t *w_off, const int32_t *w_amt,
                                               int32_t *s_in, const uint16_t *s_x, int lane, int64_t next_base,
                                               bool next_exc)
{
    const uint4 *rt4 = reinterpret_cast<const uint4 *>(n.tgt16 + base);
    int4 *rw4 = reinterpret_cast<int4 *>(n.w + base);
    int4 *rs4 = reinterpret_cast<int4 *>(n.sd + base);
    // what the row needs at all: its chunks' loads go out before the bucket
    // search so that the search runs under their latency
    const bool row_w = kDeriv || fbits != 0;
    const bool row_sd = kExc && (kDeriv || ltp_on || (stdp && fbits != 0));
    const uint32_t staged = kSlots * n.npc;
    for (int c = lane; c * 8 < m; c += 32) {
        const int k0 = c * 8;
        // the warp's next 256-synapse segment (in this row or at the
        // start of its next row) goes to L2 while this chunk is processed: a
        // pipeline that costs no registers
        if (lane == 0) {
            const int ka = k0 + kPrefetchAhead * 256, mr = (m + 255) & ~255;
            if (ka < m) prefetch_segment(n, base + ka, row_w, row_sd);
            else if (next_base >= 0) prefetch_segment(n, next_base + (ka - mr), true, next_exc);
        }
        if (out_of_range(n, base + k0 + 8 <= n.S)) continue;
        const uint4 tv = rt4[c];
        int4 wa = make_int4(0, 0, 0, 0), wb = wa, sa = wa, sb = wa;
        if (row_w) {
            wa = rw4[2 * c];
            wb = rw4[2 * c + 1];
        }
        if (row_sd) {
            sa = rs4[2 * c];
            sb = rs4[2 * c + 1];
        }
        // bucket of k0 (first d with end > k0): delays are near uniform along
        // a row, so the interpolated guess is right or one off almost always
        int lo = min(D, 1 + (int)((float)k0 * scale));
        while (w_off[lo] <= k0) ++lo;         // bucket D ends at m > k0
        while (w_off[lo - 1] > k0) --lo;      // w_off[0] = 0 <= k0
        const int nv = min(8, m - k0);        // valid positions (the row's last chunk is short)
        const int e0 = w_off[lo];
        const int n0 = min(e0 - k0, nv);      // positions in bucket lo
        uint32_t fmask = ((fbits >> lo) & 1u) ? (1u << n0) - 1u : 0u;
        const int32_t a0 = kExc ? w_amt[lo] : 0;
        int32_t a1 = 0;
        int n1 = n0;                          // positions before n1 are in bucket lo or lo + 1
        if (n0 < nv && w_off[lo + 1] >= k0 + nv) {   // lo < D here: bucket D ends at m
            n1 = nv;
            fmask |= ((fbits >> (lo + 1)) & 1u) ? ((1u << nv) - 1u) & ~((1u << n0) - 1u) : 0u;
            if (kExc) a1 = w_amt[lo + 1];
        }
        int32_t am[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) am[u] = (u < n0) ? a0 : ((u < nv) ? a1 : 0);
        if (n1 < nv) {
            // three or more buckets (or an empty one) inside the chunk
            int d = lo, nb = e0;
            fmask = 0;
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int k = k0 + u;
                if (u < nv) {
                    while (k >= nb) nb = w_off[++d];
                    fmask |= ((fbits >> d) & 1u) << u;
                    am[u] = kExc ? w_amt[d] : 0;
                }
            }
        }
        const uint32_t tw[4] = {tv.x, tv.y, tv.z, tv.w};
        int32_t wv[8] = {wa.x, wa.y, wa.z, wa.w, wb.x, wb.y, wb.z, wb.w};
        if (!kExc) {
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const uint32_t v = (u & 1) ? (tw[u >> 1] >> 16) : (tw[u >> 1] & 0xffffu);
                if (out_of_range(n, v < staged)) continue;
                if ((fmask >> u) & 1u) atomicAdd(&s_in[v], wv[u]);
            }
            continue;
        }
        int32_t sv[8] = {sa.x, sa.y, sa.z, sa.w, sb.x, sb.y, sb.z, sb.w};
        bool sd_dirty = kDeriv;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const bool f = (fmask >> u) & 1u;
            const uint32_t v = (u & 1) ? (tw[u >> 1] >> 16) : (tw[u >> 1] & 0xffffu);
            if (out_of_range(n, v < staged)) continue;
            const uint32_t x = s_x[v];
            int32_t sdv = sv[u];
            if ((x & kFiredLast) && am[u]) {
                sdv += am[u];
                sd_dirty = true;
            }
            if (kDeriv && u < nv) {
                wv[u] = deriv_w(n, wv[u], sdv);
                sdv = deriv_sd(n, sdv);
            }
            if (f) {
                atomicAdd(&s_in[v], wv[u]);
                const int32_t dep = (int32_t)(x & kDepMask);
                sdv -= dep;
                sd_dirty |= dep != 0;
            }
            sv[u] = sdv;
        }
        if (sd_dirty) {
            rs4[2 * c] = make_int4(sv[0], sv[1], sv[2], sv[3]);
            rs4[2 * c + 1] = make_int4(sv[4], sv[5], sv[6], sv[7]);
        }
        if (kDeriv) {
            rw4[2 * c] = make_int4(wv[0], wv[1], wv[2], wv[3]);
            rw4[2 * c + 1] = make_int4(wv[4], wv[5], wv[6], wv[7]);
        }
    }
}

// The deliver flags of the 32 positions from q0 < m (bit i: the source fired
// d ms before t, d being the delay bucket of position q0 + i).
__device__ __forceinline__ uint32_t word_flags(int q0, int m, int D, float scale, uint32_t fbits, const int32_t *w_off)
{
    int d = min(D, 1 + (int)((float)q0 * scale));
    while (w_off[d] <= q0) ++d;           // bucket D ends at m > q0
    while (w_off[d - 1] > q0) --d;        // w_off[0] = 0 <= q0
    const int end = min(32, m - q0);
    uint32_t f = 0;
    for (int a = 0; a < end; ++d) {
        const int b = min(w_off[d] - q0, end);
        if ((fbits >> d) & 1u) f |= (0xffffffffu >> (32 - b)) & (0xffffffffu << a);   // a < 32, 0 < b <= 32
        a = b;
    }
    return f;
}

__device__ __forceinline__ void dense_body(const DevNet &n, const int *t_now, const Part &g)
{
    extern __shared__ int4 smem_i4[];
    const int t = *t_now;
    if (!dense_selected(n, t) || deferring(n, t)) return;
    const uint32_t npc = n.npc;
    const uint32_t nwarps = blockDim.x >> 5;
    int32_t *s_lutp = reinterpret_cast<int32_t *>(smem_i4);
    int32_t *s_lutm = s_lutp + kLut;
    int32_t *s_in = s_lutm + kLut;                              // [kSlots * npc]
    int32_t *s_off = s_in + kSlots * npc;                       // [nwarps][32] bucket end offsets
    int32_t *s_amt = s_off + nwarps * 32;                       // [nwarps][32] LTP amount
    uint16_t *s_x = reinterpret_cast<uint16_t *>(s_amt + nwarps * 32);   // [kSlots * npc] packed words
    __shared__ uint32_t s_col[kSlots];

    const bool stdp = !(n.flags & SNN_STDP_OFF);
    const bool deliver_on = !(n.flags & SNN_DELIVERY_OFF);
    const bool owed = n.ctr->ltp_pending == t - 1;
    const bool ltp_on = owed && stdp;
    const bool deriv_on = owed && n.deriv_period && (t % (int)n.deriv_period) == 0;
    const uint32_t chunks = (npc + n.dense_rows - 1) / n.dense_rows;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < kLut; i += blockDim.x) {
        s_lutp[i] = n.lut_p[i];
        s_lutm[i] = n.lut_m[i];
    }
    drive(n, t, part_tid(g), part_threads(g));
    int32_t *w_off = s_off + warp * 32;
    int32_t *w_amt = s_amt + warp * 32;
    const int D = (int)n.D;
    const uint32_t dmask = (2u << D) - 2u;            // buckets 1..D
    unsigned long long ev_all = 0, ev_exc = 0;
    // the grid is at most one wave of resident blocks; a block takes work
    // units (a column and a chunk of its rows) from a step-wide cursor
    __shared__ uint32_t s_unit;
    for (uint32_t unit = g.bid; unit < n.C * chunks;) {
        const uint32_t col = unit / chunks;
        const uint32_t r0 = (unit - col * chunks) * n.dense_rows;
        const uint32_t r1 = min(npc, r0 + n.dense_rows);
        if (threadIdx.x < kSlots) s_col[threadIdx.x] = (uint32_t)n.nbr[col * kSlotStride + threadIdx.x];
        // every warp's first row starts streaming into L2 while the block stages
        if (lane == 0 && r0 + warp < r1) {
            const int64_t b = row_base(n, col * npc + r0 + warp);
            for (int sgm = 0; sgm < kPrefetchAhead; ++sgm)
                prefetch_segment(n, b + sgm * 256, true, r0 + warp < n.ne);
        }
        __syncthreads();
        for (int sl = 0; sl < kSlots; ++sl) {
            const int32_t *ls = n.last_spike + (size_t)s_col[sl] * npc;
            uint16_t *x_row = s_x + sl * npc;
            int32_t *in_row = s_in + sl * npc;
            for (uint32_t loc = threadIdx.x; loc < npc; loc += blockDim.x) {
                const int lag = lag_of(t, ls[loc]);
                x_row[loc] = (uint16_t)((lag == 1 ? kFiredLast : 0u) | (stdp ? (uint32_t)s_lutm[lag] : 0u));
                in_row[loc] = 0;
            }
        }
        __syncthreads();
        // row metadata goes out one row ahead: the spike-history word and, in lane
        // d <= D, the end of delay bucket d
        uint2 hv_next = make_uint2(0u, 0u);
        int off_next = 0;
        if (r0 + warp < r1) {
            const uint32_t p = col * npc + r0 + warp;
            hv_next = n.hl[p];
            off_next = (lane <= D) ? (int)n.doff[(size_t)p * kDoffStride + lane] : 0;
        }
        for (uint32_t r = r0 + warp; r < r1; r += nwarps) {
            const uint32_t p = col * npc + r;
            const bool exc = r < n.ne;
            const uint2 hv = hv_next;
            const int hi = off_next;
            if (r + nwarps < r1) {
                hv_next = n.hl[p + nwarps];
                off_next = (lane <= D) ? (int)n.doff[(size_t)(p + nwarps) * kDoffStride + lane] : 0;
            }
            const uint32_t h = hv.x;                      // bit k: fired at t - 1 - k
            const uint32_t fbits = deliver_on ? (h << 1) & dmask : 0u;
            const int lo = __shfl_up_sync(0xffffffffu, hi, 1);
            const int m = __shfl_sync(0xffffffffu, hi, D);
            // lane d (1..D) prepares bucket d
            int len = 0;
            int32_t amt = 0;
            if (lane == 0) w_off[0] = 0;
            if (lane >= 1 && lane <= D) {
                len = hi - lo;
                w_off[lane] = hi;
                if (exc && ltp_on && len) {
                    const uint32_t recent = h & (0xffffffffu << lane);
                    amt = s_lutp[recent ? __ffs(recent) - 1 - lane : lag_of(t - 1 - lane, (int)hv.y)];
                }
                w_amt[lane] = amt;
            }
            const int delivered = ((fbits >> lane) & 1u) ? len : 0;
            const bool busy = fbits != 0 || __any_sync(0xffffffffu, amt != 0) || (exc && deriv_on);
            const int dl = __reduce_add_sync(0xffffffffu, delivered);
            if (lane == 0) {
                ev_all += (unsigned long long)dl;
                if (exc) ev_exc += (unsigned long long)dl;
            }
            __syncwarp();
            if (!exc && n.D_inh == 1) {
                // inhibitory row of a generated net: one bucket (delay 1), one
                // weight, nothing plastic
                if (fbits & 2u) {
                    const int64_t base = row_base(n, p);
                    const uint4 *rt4 = reinterpret_cast<const uint4 *>(n.tgt16 + base);
                    const int64_t nbase = r + nwarps < r1 ? row_base(n, p + nwarps) : -1;
                    for (int c = lane; c * 8 < m; c += 32) {
                        if (lane == 0) {        // next segment of targets, as in the row walk
                            const int ka = c * 8 + 256, mr = (m + 255) & ~255;
                            if (ka < m) prefetch_segment(n, base + ka, false, false);
                            else if (nbase >= 0) prefetch_segment(n, nbase + (ka - mr), false, false);
                        }
                        if (out_of_range(n, base + c * 8 + 8 <= n.S)) continue;
                        const uint4 tv = rt4[c];
                        const int nv = min(8, m - c * 8);
                        const uint32_t tw[4] = {tv.x, tv.y, tv.z, tv.w};
#pragma unroll
                        for (int u = 0; u < 8; ++u) {
                            const uint32_t v = (u & 1) ? (tw[u >> 1] >> 16) : (tw[u >> 1] & 0xffffu);
                            if (u < nv && !out_of_range(n, v < kSlots * npc)) atomicAdd(&s_in[v], n.w_inh);
                        }
                    }
                }
            } else if (busy) {
                const float scale = (float)D / (float)m;
                const int64_t base = row_base(n, p);     // a multiple of 8: rows are padded
                const int64_t nbase = r + nwarps < r1 ? row_base(n, p + nwarps) : -1;
                const bool nexc = r + nwarps < n.ne;
                if (!exc)
                    dense_row_walk<false, false>(n, base, m, D, scale, fbits, stdp, ltp_on, w_off, w_amt, s_in, s_x,
                                                 lane, nbase, nexc);
                else if (deriv_on)
                    dense_row_walk<true, true>(n, base, m, D, scale, fbits, stdp, ltp_on, w_off, w_amt, s_in, s_x,
                                               lane, nbase, nexc);
                else
                    dense_row_walk<true, false>(n, base, m, D, scale, fbits, stdp, ltp_on, w_off, w_amt, s_in, s_x,
                                                lane, nbase, nexc);
            }
            __syncwarp();
        }
        __syncthreads();
        for (int sl = 0; sl < kSlots; ++sl) {
            int32_t *dst = n.I + (size_t)s_col[sl] * npc;
            const int32_t *in_row = s_in + sl * npc;
            for (uint32_t loc = threadIdx.x; loc < npc; loc += blockDim.x) {
                const int32_t v = in_row[loc];
                if (v) red_add(&dst[loc], v);
            }
        }
        if (threadIdx.x == 0) s_unit = g.nblk + atomicAdd(&n.ctr->dense_cursor, 1u);
        __syncthreads();
        unit = s_unit;
    }
    if (lane != 0) ev_all = ev_exc = 0;
    const unsigned long long ba = block_sum(ev_all);
    const unsigned long long be = block_sum(ev_exc);
    if (threadIdx.x == 0) {
        if (ba) {
            atomicAdd(&n.ctr->e_all, ba);
            atomicAdd(&n.ctr->e_exc, be);
            atomicAdd(&n.ctr->dense_e_all, ba);
            atomicAdd(&n.ctr->dense_e_exc, be);
        }
        if (g.bid == 0) {
            // potentiation visits: every incoming excitatory synapse of the
            // neurons that fired at t - 1 (counted when those spikes closed)
            if (ltp_on) n.ctr->dense_l_exc += n.ctr->l_exc_last;
            n.ctr->dense_steps += 1;
            if (deriv_on) n.ctr->dense_deriv_steps += 1;
        }
    }
}

// ---------------------------------------------------------------------------
// A dense step whose STDP is left to the window's pass: targets and, on
// excitatory rows, weights -- no derivatives, no post-spike words.  Without
// them a thread needs 32 registers, so two blocks of 1024 threads reside per
// SM and their 64 warps hide the loads that the fused pass above prefetches
// (its bulk prefetches would cost a third of the instructions here).  The
// delay buckets are looked up once per 1024 synapses, each lane the flags of
// 32 positions, and not at all when the source fired in each of the last D
// steps; where some are due, the chunks of 8 that hold one are listed, so that
// all lanes have one (a third of the synapses due 0.68 ms, 0.75 with the lanes
// of the others idle; half 0.88 and 0.91).  Inside a chunk that has a due position the others add 0: a condition
// around each addition costs a branch and a reconvergence, several times the
// addition.  1.28 M neurons of 1125 synapses: 1.2 ms a step, 0.95 of the copy
// bandwidth (1.5 ms inside the fused pass's kernel with 32 warps, 2.9 ms with
// the STDP); 320 000: 0.34 ms, with the L1's shared-memory passes at 0.8.
// ---------------------------------------------------------------------------
size_t dense_light_smem_bytes(uint32_t npc, uint32_t block)
{
    return (size_t)kSlots * npc * 4            // staged input
           + (block / 32) * 32 * 4             // per-warp bucket offsets
           + (block / 32) * 128 * 2;           // per-warp chunks that are due
}

// 8 synapses of a row into the staged input; those outside fmask add 0
__device__ __forceinline__ void light_chunk(const DevNet &n, const uint4 *t4, const int4 *w4, bool exc, uint32_t fmask,
                                            uint32_t in0)
{
    if (out_of_range(n, (const uint16_t *)(t4 + 1) <= n.tgt16 + n.S)) return;
    const uint4 tv = *t4;
    int4 wa, wb;
    if (exc) {
        wa = w4[0];
        wb = w4[1];
    } else {
        wa = wb = make_int4(n.w_inh, n.w_inh, n.w_inh, n.w_inh);
    }
    const uint32_t tw[4] = {tv.x, tv.y, tv.z, tv.w};
    const int32_t wv[8] = {wa.x, wa.y, wa.z, wa.w, wb.x, wb.y, wb.z, wb.w};
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        const uint32_t v = (u & 1) ? (tw[u >> 1] >> 16) : (tw[u >> 1] & 0xffffu);
        if (out_of_range(n, v < kSlots * n.npc)) continue;
        red_shared(in0 + 4u * v, (fmask >> u) & 1u ? wv[u] : 0);
    }
}

// a row whose buckets are all due
__device__ __forceinline__ void light_row(const DevNet &n, int64_t base, bool exc, uint32_t in0, int lane)
{
    const int m = (int)n.canon_m;
    const uint4 *t4 = reinterpret_cast<const uint4 *>(n.tgt16 + base) + lane;
    const int4 *w4 = reinterpret_cast<const int4 *>(n.w + base) + 2 * lane;
    for (int left = m - 8 * lane; left > 0; left -= 256, t4 += 32, w4 += 64)
        light_chunk(n, t4, w4, exc, left >= 8 ? 0xffu : (1u << left) - 1u, in0);
}

// A row with some buckets due: its chunks of 8 synapses that hold a due one
// are listed first, so that every lane has one (a due bucket of 56 synapses is
// 7 of a row's 141 chunks).
__device__ __forceinline__ void light_row_part(const DevNet &n, int64_t base, bool exc, uint32_t fbits,
                                               const int32_t *w_off, uint16_t *w_list, uint32_t in0, int lane)
{
    const int D = (int)n.D, m = (int)n.canon_m;
    const float scale = (float)D / (float)m;
    for (int s = 0; s < m; s += 1024) {
        const int q0 = s + 32 * lane;
        const uint32_t flags = q0 < m ? word_flags(q0, m, D, scale, fbits, w_off) : 0u;
        const uint32_t any = ((flags & 0xffu) ? 1u : 0u) | ((flags & 0xff00u) ? 2u : 0u) | ((flags & 0xff0000u) ? 4u : 0u) |
                             (flags >> 24 ? 8u : 0u);
        const uint32_t own = __popc(any);
        const uint32_t b0 = __ballot_sync(0xffffffffu, own & 1u), b1 = __ballot_sync(0xffffffffu, own & 2u),
                       b2 = __ballot_sync(0xffffffffu, own & 4u), lt = lanemask_lt();
        uint32_t at = __popc(b0 & lt) + 2 * __popc(b1 & lt) + 4 * __popc(b2 & lt);
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if ((any >> j) & 1u) w_list[at++] = (uint16_t)((4 * lane + j) << 8 | ((flags >> (8 * j)) & 0xffu));
        __syncwarp();
        const uint32_t count = __popc(b0) + 2 * __popc(b1) + 4 * __popc(b2);
        for (uint32_t i = lane; i < count; i += 32) {
            const uint32_t it = w_list[i], c = (uint32_t)s / 8u + (it >> 8);
            light_chunk(n, reinterpret_cast<const uint4 *>(n.tgt16 + base) + c, reinterpret_cast<const int4 *>(n.w + base) + 2 * c,
                        exc, it & 0xffu, in0);
        }
        __syncwarp();
    }
}

__device__ __forceinline__ void dense_light_body(const DevNet &n, const int *t_now, const Part &g)
{
    extern __shared__ int4 smem_i4[];
    __shared__ uint32_t s_col[kSlots];
    __shared__ uint32_t s_unit;
    const int t = *t_now;
    if (!deferring(n, t) || !dense_selected(n, t)) return;
    const uint32_t npc = n.npc, nwarps = blockDim.x >> 5;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, D = (int)n.D;
    int32_t *s_in = reinterpret_cast<int32_t *>(smem_i4);       // [kSlots * npc]
    int32_t *w_off = s_in + kSlots * npc + warp * 32;           // bucket end offsets
    uint16_t *w_list = reinterpret_cast<uint16_t *>(s_in + kSlots * npc + nwarps * 32) + warp * 128;
    const uint32_t in0 = (uint32_t)__cvta_generic_to_shared(s_in);
    const uint32_t chunks = (npc + n.dense_rows - 1) / n.dense_rows;
    const uint32_t dmask = (2u << D) - 2u;
    drive(n, t, part_tid(g), part_threads(g));
    unsigned long long ev_all = 0, ev_exc = 0;
    for (uint32_t unit = g.bid; unit < n.C * chunks;) {
        const uint32_t col = unit / chunks;
        const uint32_t r0 = (unit - col * chunks) * n.dense_rows;
        const uint32_t r1 = min(npc, r0 + n.dense_rows);
        if (threadIdx.x < kSlots) s_col[threadIdx.x] = (uint32_t)n.nbr[col * kSlotStride + threadIdx.x];
        for (uint32_t k = threadIdx.x; k < kSlots * npc; k += blockDim.x) s_in[k] = 0;
        __syncthreads();
        for (uint32_t r = r0 + warp; r < r1; r += nwarps) {
            const uint32_t p = col * npc + r;
            const bool exc = r < n.ne;
            const uint32_t due = exc ? dmask : 2u;         // inhibitory rows: delay 1 alone
            const uint32_t fbits = (n.hl[p].x << 1) & due;
            if (!fbits) continue;
            int events = (int)n.canon_m;
            if (fbits != due) {
                const int hi = lane <= D ? (int)n.doff[(size_t)p * kDoffStride + lane] : 0;
                const int lo = __shfl_up_sync(0xffffffffu, hi, 1);
                __syncwarp();
                w_off[lane] = hi;                          // lane d: end of bucket d, lane 0: 0
                events = __reduce_add_sync(0xffffffffu, (lane && ((fbits >> lane) & 1u)) ? hi - lo : 0);
                __syncwarp();
            }
            if (lane == 0) {
                ev_all += (unsigned long long)events;
                if (exc) ev_exc += (unsigned long long)events;
            }
            if (fbits == due) light_row(n, row_base(n, p), exc, in0, lane);
            else light_row_part(n, row_base(n, p), exc, fbits, w_off, w_list, in0, lane);
        }
        __syncthreads();
        for (int sl = 0; sl < kSlots; ++sl) {
            int32_t *dst = n.I + (size_t)s_col[sl] * npc;
            const int32_t *in_row = s_in + sl * npc;
            for (uint32_t loc = threadIdx.x; loc < npc; loc += blockDim.x) {
                const int32_t v = in_row[loc];
                if (v) red_add(&dst[loc], v);
            }
        }
        if (threadIdx.x == 0) s_unit = g.nblk + atomicAdd(&n.ctr->dense_cursor, 1u);
        __syncthreads();
        unit = s_unit;
        __syncthreads();
    }
    if (lane != 0) ev_all = ev_exc = 0;
    const unsigned long long ba = block_sum(ev_all);
    const unsigned long long be = block_sum(ev_exc);
    if (threadIdx.x == 0) {
        if (ba) {
            atomicAdd(&n.ctr->e_all, ba);
            atomicAdd(&n.ctr->e_exc, be);
            atomicAdd(&n.ctr->dense_e_all, ba);
            atomicAdd(&n.ctr->dense_e_exc, be);
        }
        if (g.bid == 0) {
            n.ctr->dense_l_exc += n.ctr->l_exc_last;       // visits that the window's pass makes
            n.ctr->dense_steps += 1;
        }
    }
}

// the dense pass of nets whose deferred dense steps have no launch of their own
__device__ __forceinline__ void dense_any(const DevNet &n, const int *t_now, const Part &g)
{
    if (n.light_in_dense && deferring(n, *t_now)) dense_light_body(n, t_now, g);
    else dense_body(n, t_now, g);
}

__global__ void __launch_bounds__(1024) k_dense(DevNet n, const int *t_now) { dense_any(n, t_now, whole_grid()); }

__global__ void __launch_bounds__(kOrderedMaxBlock, 2) k_deliver_ordered(DevNet n, const int *t_now)
{
    deliver_ordered(n, t_now, whole_grid());
}

__global__ void __launch_bounds__(kOrderedMaxBlock, 2) k_deliver_ordered_b(BatchLaunch b)
{
    const BatchBlock x = batch_block(b);
    const DevNet n = b.nets[x.net];
    deliver_ordered(n, x.t_now, x.part);
}

// Both in one launch, for shapes that give them the same blocks (a step takes
// one of them; the other alone would be a launch that returns, 3 us).
__global__ void __launch_bounds__(kOrderedMaxBlock, 2) k_deliver_dense(DevNet n, const int *t_now)
{
    if (ordered_selected(n, *t_now)) deliver_ordered(n, t_now, whole_grid());
    else dense_any(n, t_now, whole_grid());
}

__global__ void __launch_bounds__(1024) k_dense_b(BatchLaunch b)
{
    const BatchBlock x = batch_block(b);
    const DevNet n = b.nets[x.net];
    dense_any(n, x.t_now, x.part);
}

__global__ void __launch_bounds__(kDenseLightBlock, 2) k_dense_light(DevNet n, const int *t_now)
{
    dense_light_body(n, t_now, whole_grid());
}

__global__ void __launch_bounds__(kDenseLightBlock, 2) k_dense_light_b(BatchLaunch b)
{
    const BatchBlock x = batch_block(b);
    const DevNet n = b.nets[x.net];
    dense_light_body(n, x.t_now, x.part);
}

}  // namespace snn
