// snn_deliver.cuh -- the column-ordered event-driven delivery of a step (S1 of
// compact nets, see snn_step.cu), for the kernels that run it alone and beside
// the dense pass.
#pragma once

#include "snn_internal.cuh"

namespace snn {

// The column-ordered delivery.  Per column a block lists the inhibitory rows
// that fired at t - 1 and the due (row, delay) items, walks both with all of
// its threads (walk_inhibitory, walk_items) and flushes the column's own input
// with one coalesced reduction per touched neuron; a target on another column
// is a reduction into its input and, with kStdp, a gather of its last spike,
// both on the band of columns in flight, which stays in L2.  The next column is
// claimed two columns ahead, and its histories and last spikes are copied into
// shared memory while this one is walked.  Bound by latency and instruction
// issue (half of it) at 64 registers and two blocks of 512 threads per SM; with
// three at 40 registers it spilled (busy 32x32 net, before the walk by chunks:
// 142 us per step, 129 with two), and five of 256 threads left a wave of 1024
// columns two thirds full.
// Tried for steps without depression: all 13 columns' input in shared memory
// in the deferred dense step's kernel, which needs no distinction of targets
// but flushes 13 columns (70 us at any rate on the 32x32 net).
template <bool kStdp>
__device__ __forceinline__ void deliver_columns(const DevNet &n, int t, const Part &g)
{
    extern __shared__ int4 smem_i4[];
    __shared__ uint32_t s_col[2][kSlotStride], s_next[2];
    __shared__ unsigned s_items_n, s_inh_n;
    const uint32_t npc = n.npc, ne = n.ne;
    int32_t *const s_lut = reinterpret_cast<int32_t *>(smem_i4);
    int32_t *const s_in = s_lut + kLut;                                   // [npc] input of the column
    uint32_t *const s_hist = reinterpret_cast<uint32_t *>(s_in + npc);    // [2][npc] bit k: fired at t - 1 - k
    int32_t *const s_last = reinterpret_cast<int32_t *>(s_hist + 2 * npc);   // [2][npc] last spikes
    uint32_t *const s_inh = reinterpret_cast<uint32_t *>(s_last + 2 * npc);  // [npc]
    uint32_t *const s_items = s_inh + npc;                                // [kItems]
    int32_t *const w_ab = reinterpret_cast<int32_t *>(s_items + kItems) + (threadIdx.x >> 5) * 64;
    const int lane = threadIdx.x & 31;
    const uint32_t dmask = (2u << n.D) - 2u;
    const int64_t col_syn = (int64_t)npc * n.uniform_m;
    const int lg = bucket_lanes(n);
    // buckets of more than 12 synapses, without depression of more than 6, go
    // chunk by chunk: 32x32 net with buckets of 15, a tenth of the synapses due,
    // 185 -> 88 us, with depression 169 -> 160; 64x32 with 56, with depression,
    // onset 6.6 -> 6.4 ms; 64x64 with 10 100 -> 93 us, with depression 1 to 4 %
    // slower
    const bool chunked = !n.tile && lg >= (kStdp ? 5 : 4);
    if (kStdp)
        for (int i = threadIdx.x; i < kLut; i += blockDim.x) s_lut[i] = n.lut_m[i];
    drive(n, t, part_tid(g), part_threads(g));
    if (n.flags & SNN_DELIVERY_OFF) return;
    auto copy = [&](uint32_t col, int b) {
        if (threadIdx.x < kSlotStride) copy4_async(&s_col[b][threadIdx.x], n.nbr + col * kSlotStride + threadIdx.x);
        for (uint32_t i = threadIdx.x; i < npc; i += blockDim.x) {
            copy4_async(s_hist + b * npc + i, &n.hl[(size_t)col * npc + i].x);
            if (kStdp) copy4_async(s_last + b * npc + i, n.last_spike + (size_t)col * npc + i);
        }
    };
    uint32_t col = g.bid;
    if (col < n.C) copy(col, 0);
    for (uint32_t i = threadIdx.x; i < npc; i += blockDim.x) s_in[i] = 0;
    if (threadIdx.x == 0) {
        s_next[0] = g.nblk + atomicAdd(&n.ctr->staged_cursor, 1u);
        s_items_n = s_inh_n = 0;
    }
    unsigned long long ev_all = 0, ev_exc = 0;
    for (int b = 0; col < n.C; b ^= 1) {
        wait_async();
        __syncthreads();
        const uint32_t next = s_next[b];
        uint32_t claimed = n.C;
        if (next < n.C) {
            copy(next, b ^ 1);
            if (threadIdx.x == 0) claimed = g.nblk + atomicAdd(&n.ctr->staged_cursor, 1u);
        }
        const uint32_t *hist = s_hist + b * npc, *cols = s_col[b];
        const int32_t *last = s_last + b * npc;
        const int64_t cbase = (int64_t)col * col_syn;                     // first synapse of the column (8-aligned)
        const uint16_t *tg = n.tgt16 + cbase;
        int32_t *const sd = n.sd + cbase;
        // slots that lead back to the column (rings of a small torus)
        const uint32_t local = __ballot_sync(0xffffffffu, lane < kSlots && cols[lane] == col);
        const bool mine = !n.tile || owned_column(n, col);                // inhibitory targets lie in the column
        if (mine) list_fired(blockDim.x, hist, ne, npc, 0, s_inh, &s_inh_n);
        // excitatory rows: all of them at once in a sparse step; where their
        // items do not fit the list, in ranges, halved until they do
        uint32_t range = ne;
        bool begun = false;
        for (uint32_t r0 = 0; r0 < ne;) {
            list_items(blockDim.x, hist, r0, min(ne, r0 + range), 0, dmask, s_items, &s_items_n);
            __syncthreads();
            const uint32_t items = s_items_n;
            if (items > kItems) {
                range = max(kItems / n.D, range / 2);
                __syncthreads();
                if (threadIdx.x == 0) s_items_n = 0;
                __syncthreads();
                continue;
            }
            unsigned seen = 0;                                            // a tile's events on its own columns
            unsigned walked;
            auto inhibitory = [&] {
                if (begun) return;
                walk_inhibitory(blockDim.x, n, s_inh, s_inh_n, tg, col_syn, (uint32_t)__cvta_generic_to_shared(s_in));
                if (threadIdx.x == 0) ev_all += (unsigned long long)s_inh_n * n.canon_m;
            };
            if (!chunked) {
                walked = walk_items(
                    blockDim.x, n, col, s_items, items, w_ab, lg, tg, n.w + cbase, col_syn, inhibitory,
                    [&](uint32_t v, int32_t w) -> int32_t {
                        const uint32_t slot = __umulhi(v, n.npc_recip), loc = v - slot * npc;
                        if (n.tile) {
                            if (!owned_column(n, cols[slot])) return kNever;  // another tile's target
                            ++seen;
                        }
                        if ((local >> slot) & 1u) {
                            atomicAdd(&s_in[loc], w);
                            return kStdp ? last[loc] : 0;
                        }
                        const uint32_t gid = cols[slot] * npc + loc;
                        red_add(&n.I[gid], w);
                        return kStdp ? n.last_spike[gid] : 0;
                    },
                    [&](int32_t x, int at) {
                        if (!kStdp) return;
                        const int32_t amount = s_lut[lag_of(t, x)];   // lag >= 1
                        if (amount) red_add(&sd[at], -amount);                // no load: most amounts are 0
                    });
            } else {
                const uint32_t in0 = (uint32_t)__cvta_generic_to_shared(s_in);
                const uint4 *t4 = reinterpret_cast<const uint4 *>(tg);
                const int4 *w4 = reinterpret_cast<const int4 *>(n.w + cbase);
                walked = walk_chunks(blockDim.x, n, col, s_items, items, w_ab, inhibitory, [&](uint32_t c, uint32_t mask) {
                    if (out_of_range(n, 8 * (int64_t)c + 8 <= col_syn)) return;
                    const uint4 tv = t4[c];
                    const int4 wa = w4[2 * c], wb = w4[2 * c + 1];
                    const uint32_t tw[4] = {tv.x, tv.y, tv.z, tv.w};
                    const int32_t wv[8] = {wa.x, wa.y, wa.z, wa.w, wb.x, wb.y, wb.z, wb.w};
                    int32_t x[8];
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        const uint32_t v = (u & 1) ? (tw[u >> 1] >> 16) : (tw[u >> 1] & 0xffffu);
                        x[u] = kNever;
                        if (out_of_range(n, v < kSlots * npc)) continue;
                        const uint32_t slot = __umulhi(v, n.npc_recip), loc = v - slot * npc;
                        const bool due = (mask >> u) & 1u, here = (local >> slot) & 1u;
                        red_shared(in0 + 4u * loc, due && here ? wv[u] : 0);      // adds 0 elsewhere: no branch
                        if (kStdp) x[u] = last[loc];
                        if (due && !here) {
                            const uint32_t gid = cols[slot] * npc + loc;
                            red_add(&n.I[gid], wv[u]);
                            if (kStdp) x[u] = n.last_spike[gid];
                        }
                    }
                    if (!kStdp) return;
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        const int32_t amount = s_lut[lag_of(t, x[u])];    // lag >= 1
                        if (amount && ((mask >> u) & 1u)) red_add(&sd[8 * c + u], -amount);   // no load: most are 0
                    }
                });
            }
            if (n.tile) {
                ev_all += seen;
                ev_exc += seen;
            } else if (lane == 0) {
                ev_all += walked;
                ev_exc += walked;
            }
            begun = true;
            r0 += range;
            __syncthreads();                                              // the items and the column's input are done
            if (threadIdx.x == 0) s_items_n = 0;
            if (r0 < ne) __syncthreads();
        }
        if (threadIdx.x == 0) {
            s_next[b ^ 1] = claimed;
            s_inh_n = 0;
        }
        int32_t *dst = n.I + (size_t)col * npc;
        for (uint32_t loc = threadIdx.x; loc < npc; loc += blockDim.x) {
            const int32_t x = s_in[loc];
            if (x) {
                red_add(&dst[loc], x);
                s_in[loc] = 0;
            }
        }
        col = next;
    }
    if (lane != 0 && !n.tile) ev_all = ev_exc = 0;
    const unsigned long long ba = block_sum(ev_all);
    const unsigned long long be = block_sum(ev_exc);
    if (threadIdx.x == 0 && ba) {
        atomicAdd(&n.ctr->e_all, ba);
        atomicAdd(&n.ctr->e_exc, be);
    }
}

__device__ __forceinline__ void deliver_ordered(const DevNet &n, const int *t_now, const Part &g)
{
    const int t = *t_now;
    if (!ordered_selected(n, t)) return;
    if (!(n.flags & SNN_STDP_OFF) && !deferring(n, t)) deliver_columns<true>(n, t, g);
    else deliver_columns<false>(n, t, g);
}

}  // namespace snn
