// snn_resident.cu -- many steps of a small net in one launch.
//
// The step kernels of snn_step.cu cost a net of a few columns its launches and
// a chain of first loads per kernel, and one block per column leaves most of
// the GPU idle.  Here a cooperative grid holds the whole net for a window of
// steps: `parts` blocks per column, each with the state of its slice of the
// column's neurons in shared memory for the whole window.  Per step a block
//   delivers the due delay buckets of its own neurons' rows (S1; targets in its
//     own column through shared memory, others by reductions into the step's
//     input array, of which there are two, by the step's parity),
//   waits for the other blocks (one grid barrier per step; none for a net of
//     one block),
//   updates its neurons (S2) and keeps the spikes as bits (S3).
// The STDP of the window is left to snn_window.cu's pass, so the delivery
// touches no derivative and needs no other block's spikes.  k_emit then writes
// what the step kernels would have: spike lists, raster, counters, clock.
//
// Bound by latency: per step a chain of a list, the buckets' bounds, their
// synapses, the reductions' way to L2 under the barrier (1.6 us alone) and the
// update.  us per step of long calls, emission and pass included (in brackets
// the step kernels before there were grids): one column of 1250 neurons 4.3
// (21), in FP64 5.7 (33), 8x8 torus of the paper's columns 9.8 (54), 16x16 23
// (62); of the last the grid itself takes 13 in the mean of the first 200 steps
// and 16.6 in their busiest 50.  Tried without gain: delivering the next step's
// arrivals from earlier spikes while the barrier fills, with three inputs in
// turn (8x8 10.1, one column 4.9).  The kernels need all of their 64 registers:
// one more value held through a step shows in the delivery (see resident_grid).
//
// Nets with target lists have no columns in this sense: a block owns a slice of
// all neurons, inhibitory rows are walked by delay like the others, and every
// target outside the slice is a reduction (a checkpointed net of 5000 neurons
// and 500000 synapses at 100 Hz, 49000 events per step: 10 us per step with its
// pass, 31 with the step kernels).
//
// A grid runs while its steps stay sparse: from a step with enough spikes for
// the dense pass on it stops, and the host goes on with the step kernels (nets
// with lists have no dense pass and run to the window's end).
#include <type_traits>

#include "snn_internal.cuh"

namespace snn {

constexpr uint32_t kEmitList = 4096;         // spikes listed at a time
constexpr uint32_t kResItems = 2048;         // pending (row, delay) items of a block
constexpr int kResFlight = 4;                // buckets of a group of lanes in flight
constexpr uint32_t kResThal = 512;           // thalamic events of a column drawn ahead
constexpr int kBarrierPolls = 1 << 22;       // about two seconds, then the kernel gives up

__host__ __device__ __forceinline__ uint32_t res_slice(uint32_t npc, uint32_t parts) { return (npc + parts - 1) / parts; }

size_t resident_smem_bytes(uint32_t npc, uint32_t parts, bool fp64, bool lists)
{
    const size_t ns = res_slice(npc, parts);
    return ns * (fp64 ? 16 : 8)                                // v, u
           + ns * 8                                            // spike train of the window
           + ns * 8                                            // history word, older spike
           + ns * 4                                            // inhibitory rows that fired
           + (lists ? ns : (size_t)npc) * 4                    // input of the column (of the own neurons)
           + kResItems * 4                                     // items
           + (size_t)(kResBlock / 32) * 64 * 4;                // per warp: a tile's buckets
}

// All blocks of the grid; false when one of them did not come within
// kBarrierPolls looks.  The arrival releases and the end acquires for the whole
// block (thread 0 behind and before a block barrier); the polls between are
// relaxed.  Arrivals count from 0; a test starts them below.
__device__ __forceinline__ bool grid_barrier(DevWindow *win, unsigned target, int *s_ok)
{
    __syncthreads();
    if (threadIdx.x == 0) {
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(&win->bar) : "memory");
        int left = kBarrierPolls;
        unsigned seen;
        do {
            asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(&win->bar) : "memory");
        } while ((int)(seen - target) < 0 && --left);
        *s_ok = left != 0;
        asm volatile("fence.acq_rel.gpu;" ::: "memory");
    }
    __syncthreads();
    return *s_ok != 0;
}

template <typename F, bool kLists>
__device__ __forceinline__ void resident_body(const DevNet &n, int p0, int steps)
{
    extern __shared__ int4 smem_i4[];
    __shared__ uint32_t s_col[kSlots];
    __shared__ unsigned s_items_n, s_inh_n;
    __shared__ int s_fired[2];                 // spikes of the step: exc, inh
    __shared__ int s_ok, s_stop;
    __shared__ std::conditional_t<kLists, uint32_t, uint16_t> s_thal[kResThal];
    DevWindow *const win = n.win;
    // not when the net's clock stands elsewhere (an earlier window of the call
    // stopped) or the first step is one for the dense pass
    const bool go = n.ctr->t_slot[p0 & 1] == p0 && !dense_selected(n, p0) && n.ctr->error == 0;
    if (blockIdx.x == 0 && threadIdx.x < kWinSlots) {
        win->cnt[threadIdx.x] = 0;          // added to behind the first barrier
        if (threadIdx.x == 0) {
            win->p0 = p0;
            win->p1 = p0 - 1;
            win->defer_from = kNoDefer;
            win->steps_done = 0;
        }
    }
    if (!go) return;
    const uint32_t npc = kLists ? n.N : n.npc, parts = kLists ? gridDim.x : n.res_parts;
    const uint32_t ns_max = res_slice(npc, parts);
    const uint32_t col = kLists ? 0u : blockIdx.x / parts, part = blockIdx.x - col * parts;
    const uint32_t lo = min(npc, part * ns_max), hi = min(npc, lo + ns_max), ns = hi - lo;   // own neurons
    const uint32_t g0 = col * npc + lo;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int kWarps = (int)kResBlock / 32;
    const int D = (int)n.D;
    const uint32_t dmask = (2u << D) - 2u;
    const bool more = gridDim.x > 1;

    F *const s_v = reinterpret_cast<F *>(smem_i4);
    F *const s_u = s_v + ns_max;
    unsigned long long *const s_train = reinterpret_cast<unsigned long long *>(s_u + ns_max);
    uint32_t *const s_hist = reinterpret_cast<uint32_t *>(s_train + ns_max);
    int32_t *const s_old = reinterpret_cast<int32_t *>(s_hist + ns_max);
    uint32_t *const s_inh = reinterpret_cast<uint32_t *>(s_old + ns_max);
    int32_t *const s_in = reinterpret_cast<int32_t *>(s_inh + ns_max);
    const uint32_t in_lo = kLists ? lo : 0u, in_n = kLists ? ns_max : npc;      // the neurons that s_in covers
    uint32_t *const s_items = reinterpret_cast<uint32_t *>(s_in + in_n);
    int32_t *const w_a = reinterpret_cast<int32_t *>(s_items + kResItems) + warp * 64;
    int32_t *const w_b = w_a + 32;
    F *const gv = sizeof(F) == 8 ? (F *)n.vd : (F *)n.v;
    F *const gu = sizeof(F) == 8 ? (F *)n.ud : (F *)n.u;

    for (uint32_t i = threadIdx.x; i < ns; i += kResBlock) {
        s_v[i] = gv[g0 + i];
        s_u[i] = gu[g0 + i];
        const uint2 h = n.hl[g0 + i];
        n.hl0[g0 + i] = h;
        s_hist[i] = h.x;
        s_old[i] = (int32_t)h.y;
        const int lag = h.x ? __ffs(h.x) : lag_of(p0, (int)h.y);       // of the latest spike before the window
        s_train[i] = (unsigned long long)lag << kWinBits;
    }
    // empty spike bits: a slice's first and last words are also its
    // neighbours', which set bits in them behind the first barrier
    for (uint32_t i = threadIdx.x; i < (uint32_t)steps * kWinSlots; i += kResBlock) {
        const uint32_t k = i / kWinSlots;
        for (uint32_t w = (g0 >> 5) + i % kWinSlots; ns && w <= (g0 + ns - 1) >> 5; w += kWinSlots)
            n.spk[(size_t)((p0 + k) & (kWinSlots - 1)) * n.spk_words + w] = 0;
    }
    for (uint32_t i = threadIdx.x; i < in_n; i += kResBlock) s_in[i] = 0;
    if (!kLists && threadIdx.x < kSlots) s_col[threadIdx.x] = (uint32_t)n.nbr[col * kSlotStride + threadIdx.x];
    // the window's thalamic events of the column (of all columns), drawn at once
    const uint32_t thal = kLists ? n.C * n.thal_per_col : n.thal_per_col;
    auto target = [&](int t, uint32_t e) -> uint32_t {
        if (!kLists) return draw_below(philox10(make_uint4((uint32_t)t, col, 1u, e), n.seed_lo, n.seed_hi).x, npc);
        const uint32_t c = e / n.thal_per_col;
        return c * n.npc +
               draw_below(philox10(make_uint4((uint32_t)t, c, 1u, e - c * n.thal_per_col), n.seed_lo, n.seed_hi).x, n.npc);
    };
    const bool drawn = (uint32_t)steps * thal <= kResThal;      // (no net has more than fit 32 bits: kResThalMax)
    if (drawn)
        for (uint32_t e = threadIdx.x; e < (uint32_t)steps * thal; e += kResBlock) {
            const uint32_t k = e / thal;
            s_thal[e] = (std::conditional_t<kLists, uint32_t, uint16_t>)target(p0 + (int)k, e - k * thal);
        }
    if (threadIdx.x == 0) {
        s_stop = 0;
        s_fired[0] = s_fired[1] = 0;
    }
    const int64_t cbase = kLists ? 0 : (int64_t)col * npc * n.uniform_m;   // first synapse of the column (8-aligned)
    const uint16_t *const tg = n.tgt16 + cbase;
    const int32_t *const wt = n.w + cbase;
    const uint4 *const t4 = reinterpret_cast<const uint4 *>(tg);
    const int64_t col_syn = kLists ? n.S : (int64_t)npc * n.uniform_m;
    const uint32_t row_chunks = n.uniform_m / 8u, m = n.canon_m, cpr = (m + 7u) / 8u;
    // own excitatory neurons: slice rows [0, e_hi) (lists: rows of both kinds)
    const uint32_t e_hi = kLists ? ns : lo < n.ne ? min(hi, n.ne) - lo : 0u;
    auto excitatory = [&](uint32_t loc) { return kLists ? loc % n.npc < n.ne : loc < n.ne; };
    const uint32_t dmask_i = (2u << n.D_inh) - 2u;
    // slots that lead back to the column (rings of a small torus)
    __syncthreads();
    uint32_t local = 0;
    for (int q = 0; q < kSlots && !kLists; ++q) local |= (s_col[q] == col ? 1u : 0u) << q;
    // lanes per bucket: the power of two that a mean bucket (M / D synapses)
    // fills best, 8 at least
    const uint32_t mean = kLists ? (uint32_t)(n.S / n.N) / (uint32_t)D : m / (uint32_t)D;
    const int lg = mean <= 6 ? 3 : mean <= 12 ? 4 : 5;
    const uint32_t gl = lane & ((1u << lg) - 1u), gi = lane >> lg, groups = 32u >> lg;
    // a net of one block has its whole input in shared memory, but for
    // external events and what a checkpoint left
    const bool input = more || (n.stim_t0 < p0 + steps && n.stim_t1 > p0);
    unsigned long long ev_all = 0, ev_exc = 0;
    int done = 0;
    bool ok = true;
    for (int k = 0; k < steps; ++k) {
        const int t = p0 + k;
        int32_t *const I = (k & 1) ? n.I2 : n.I;
        if (threadIdx.x == 0) {
            s_items_n = 0;
            s_inh_n = 0;
        }
        __syncthreads();                                // history, input and counters of the last step are in
        // ---- S1: rows that are due ------------------------------------------
        for (uint32_t i = e_hi + threadIdx.x; i - lane < ns; i += kResBlock) {
            const bool on = i < ns && (s_hist[i] & 1u);
            const uint32_t b = __ballot_sync(0xffffffffu, on);
            if (!b) continue;
            unsigned at = 0;
            if (lane == 0) at = atomicAdd(&s_inh_n, (unsigned)__popc(b));
            at = __shfl_sync(0xffffffffu, at, 0) + __popc(b & lanemask_lt());
            if (on) s_inh[at] = lo + i;
        }
        // thalamic drive of the own neurons, external events through the
        // step's input
        for (uint32_t e = threadIdx.x; e < thal; e += kResBlock) {
            const uint32_t loc = drawn ? s_thal[(uint32_t)k * thal + e] : target(t, e);
            if (loc >= lo && loc < hi) atomicAdd(&s_in[loc - in_lo], n.thal_amp);
        }
        if (t >= n.stim_t0 && t < n.stim_t1) {
            const int64_t a = n.stim_off[t - n.stim_t0], b = n.stim_off[t - n.stim_t0 + 1];
            for (int64_t e = a + blockIdx.x * kResBlock + threadIdx.x; e < b; e += (int64_t)gridDim.x * kResBlock)
                red_add(&I[n.stim_gid[e]], n.stim_q16[e]);
        }
        // excitatory rows: all of them at once in a sparse step; where their
        // items do not fit the list, in ranges that are sure to
        uint32_t range = max(e_hi, 1u);
        bool inh_left = true;
        for (uint32_t r0 = 0;;) {
            for (uint32_t i = r0 + threadIdx.x; i - lane < min(e_hi, r0 + range); i += kResBlock) {
                uint32_t f = i < min(e_hi, r0 + range) ? s_hist[i] << 1 : 0u;
                f &= !kLists || excitatory(lo + i) ? dmask : dmask_i;
                if (!__any_sync(0xffffffffu, f != 0)) continue;
                const uint32_t own = __popc(f);
                uint32_t incl = own;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += y;
                }
                unsigned at = 0;
                if (lane == 31) at = atomicAdd(&s_items_n, incl);
                at = __shfl_sync(0xffffffffu, at, 31) + incl - own;
                if (at + own > kResItems) continue;
                for (; f; f &= f - 1u) s_items[at++] = ((lo + i) << 5) | (uint32_t)(__ffs(f) - 1);
            }
            __syncthreads();
            const uint32_t items = s_items_n;
            if (items > kResItems) {
                range = kResItems / (uint32_t)D;
                __syncthreads();
                if (threadIdx.x == 0) s_items_n = 0;
                __syncthreads();
                continue;
            }
            // a warp's share of the items, 32 at a time: where their buckets lie
            const uint32_t share = (items + kWarps - 1) / kWarps;
            const uint32_t i_hi = min(items, (warp + 1) * share);
            uint32_t i_lo = warp * share;
            int a = 0, b = 0, first = 0;
            uint32_t row = 0;
            auto fetch = [&]() {
                a = b = 0;
                if (i_lo + lane < i_hi) {
                    const uint32_t it = s_items[i_lo + lane];
                    row = it >> 5;
                    const uint16_t *off = n.doff + (size_t)(col * npc + row) * kDoffStride + (it & 31u);
                    a = off[-1];
                    b = off[0];
                    if (kLists) first = (int)row_base(n, row);
                }
            };
            fetch();
            if (!kLists && inh_left) {
                // inhibitory rows that fired at t - 1: the whole row, one
                // weight, targets of the own column; all threads share them
                const uint32_t ninh = s_inh_n;
                for (uint32_t c = threadIdx.x; c < ninh * cpr; c += kResBlock) {
                    const uint32_t q = c / cpr, ci = c - q * cpr;
                    const uint32_t at = s_inh[q] * row_chunks + ci;
                    if (out_of_range(n, 8 * (int64_t)at + 8 <= col_syn)) continue;
                    const uint4 tv = t4[at];
                    const uint32_t nv = min(8u, m - 8u * ci);
                    const uint32_t tw[4] = {tv.x, tv.y, tv.z, tv.w};
                    const uint32_t in0 = (uint32_t)__cvta_generic_to_shared(s_in);
                    if (nv == 8) {
#pragma unroll
                        for (int u = 0; u < 8; ++u) {
                            const uint32_t v = (tw[u >> 1] >> (16 * (u & 1))) & 0xffffu;
                            if (!out_of_range(n, v < npc)) red_shared(in0 + 4u * v, n.w_inh);
                        }
                    } else {
                        for (uint32_t u = 0; u < nv; ++u) {
                            const uint32_t v = tg[8 * (int64_t)at + u];
                            if (!out_of_range(n, v < npc)) red_shared(in0 + 4u * v, n.w_inh);
                        }
                    }
                }
                if (threadIdx.x == 0) ev_all += (unsigned long long)ninh * m;
                inh_left = false;
            }
            while (i_lo < i_hi) {
                const int tile = (int)min(32u, i_hi - i_lo);
                const int events = __reduce_add_sync(0xffffffffu, b - a);
                const int plastic = kLists ? __reduce_add_sync(0xffffffffu, b > a && excitatory(row) ? b - a : 0) : events;
                if (lane == 0) {
                    ev_all += (unsigned long long)events;
                    ev_exc += (unsigned long long)plastic;
                }
                const int base = kLists ? first : (int)(row * n.uniform_m);
                w_a[lane] = base + a;
                w_b[lane] = base + b;
                __syncwarp();
                i_lo += 32;
                fetch();                                 // the next tile's buckets, under this tile's walk
                // a lane per synapse, a group of lanes per bucket, kResFlight
                // buckets of every group in flight
                for (int q0 = 0; q0 < tile; q0 += kResFlight * (int)groups) {
                    int at[kResFlight], end[kResFlight];
                    int left = 0;
#pragma unroll
                    for (int h = 0; h < kResFlight; ++h) {
                        const int q = q0 + h * (int)groups + (int)gi;
                        at[h] = q < tile ? w_a[q] + (int)gl : 0;
                        end[h] = q < tile ? w_b[q] : 0;
                        left |= at[h] < end[h];
                    }
                    while (__any_sync(0xffffffffu, left)) {
                        uint32_t v[kResFlight];
                        int32_t w[kResFlight];
                        left = 0;
#pragma unroll
                        for (int h = 0; h < kResFlight; ++h) {
                            v[h] = 0xffffffffu;
                            if (at[h] < end[h] && !out_of_range(n, at[h] >= 0 && at[h] < col_syn)) {
                                v[h] = kLists ? (uint32_t)n.tgt[at[h]] : tg[at[h]];
                                w[h] = wt[at[h]];
                            }
                            at[h] += 1 << lg;
                            left |= at[h] < end[h];
                        }
#pragma unroll
                        for (int h = 0; h < kResFlight; ++h) {
                            if (v[h] == 0xffffffffu || out_of_range(n, v[h] < (kLists ? n.N : kSlots * npc))) continue;
                            if (kLists) {
                                if (v[h] - lo < ns) atomicAdd(&s_in[v[h] - lo], w[h]);
                                else red_add(&I[v[h]], w[h]);
                                continue;
                            }
                            const uint32_t slot = __umulhi(v[h], n.npc_recip), loc = v[h] - slot * npc;
                            if ((local >> slot) & 1u) atomicAdd(&s_in[loc], w[h]);
                            else red_add(&I[s_col[slot] * npc + loc], w[h]);
                        }
                    }
                }
                __syncwarp();
            }
            __syncthreads();                             // the items are done, the input of the column is in
            r0 += range;
            if (r0 >= e_hi) break;
            if (threadIdx.x == 0) s_items_n = 0;
            __syncthreads();
        }
        if (!kLists && parts > 1) {                      // the column's other slices
            for (uint32_t i = threadIdx.x; i < npc; i += kResBlock) {
                if (i >= lo && i < hi) continue;
                const int32_t x = s_in[i];
                if (x) {
                    red_add(&I[col * npc + i], x);
                    s_in[i] = 0;
                }
            }
        }
        // the spikes of step k - 1 (all blocks add theirs before the barrier)
        if (threadIdx.x == 0 && k > 0) {
            atomicAdd(&win->cnt[k - 1], (unsigned long long)s_fired[0] | ((unsigned long long)s_fired[1] << 32));
            s_fired[0] = s_fired[1] = 0;
        }
        if (more) {
            if (!(ok = grid_barrier(win, (unsigned)(k + 1) * gridDim.x, &s_ok))) break;
        } else {
            __syncthreads();
        }
        if (threadIdx.x == 0 && k > 0) {
            const unsigned long long c = __ldcg(&win->cnt[k - 1]);
            s_stop = !kLists && (c & 0xffffffffull) + (c >> 32) >= n.dense_min_spikes;
        }
        // ---- S2, S3 of the own neurons: threads on word boundaries of the
        // spike bits, the words at the slice's ends shared with its neighbours
        uint32_t *const bits = n.spk + (size_t)(t & (kWinSlots - 1)) * n.spk_words;
        const uint32_t first = g0 & 31u;
        for (uint32_t i = threadIdx.x; i - lane < ns + first; i += kResBlock) {
            const bool own = i >= first && i - first < ns;
            const uint32_t q = i - first;
            bool fired = false;
            if (own) {
                const uint32_t loc = lo + q;
                int32_t iq = s_in[loc - in_lo];
                s_in[loc - in_lo] = 0;
                if (input || k == 0) {
                    iq += __ldcg(&I[g0 + q]);
                    I[g0 + q] = 0;
                }
                F v = s_v[q], u = s_u[q];
                fired = izhikevich_step(v, u, iq, excitatory(loc));
                s_v[q] = v;
                s_u[q] = u;
                const uint32_t h = s_hist[q];
                if (h & 0x80000000u) s_old[q] = t - 32;
                s_hist[q] = (h << 1) | (fired ? 1u : 0u);
                if (fired) {
                    n.last_spike[g0 + q] = t;
                    s_train[q] |= 1ull << k;
                }
            }
            const uint32_t word = __ballot_sync(0xffffffffu, fired);
            const uint32_t exc = __ballot_sync(0xffffffffu, fired && excitatory(lo + q));
            const uint32_t owned = __ballot_sync(0xffffffffu, own);
            if (lane == 0 && owned) {
                uint32_t *p = bits + ((g0 + q) >> 5);
                if (owned == 0xffffffffu) *p = word;
                else if (word) atomicOr(p, word);
                if (word) {
                    atomicAdd(&s_fired[0], __popc(exc));
                    atomicAdd(&s_fired[1], __popc(word & ~exc));
                }
            }
        }
        done = k + 1;
        __syncthreads();
        if (s_stop) break;
    }
    if (!ok && threadIdx.x == 0) atomicCAS(&n.ctr->error, 0, SNN_ETIMEOUT);
    for (uint32_t i = threadIdx.x; i < ns; i += kResBlock) {
        gv[g0 + i] = s_v[i];
        gu[g0 + i] = s_u[i];
        n.hl[g0 + i] = make_uint2(s_hist[i], (uint32_t)s_old[i]);
        n.train[g0 + i] = s_train[i];
    }
    if (threadIdx.x == 0 && done)
        atomicAdd(&win->cnt[done - 1], (unsigned long long)s_fired[0] | ((unsigned long long)s_fired[1] << 32));
    if (lane != 0) ev_all = ev_exc = 0;
    const unsigned long long ba = block_sum(ev_all), be = block_sum(ev_exc);
    if (threadIdx.x == 0) {
        if (ba) {
            atomicAdd(&n.ctr->e_all, ba);
            atomicAdd(&n.ctr->e_exc, be);
        }
        if (blockIdx.x == 0) win->steps_done = done;
    }
}

__global__ void __launch_bounds__(kResBlock, 2) k_resident_f32(DevNet n, int t0, int steps)
{
    resident_body<float, false>(n, t0, steps);
}

__global__ void __launch_bounds__(kResBlock, 2) k_resident_f64(DevNet n, int t0, int steps)
{
    resident_body<double, false>(n, t0, steps);
}

// nets with target lists (explicit ones, columns above 4096 neurons)
__global__ void __launch_bounds__(kResBlock, 2) k_resident_lists_f32(DevNet n, int t0, int steps)
{
    resident_body<float, true>(n, t0, steps);
}

__global__ void __launch_bounds__(kResBlock, 2) k_resident_lists_f64(DevNet n, int t0, int steps)
{
    resident_body<double, true>(n, t0, steps);
}

// spikes of word w of a step's bits by kind: exc | inh << 16
__device__ __forceinline__ uint32_t word_kinds(const DevNet &n, uint32_t w, uint32_t x)
{
    if (!x) return 0;
    const uint32_t all = __popc(x), loc = (w * 32u) % n.npc;
    uint32_t exc;
    if (loc + 32 <= n.ne) {
        exc = all;
    } else if (loc >= n.ne && loc + 32 <= n.npc) {
        exc = 0;
    } else {
        exc = 0;
        for (uint32_t f = x; f; f &= f - 1u) exc += (loc + __ffs(f) - 1) % n.npc < n.ne ? 1u : 0u;
    }
    return exc | ((all - exc) << 16);
}

// What the step kernels' compaction writes, from a resident window's spike
// bits: the blocks of a step (kEmitWords words of its bits each) list its
// spikes in ascending order into the raster and, in the last D steps, into the
// delay ring, and sum their in-degrees; the last block closes the window's
// steps (counters, offsets, clock).
__global__ void __launch_bounds__(kEmitBlock) k_emit(DevNet n)
{
    __shared__ uint32_t s_bits[kEmitWords];
    __shared__ uint32_t s_list[kEmitList];
    __shared__ uint32_t s_warp[kEmitBlock / 32];
    __shared__ unsigned s_ring[2];
    __shared__ unsigned long long s_cnt[kWinSlots];
    __shared__ bool s_last;
    DevWindow *const win = n.win;
    const int steps = win->steps_done, p0 = win->p0, k = blockIdx.y;
    DevCounters *const c = n.ctr;
    if (k >= steps) return;
    const int t = p0 + k;
    const uint32_t words = n.spk_words, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr uint32_t kWarps = kEmitBlock / 32;
    const uint32_t w_lo = blockIdx.x * kEmitWords, count_w = min(words - w_lo, kEmitWords);
    const uint32_t *bits = n.spk + (size_t)(t & (kWinSlots - 1)) * words;
    if (threadIdx.x < kWinSlots) s_cnt[threadIdx.x] = (int)threadIdx.x < steps ? win->cnt[threadIdx.x] : 0ull;
    if (threadIdx.x < 2) s_ring[threadIdx.x] = 0;
    const unsigned long long raster0 = c->raster_total;
    for (uint32_t w = threadIdx.x; w < kEmitWords; w += kEmitBlock) s_bits[w] = w < count_w ? bits[w_lo + w] : 0u;
    __syncthreads();
    // the step's spikes in the words of the blocks before this one
    uint32_t exc = 0, inh = 0;
    for (uint32_t w = threadIdx.x; w < w_lo; w += kEmitBlock) {
        const uint32_t kinds = word_kinds(n, w, bits[w]);
        exc += kinds & 0xffffu;
        inh += kinds >> 16;
    }
    exc = __reduce_add_sync(0xffffffffu, exc);
    inh = __reduce_add_sync(0xffffffffu, inh);
    if (lane == 0 && exc) atomicAdd(&s_ring[0], exc);
    if (lane == 0 && inh) atomicAdd(&s_ring[1], inh);
    __syncthreads();
    unsigned long long at = raster0 + s_ring[0] + s_ring[1];
    for (int q = 0; q < k; ++q) at += (s_cnt[q] & 0xffffffffull) + (s_cnt[q] >> 32);
    const bool listed = k + (int)n.D >= steps;                 // still in the ring after the window
    int32_t *const ring = n.ring_ids + (size_t)(t % (int)n.D) * n.N;
    unsigned long long indeg = 0;
    // 32 words per warp and pass: a list of at most kEmitList spikes in shared
    // memory, then a thread per spike
    static_assert(kEmitList >= kWarps * 32 * 8, "a quarter of a pass's neurons");
    for (uint32_t b = 0; b < count_w; b += kWarps * 32) {
        const uint32_t x0 = b + threadIdx.x < kEmitWords ? s_bits[b + threadIdx.x] : 0u;
        // a word's spikes in up to four rounds of 8 neurons, so that they fit
        const int rounds = __syncthreads_or(__popc(x0) > 8) ? 4 : 1;
        for (int r = 0; r < 4; r += 4 / rounds) {
            uint32_t x = rounds == 1 ? x0 : x0 & (0xffu << (8 * r));
            const uint32_t own = __popc(x);
            uint32_t incl = own;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= (uint32_t)o) incl += y;
            }
            if (lane == 31) s_warp[warp] = incl;
            __syncthreads();
            uint32_t before = 0, total = 0;
            for (uint32_t q = 0; q < kWarps; ++q) {
                if (q == warp) before = total;
                total += s_warp[q];
            }
            for (uint32_t q = before + incl - own; x; x &= x - 1u, ++q)
                s_list[q] = (w_lo + b + threadIdx.x) * 32 + __ffs(x) - 1;
            __syncthreads();
            for (uint32_t q = threadIdx.x; q - lane < total; q += kEmitBlock) {      // warp-uniform
                const uint32_t id = q < total ? s_list[q] : n.N;
                const bool in = id < n.N;
                if (in && at + q < n.raster_cap) n.raster_gid[at + q] = (int32_t)id;
                if (in) indeg += (unsigned long long)(n.rin_off[id + 1] - n.rin_off[id]);
                if (!listed) continue;
                // a position per warp and kind, any order inside a step
                const bool e = in && id % n.npc < n.ne;
                const uint32_t be = __ballot_sync(0xffffffffu, e), bi = __ballot_sync(0xffffffffu, in && !e);
                unsigned pe = 0, pi = 0;
                if (lane == 0) {
                    pe = atomicAdd(&s_ring[0], (unsigned)__popc(be));
                    pi = atomicAdd(&s_ring[1], (unsigned)__popc(bi));
                }
                pe = __shfl_sync(0xffffffffu, pe, 0) + __popc(be & lanemask_lt());
                pi = __shfl_sync(0xffffffffu, pi, 0) + __popc(bi & lanemask_lt());
                if (in) ring[e ? pe : n.N - 1 - pi] = (int32_t)id;
            }
            at += total;
            __syncthreads();
        }
    }
    const unsigned long long deg = block_sum(indeg);
    if (threadIdx.x == 0) {
        if (deg) atomicAdd(&c->l_exc, deg);
        if (deg && k == steps - 1) atomicAdd(&win->last_deg, deg);
        __threadfence();
        s_last = atomicAdd(&c->done_blocks, 1u) == (unsigned)steps * gridDim.x - 1;
    }
    __syncthreads();
    if (!s_last || threadIdx.x != 0) return;
    __threadfence();
    c->l_exc_last = __ldcg(&win->last_deg);
    win->last_deg = 0;
    unsigned long long rt = raster0, spikes = c->spikes, dropped = c->raster_dropped;
    for (int q = 0; q < steps; ++q) {
        const int tq = p0 + q, slot = tq % (int)n.D;
        const unsigned long long x = s_cnt[q], all = (x & 0xffffffffull) + (x >> 32);
        if (q + (int)n.D >= steps) {
            n.ring_cnt[2 * slot] = (int)(x & 0xffffffffull);
            n.ring_cnt[2 * slot + 1] = (int)(x >> 32);
        }
        spikes += all;
        const unsigned long long room = n.raster_cap > rt ? n.raster_cap - rt : 0ull;
        const unsigned long long kept = all < room ? all : room;
        if (kept < all) {
            if (dropped == 0) c->raster_first_drop_t = tq;
            dropped += all - kept;
        }
        rt += kept;
        if (n.raster_step_off) n.raster_step_off[tq + 1 - n.raster_t0] = (int64_t)rt;
    }
    c->spikes = spikes;
    c->raster_dropped = dropped;
    c->raster_total = rt;
    // as the step kernels leave them: the last step's spikes, the next one's none
    for (int q = 0; q < 8; ++q) c->step_cnt[q >> 2][q & 3] = 0;
    c->step_cnt[(p0 + steps - 1) & 1][0] = (int)(s_cnt[steps - 1] & 0xffffffffull);
    c->step_cnt[(p0 + steps - 1) & 1][1] = (int)(s_cnt[steps - 1] >> 32);
    c->l_exc_mark = __ldcg(&c->l_exc);
    c->ltp_pending = p0 + steps - 1;
    c->done_blocks = 0;
    c->t_slot[(p0 + steps) & 1] = p0 + steps;
    win->p1 = p0 + steps - 1;
    win->defer_from = p0;                 // all of the window's STDP
    win->bar = 0;
}

}  // namespace snn
