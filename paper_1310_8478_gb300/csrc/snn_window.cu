// snn_window.cu -- the STDP of a window of steps in one pass over the
// synapses (paper Sec. 2, cycle steps 2.1 and 2.4 "Synaptic update", and, at a
// period's end, Table 2 "long term synaptic plasticity").
//
// Inside a period the weights do not change and a derivative is a sum of
// integer amounts, so it does not matter when they are added: a call that
// runs many steps may leave the amounts of a window of up to kWinSteps steps
// to one pass at the window's end (still inside the call).  The pass needs,
// per synapse, the spike trains of its source and target over the window, and
// reads and writes the derivative once instead of once per step:
//   potentiation: for each post spike at p0 + k, the amount at the lag to the
//       source's latest arrival at or before it;
//   depression: for each arrival at p0 + k, the amount at the lag to the
//       target's latest spike before it.
// A dense step then moves 6 bytes per synapse (target and weight) instead of
// 14: at 1.28 M neurons of 1125 synapses about 1.5 ms instead of 2.9, plus the
// pass, 7.5 ms per 50 steps (bound by instruction issue: two sums over 50-bit
// trains per synapse).  A train is a 64-bit word: 56 step bits and, in the top 8, the lag of
// the latest event before the window (255: none that matters).
#include "snn_internal.cuh"

namespace snn {

constexpr unsigned long long kTrainMask = (1ull << kWinBits) - 1ull;

size_t stdp_smem_bytes(uint32_t npc, uint32_t block)
{
    return (size_t)kSlots * npc * 8            // trains of the 13 columns the rows reach
           + (size_t)(block / 32) * 32 * 8     // per warp: arrival trains, one per delay
           + (size_t)(block / 32) * 32 * 4     // per warp: bucket ends
           + 2 * kLut * 4;                     // amounts
}

__device__ __forceinline__ int top_bit(unsigned long long x) { return 63 - __clzll((long long)x); }

// Sum of lut[lag] over the set bits k of `at`: lag to the latest bit of
// `of` at or before k - `gap` (gap 0 or 1), else k + before (the lag of the
// latest event before the window), beyond the table 0.  Few bits are taken
// one by one; many are counted lag by lag, which ends after the longest
// gap between two bits of `of`.
__device__ __forceinline__ int32_t nearest_sum(unsigned long long at, unsigned long long of, int gap, int before,
                                               const int32_t *lut)
{
    int32_t sum = 0;
    if (__popcll(at) > 6) {
        const unsigned long long first = (of & (0ull - of)) << gap;      // first bit that has a predecessor
        unsigned long long early = of ? at & (first - 1ull) : at;
        at ^= early;
        unsigned long long s = of << gap;
        for (int lag = gap; at; ++lag, s <<= 1) {
            const unsigned long long hit = at & s;
            if (hit) {
                sum += lut[lag] * __popcll(hit);
                at ^= hit;
            }
        }
        at = early;
        while (at) {
            const int lag = __ffsll((long long)at) - 1 + before;
            if (lag >= kLut - 1) break;
            sum += lut[lag];
            at &= at - 1ull;
        }
        return sum;
    }
    while (at) {
        const int k = __ffsll((long long)at) - 1;
        at &= at - 1ull;
        const unsigned long long m = of & ((1ull << (k + 1 - gap)) - 1ull);
        const int lag = m ? k - top_bit(m) : min(k + before, kLut - 1);
        sum += lut[lag];
    }
    return sum;
}

__device__ __forceinline__ void win_open_body(const DevNet &n, const int *t_now, int steps, const Part &g)
{
    if (!n.win) return;
    const uint32_t tid = part_tid(g), threads = part_threads(g);
    for (uint32_t i = tid; i < n.N; i += threads) n.hl0[i] = n.hl[i];
    if (tid == 0) {
        n.win->p0 = *t_now;
        n.win->p1 = *t_now + steps - 1;
        n.win->defer_from = kNoDefer;
        n.win->cursor = 0;
        n.win->done = 0;
    }
}

// The window's spike bits (a word of 32 neurons per step) turned into one
// train word per neuron.  A warp takes 8 words: its loads are full sectors,
// 32 ballots turn 32 steps of 32 neurons.
__device__ __forceinline__ void train_body(const DevNet &n, const int *t_now, const Part &g)
{
    __shared__ uint32_t s_bits[8][kWinSlots][8];
    if (!n.win || !deferring(n, *t_now)) return;
    const int p0 = n.win->p0, steps = n.win->p1 - p0 + 1;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t warps = part_threads(g) >> 5, nw = (n.N + 31u) / 32u;
    uint32_t (*bits)[8] = s_bits[warp];
    for (uint32_t w0 = (part_tid(g) >> 5) * 8u; w0 < nw; w0 += warps * 8u) {
        const uint32_t w = w0 + (lane & 7);
        for (int k = lane >> 3; k < kWinSlots; k += 4)
            bits[k][lane & 7] = (k < steps && w < nw) ? n.spk[(size_t)((p0 + k) & (kWinSlots - 1)) * n.spk_words + w] : 0u;
        __syncwarp();
        for (int q = 0; q < 8; ++q) {
            const uint32_t x0 = bits[lane][q], x1 = bits[lane + 32][q];
            uint32_t lo = 0, hi = 0;
#pragma unroll
            for (int b = 0; b < 32; ++b) {
                const uint32_t y0 = __ballot_sync(0xffffffffu, (x0 >> b) & 1u);
                const uint32_t y1 = __ballot_sync(0xffffffffu, (x1 >> b) & 1u);
                if (lane == b) {
                    lo = y0;
                    hi = y1;
                }
            }
            const uint32_t i = (w0 + q) * 32u + lane;
            if (i < n.N) {
                const uint2 h = n.hl0[i];
                const int lag = h.x ? __ffs(h.x) : p0 - (int)h.y;      // bit j: fired at p0 - 1 - j
                n.train[i] = (unsigned long long)lo | ((unsigned long long)hi << 32) |
                             ((unsigned long long)min(lag, kLut - 1) << kWinBits);
            }
        }
        __syncwarp();
    }
}

// One row: the lane takes 4 synapses per pass.
template <bool kDeriv>
__device__ __forceinline__ void stdp_row(const DevNet &n, int64_t base, int m, int D, const int32_t *w_off,
                                         const unsigned long long *w_x, const unsigned long long *s_y,
                                         const int32_t *s_lutp, const int32_t *s_lutm, unsigned long long posts,
                                         unsigned long long arrivals, int lane)
{
    const uint2 *rt2 = reinterpret_cast<const uint2 *>(n.tgt16 + base);
    int4 *rs4 = reinterpret_cast<int4 *>(n.sd + base);
    int4 *rw4 = reinterpret_cast<int4 *>(n.w + base);
    const float scale = (float)D / (float)m;
    for (int c = lane; c * 4 < m; c += 32) {
        const int k0 = c * 4;
        if (out_of_range(n, base + k0 + 4 <= n.S)) continue;
        const uint2 tv = rt2[c];
        const int4 sa = rs4[c];
        int4 wa = make_int4(0, 0, 0, 0);
        if (kDeriv) wa = rw4[c];
        int d = min(D, 1 + (int)((float)k0 * scale));
        while (w_off[d] <= k0) ++d;       // bucket D ends at m > k0
        while (w_off[d - 1] > k0) --d;    // w_off[0] = 0 <= k0
        const uint32_t tw[2] = {tv.x, tv.y};
        int32_t sv[4] = {sa.x, sa.y, sa.z, sa.w};
        int32_t wv[4] = {wa.x, wa.y, wa.z, wa.w};
        bool dirty = kDeriv;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (k0 + u >= m) continue;    // the row's padding
            while (k0 + u >= w_off[d]) ++d;
            const uint32_t v = (u & 1) ? (tw[u >> 1] >> 16) : (tw[u >> 1] & 0xffffu);
            if (out_of_range(n, v < kSlots * n.npc)) continue;
            const unsigned long long x = w_x[d], y = s_y[v];
            const unsigned long long xb = x & kTrainMask, yb = y & kTrainMask;
            const int32_t delta = nearest_sum(yb & posts, xb, 0, (int)(x >> kWinBits), s_lutp) -
                                  nearest_sum(xb & arrivals, yb, 1, (int)(y >> kWinBits), s_lutm);
            if (delta) {
                sv[u] += delta;
                dirty = true;
            }
            if (kDeriv) {
                wv[u] = deriv_w(n, wv[u], sv[u]);
                sv[u] = deriv_sd(n, sv[u]);
            }
        }
        if (dirty) rs4[c] = make_int4(sv[0], sv[1], sv[2], sv[3]);
        if (kDeriv) rw4[c] = make_int4(wv[0], wv[1], wv[2], wv[3]);
    }
}

__device__ __forceinline__ void stdp_body(const DevNet &n, const int *t_now, const Part &g)
{
    extern __shared__ int4 smem_i4[];
    const int t = *t_now;                  // the step after the window
    if (!n.win) return;
    DevWindow *win = n.win;
    if (!deferring(n, t)) {
        if (g.bid == 0 && threadIdx.x == 0) win->p1 = win->p0 - 1;   // closed, nothing was left to it
        return;
    }
    const uint32_t npc = n.npc, nwarps = blockDim.x >> 5;
    unsigned long long *s_y = reinterpret_cast<unsigned long long *>(smem_i4);      // [kSlots * npc]
    unsigned long long *s_x = s_y + kSlots * npc;                                   // [nwarps][32]
    int32_t *s_off = reinterpret_cast<int32_t *>(s_x + nwarps * 32);                // [nwarps][32]
    int32_t *s_lutp = s_off + nwarps * 32;
    int32_t *s_lutm = s_lutp + kLut;
    __shared__ uint32_t s_col[kSlots];
    __shared__ uint32_t s_unit;
    const int p0 = win->p0, from = win->defer_from;
    // arrivals from step `from` to the window's last are depressed here (later
    // ones of its spikes belong to the next); the potentiation owed by step
    // from - 1 is the window's too
    const unsigned long long arrivals = ((1ull << (t - p0)) - 1ull) & ~((1ull << (from - p0)) - 1ull);
    const unsigned long long posts = kTrainMask & ~((1ull << max(0, from - 1 - p0)) - 1ull);
    const bool closes = n.deriv_period && (t % (int)n.deriv_period) == 0;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int D = (int)n.D;
    unsigned long long *w_x = s_x + warp * 32;
    int32_t *w_off = s_off + warp * 32;
    for (int i = threadIdx.x; i < kLut; i += blockDim.x) {
        s_lutp[i] = n.lut_p[i];
        s_lutm[i] = n.lut_m[i];
    }
    const uint32_t chunks = (n.ne + n.stdp_rows - 1) / n.stdp_rows;
    for (uint32_t unit = g.bid; unit < n.C * chunks;) {
        const uint32_t col = unit / chunks;
        const uint32_t r0 = (unit - col * chunks) * n.stdp_rows;
        const uint32_t r1 = min(n.ne, r0 + n.stdp_rows);
        if (threadIdx.x < kSlots) s_col[threadIdx.x] = (uint32_t)n.nbr[col * kSlotStride + threadIdx.x];
        __syncthreads();
        for (int sl = 0; sl < kSlots; ++sl) {
            const unsigned long long *src = n.train + (size_t)s_col[sl] * npc;
            for (uint32_t loc = threadIdx.x; loc < npc; loc += blockDim.x) s_y[sl * npc + loc] = src[loc];
        }
        __syncthreads();
        for (uint32_t r = r0 + warp; r < r1; r += nwarps) {
            const uint32_t p = col * npc + r;
            const unsigned long long own = s_y[r] & kTrainMask;          // slot 0 is the row's own column
            const uint2 h = n.hl0[p];
            const int end = lane <= D ? (int)n.doff[(size_t)p * kDoffStride + lane] : 0;
            const int m = __shfl_sync(0xffffffffu, end, D);
            unsigned long long x = 0;
            if (lane >= 1 && lane <= D) {
                // arrivals by delay `lane`: source spikes of the window, and
                // before it (bit j of h.x: fired at p0 - 1 - j)
                const uint32_t recent = h.x & (0xffffffffu << lane);
                const int lag = recent ? __ffs(recent) - lane : p0 - (int)h.y - lane;
                x = ((own << lane) | (unsigned long long)(__brev(h.x) >> (32 - lane))) & kTrainMask;
                x |= (unsigned long long)min(lag, kLut - 1) << kWinBits;
            }
            w_x[lane] = x;
            w_off[lane] = end;
            // a source without an arrival inside any amount's reach changes nothing
            const bool live = (x & kTrainMask) || (lane >= 1 && lane <= D && (int)(x >> kWinBits) < kLut - 1);
            __syncwarp();
            if (closes || __any_sync(0xffffffffu, live)) {
                const int64_t base = row_base(n, p);
                if (closes) stdp_row<true>(n, base, m, D, w_off, w_x, s_y, s_lutp, s_lutm, posts, arrivals, lane);
                else stdp_row<false>(n, base, m, D, w_off, w_x, s_y, s_lutp, s_lutm, posts, arrivals, lane);
            }
            __syncwarp();
        }
        if (threadIdx.x == 0) s_unit = g.nblk + atomicAdd(&win->cursor, 1u);
        __syncthreads();
        unit = s_unit;
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(&win->done, 1u) == g.nblk - 1) {
            // every block has read the window: it closes, nothing is owed
            win->p1 = win->p0 - 1;
            win->defer_from = kNoDefer;
            win->cursor = 0;
            win->done = 0;
            n.ctr->ltp_pending = kNoPending;
            n.ctr->fold_cursor = 0;
        }
    }
}

__global__ void __launch_bounds__(1024) k_win_open(DevNet n, const int *t_now, int steps)
{
    win_open_body(n, t_now, steps, whole_grid());
}

__global__ void __launch_bounds__(256) k_train(DevNet n, const int *t_now) { train_body(n, t_now, whole_grid()); }

__global__ void __launch_bounds__(kStdpBlock) k_stdp(DevNet n, const int *t_now) { stdp_body(n, t_now, whole_grid()); }

__global__ void __launch_bounds__(1024) k_win_open_b(BatchLaunch b, int steps)
{
    const BatchBlock x = batch_block(b);
    const DevNet n = b.nets[x.net];
    win_open_body(n, x.t_now, steps, x.part);
}

__global__ void __launch_bounds__(256) k_train_b(BatchLaunch b)
{
    const BatchBlock x = batch_block(b);
    const DevNet n = b.nets[x.net];
    train_body(n, x.t_now, x.part);
}

__global__ void __launch_bounds__(kStdpBlock) k_stdp_b(BatchLaunch b)
{
    const BatchBlock x = batch_block(b);
    const DevNet n = b.nets[x.net];
    stdp_body(n, x.t_now, x.part);
}

}  // namespace snn
