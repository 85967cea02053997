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
// 14: at 1.28 M neurons of 1125 synapses 1.2 ms instead of 2.9, plus the pass,
// 3 to 8 ms per 50 steps (bound by instruction issue: two sums over 50-bit
// trains per synapse; 0.72 of the issue slots).  A train is a 64-bit word: 56 step bits and, in the top 8, the lag of
// the latest event before the window (255: none that matters).
#include <type_traits>

#include "snn_internal.cuh"

namespace snn {

constexpr unsigned long long kTrainMask = (1ull << kWinBits) - 1ull;

constexpr int kSpikeCap = 96;          // spikes of a row that arrive in a window: at most 31 + kWinSteps
constexpr int kChunks = 22;            // chunks of 4 steps, -31 .. 56, of a row's potentiation amounts
constexpr int kChunkStride = 20;       // a sum per set of a chunk's steps; 4 more words, so that the empty sets of
                                       // eight chunks lie in different banks
constexpr int kAmounts = kChunks * kChunkStride;
constexpr int kFewSpikes = 14;         // up to here a row's arrivals are taken one by one

size_t stdp_smem_bytes(uint32_t npc, uint32_t block)
{
    return (size_t)kSlots * npc * 8            // trains of the 13 columns the rows reach
           + (size_t)(block / 32) * 32 * 8     // per warp: arrival trains, one per delay
           + (size_t)(block / 32) * 64 * 4     // per warp: bucket ends, sums for saturated targets
           + (size_t)(block / 32) * kSpikeCap  // per warp: the row's spike times
           + (size_t)(block / 32) * kAmounts * 4   // per warp: the row's potentiation amounts
           + 2 * kLut * 4;                     // amounts
}

__device__ __forceinline__ void win_open_body(const DevNet &n, const int *t_now, int steps, const Part &g)
{
    if (!n.win) return;
    const uint32_t tid = part_tid(g), threads = part_threads(g);
    for (uint32_t i = tid; i < n.N; i += threads) n.hl0[i] = n.hl[i];
    if (tid == 0) {
        const int t = *t_now;
        n.win->p0 = t;
        n.win->p1 = t + steps - 1;
        // behind a busy window, whose pass left nothing owed, every step of this
        // one may leave its STDP to the pass (else the first step's rate
        // decides; saturated: 1.2 ms for that step instead of 3.0)
        int from = kNoDefer;
        if (t > 0 && steps >= 2 && n.ctr->ltp_pending == kNoPending) {
            const int slot = (t - 1) % (int)n.D;
            const unsigned long long total = (unsigned)n.ring_cnt[2 * slot] + (unsigned)n.ring_cnt[2 * slot + 1];
            if (total * (unsigned)steps >= n.defer_visits) from = t;
        }
        n.win->defer_from = from;
        n.win->cursor = 0;
        n.win->done = 0;
    }
}

// The window's spike bits (a word of 32 neurons per step) turned into one
// train word per neuron.  A warp takes 8 words: its loads are full sectors,
// 32 ballots turn 32 steps of 32 neurons.
__device__ __forceinline__ void train_body(const DevNet &n, const Part &g)
{
    __shared__ uint32_t s_bits[8][kWinSlots][8];
    if (!n.win || n.win->defer_from > n.win->p1) return;
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
                const int lag = h.x ? __ffs(h.x) : lag_of(p0, (int)h.y);      // bit j: fired at p0 - 1 - j
                n.train[i] = (unsigned long long)lo | ((unsigned long long)hi << 32) |
                             ((unsigned long long)lag << kWinBits);
            }
        }
        __syncwarp();
    }
}

// The potentiation of a synapse of delay b: the amounts of the row's steps
// k - b over the post spikes k, four steps at a time from the row's table.  A
// fixed 14 lookups: a warp that took the set bits one by one ran as long as its
// busiest target (16x16 torus of the paper's columns, 2 to 3 spikes per neuron
// and window: 360 us per pass, 463 bit by bit; without the padding between the
// chunks 400).
__device__ __forceinline__ int32_t row_ltp(const int32_t *w_q, int b, unsigned long long posts)
{
    const unsigned long long z = posts << ((31 - b) & 3);
    const int32_t *const q = w_q + ((31 - b) >> 2) * kChunkStride;
    int32_t sum = 0;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const uint32_t z4 = (uint32_t)(z >> (32 * h));
        const uint32_t even = z4 & 0x0f0f0f0fu, odd = (z4 >> 4) & 0x0f0f0f0fu;
#pragma unroll
        for (int i = 0; i < (h ? 3 : 4); ++i)
            sum += q[(8 * h + 2 * i) * kChunkStride + ((even >> (8 * i)) & 0xffu)] +
                   q[(8 * h + 2 * i + 1) * kChunkStride + ((odd >> (8 * i)) & 0xffu)];
    }
    return sum;
}
static_assert(kWinSteps + 3 <= 56 && 31 / 4 + 14 <= kChunks, "row_ltp's 14 chunks");

// The train word of a target that fired in every step of the window and in the
// one before it.  What such a target's synapse gains depends on the row and
// the delay alone, so a row with many spikes has one sum for it per delay: in a
// saturated net the pass then moves its 10 bytes per synapse at 0.6 of the copy
// bandwidth (3.0 ms at 1152 M plastic synapses, 5.5 with each synapse's sums).
__device__ __forceinline__ unsigned long long saturated_train(int steps)
{
    return ((1ull << steps) - 1ull) | (1ull << kWinBits);
}

// The depression of a synapse whose source has many spikes: the amounts of the
// arrivals `at` at the lag to the latest bit of y before each, else to the
// latest post spike before the window.  Counted lag by lag, which ends after
// the longest gap between two post spikes: a target that fires in every step
// is done after the first.
__device__ __forceinline__ int32_t many_ltd(unsigned long long at, unsigned long long y, const int32_t *lutm)
{
    const unsigned long long of = y & kTrainMask;
    const int before = (int)(y >> kWinBits);
    unsigned long long s = of << 1;
    unsigned long long hit = at & s;
    int32_t sum = lutm[1] * __popcll(hit);
    at ^= hit;
    if (at & 1ull) sum += lutm[before];            // the window's first step: no post spike of it is earlier
    at &= ~1ull;
    if (!at) return sum;
    const unsigned long long first = (of & (0ull - of)) << 1;        // first step behind a post spike
    unsigned long long early = of ? at & (first - 1ull) : at;
    at ^= early;
    for (int lag = 2; at; ++lag) {
        s <<= 1;
        hit = at & s;
        if (hit) {
            sum += lutm[lag] * __popcll(hit);
            at ^= hit;
        }
    }
    for (; early; early &= early - 1ull) {
        const int lag = __ffsll((long long)early) - 1 + before;
        if (lag >= kLut - 1) break;
        sum += lutm[lag];
    }
    return sum;
}

// One row: the lane takes 4 synapses per pass.
//   kFew: the row has few spikes, at times w_j[0..ns) relative to the window
//   (an arrival is delay d later); the depression of its arrivals is looked up
//   by all lanes in turn, at the lag to the target's latest post spike before
//   each.
template <bool kDeriv, bool kFew>
__device__ __forceinline__ void stdp_row(const DevNet &n, int64_t base, int m, int D, const int32_t *w_off,
                                         const unsigned long long *w_x, const signed char *w_j, int ns,
                                         const unsigned long long *s_y, const int32_t *w_q, const int32_t *s_lutm,
                                         int steps, unsigned long long posts, unsigned long long arrivals, int lane)
{
    const uint2 *rt2 = reinterpret_cast<const uint2 *>(n.tgt16 + base);
    int4 *rs4 = reinterpret_cast<int4 *>(n.sd + base);
    int4 *rw4 = reinterpret_cast<int4 *>(n.w + base);
    const float scale = (float)D / (float)m;
    const int a_min = arrivals ? __ffsll((long long)arrivals) - 1 : steps;
    for (int c = lane; c * 4 < m; c += 32) {
        const int k0 = c * 4;
        if (out_of_range(n, base + k0 + 4 <= n.S)) continue;
        const uint2 tv = rt2[c];
        const int4 sa = rs4[c];
        int4 wa = make_int4(0, 0, 0, 0);
        if (kDeriv) wa = rw4[c];
        int b = min(D, 1 + (int)((float)k0 * scale));
        int e = w_off[b];                 // end of bucket b
        while (e <= k0) e = w_off[++b];   // bucket D ends at m > k0
        for (int o; (o = w_off[b - 1]) > k0; --b) e = o;    // w_off[0] = 0 <= k0
        const uint32_t tw[2] = {tv.x, tv.y};
        int32_t delta[4];
        int d[4];                         // a synapse's delay, or a bucket that holds the row's padding
        unsigned long long y[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const uint32_t v = (u & 1) ? (tw[u >> 1] >> 16) : (tw[u >> 1] & 0xffffu);
            const bool in = k0 + u < m && !out_of_range(n, v < kSlots * n.npc);     // not the row's padding
            if (in)
                while (k0 + u >= e) e = w_off[++b];
            d[u] = in || !kFew ? b : -kSpikeCap;      // padding: every arrival lies before the window
            y[u] = in ? s_y[v] : !kFew ? saturated_train(steps) : 0ull;
        }
        if (kFew) {
            uint32_t y0[4], y1[4];        // post spikes of steps 0..31, 32..55
            int before0[4], before1[4];   // a - the latest post spike before step 0 (32): a + this
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                delta[u] = row_ltp(w_q, max(d[u], 1), y[u] & posts);
                y0[u] = (uint32_t)y[u];
                y1[u] = (uint32_t)(y[u] >> 32) & (uint32_t)(kTrainMask >> 32);
                before0[u] = (int)(y[u] >> kWinBits);
                before1[u] = y0[u] ? __clz((int)y0[u]) - 31 : before0[u];
            }
            for (int i = 0; i < ns; ++i) {
                const int j = w_j[i];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int a = j + d[u];
                    if (a < a_min || a >= steps) continue;
                    // post spikes of a's half of the window before a, the latest on top
                    const uint32_t z = ((a < 32 ? y0[u] : y1[u]) << 1) << (31 - (a & 31));
                    const int lag = z ? 1 + __clz((int)z) : a + (a < 32 ? before0[u] : before1[u]);
                    delta[u] -= s_lutm[min(lag, kLut - 1)];
                }
            }
        } else {
#pragma unroll
            for (int u = 0; u < 4; ++u) delta[u] = w_off[32 + d[u]];
            const unsigned long long all = saturated_train(steps);
            if (y[0] != all || y[1] != all || y[2] != all || y[3] != all) {
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    delta[u] = row_ltp(w_q, d[u], y[u] & posts) - many_ltd(w_x[d[u]] & arrivals, y[u], s_lutm);
            }
#pragma unroll
            for (int u = 1; u < 4; ++u)
                if (k0 + u >= m) delta[u] = 0;
        }
        const bool dirty = kDeriv || delta[0] || delta[1] || delta[2] || delta[3];
        int32_t sv[4] = {sa.x + delta[0], sa.y + delta[1], sa.z + delta[2], sa.w + delta[3]};
        if (kDeriv) {
            int32_t wv[4] = {wa.x, wa.y, wa.z, wa.w};
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (k0 + u >= m) continue;
                wv[u] = deriv_w(n, wv[u], sv[u]);
                sv[u] = deriv_sd(n, sv[u]);
            }
            rw4[c] = make_int4(wv[0], wv[1], wv[2], wv[3]);
        }
        if (dirty) rs4[c] = make_int4(sv[0], sv[1], sv[2], sv[3]);
    }
}

// What a warp keeps of a row for its synapses: bucket ends (`end` in lane d),
// arrival trains by delay, the source's spike times (ns of them) and the
// potentiation amounts.  own: the source's spikes in the window, h: its history
// before.
__device__ __forceinline__ void row_spikes(unsigned long long own, uint2 h, int end, int D, int p0, int lane, int32_t *w_off,
                                           unsigned long long *w_x, signed char *w_j, int32_t *w_q, const int32_t *s_lutp,
                                           int &ns)
{
    unsigned long long x = 0;
    if (lane >= 1 && lane <= D) {
        // arrivals by delay `lane`: source spikes of the window, and
        // before it (bit j of h.x: fired at p0 - 1 - j)
        x = ((own << lane) | (unsigned long long)(__brev(h.x) >> (32 - lane))) & kTrainMask;
    }
    w_x[lane] = x;
    w_off[lane] = end;
    // the source's spikes that arrive in the window, in order: the
    // last D steps before it and the window's own
    const uint32_t pre = h.x & (0xffffffffu >> (32 - D));
    const int npre = __popc(pre);
    ns = npre + __popcll(own);
    if ((pre >> lane) & 1u) w_j[npre - __popc(pre & (0xffffffffu >> (31 - lane)))] = (signed char)(-1 - lane);
#pragma unroll
    for (int q = lane; q < 64; q += 32)
        if ((own >> q) & 1ull) w_j[npre + __popcll(own & ((1ull << q) - 1ull))] = (signed char)q;
    // what a post spike `tau` after a spike's own step, less the delay,
    // adds: the amount at the lag to the source's latest spike; a lane sums the
    // 16 sets of its 4 steps
    if (lane < kChunks) {
        // spikes at tau + 31: bit j of h.x is tau -1 - j
        const unsigned long long c = own << 31 | (unsigned long long)(__brev(h.x) >> 1);
        const uint32_t w0 = (uint32_t)c, w1 = (uint32_t)(c >> 32), w2 = (uint32_t)(own >> 33);
        const int k = lane >> 3, sh = 4 * (lane & 7);
        const uint32_t word = k == 0 ? w0 : k == 1 ? w1 : w2;
        // the lag at the chunk's first step: to a spike of its word at or before
        // it, of the words before, of the history
        const uint32_t late = word & ((2u << sh) - 1u);
        const uint32_t p1 = k == 2 ? w1 : k == 1 ? w0 : 0u, p2 = k == 2 ? w0 : 0u;
        int lag = late ? sh - 31 + __clz((int)late)
                : p1   ? sh + 1 + __clz((int)p1)
                : p2   ? sh + 33 + __clz((int)p2)
                       : 4 * lane + ((h.x >> 31) ? 1 : lag_of(p0 - 31, (int)h.y));
        int32_t q[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (u) lag = (word >> (sh + u)) & 1u ? 0 : lag + 1;
            q[u] = s_lutp[min(lag, kLut - 1)];
        }
        const int4 a = make_int4(0, q[0], q[1], q[0] + q[1]);
        int4 *const o = reinterpret_cast<int4 *>(w_q + kChunkStride * lane);
        auto plus = [&](int32_t x) { return make_int4(a.x + x, a.y + x, a.z + x, a.w + x); };
        o[0] = a;
        o[1] = plus(q[2]);
        o[2] = plus(q[3]);
        o[3] = plus(q[2] + q[3]);
    }
}

// a source without an arrival inside any amount's reach changes nothing
__device__ __forceinline__ bool row_live(unsigned long long own, uint2 h, int p0, int D)
{
    return own || h.x || lag_of(p0 - D, (int)h.y) < kLut - 1;
}

// One row of a net with target lists (explicit targets: no alignment, no
// slots): a lane per synapse, its target's train from memory.  The net's
// trains are a few KB to a few MB and stay in L2.
template <bool kDeriv>
__device__ __forceinline__ void stdp_row_lists(const DevNet &n, int64_t base, int m, int D, const int32_t *w_off,
                                               const unsigned long long *w_x, const signed char *w_j, int ns,
                                               const int32_t *w_q, const int32_t *s_lutm, int steps,
                                               unsigned long long posts, unsigned long long arrivals, int lane)
{
    const float scale = (float)D / (float)m;
    const int a_min = arrivals ? __ffsll((long long)arrivals) - 1 : steps;
    for (int k = lane; k < m; k += 32) {
        if (out_of_range(n, base + k < n.S)) continue;
        const uint32_t v = (uint32_t)n.tgt[base + k];
        const int32_t sd = n.sd[base + k];
        const int32_t w = kDeriv ? n.w[base + k] : 0;
        if (out_of_range(n, v < n.N)) continue;
        const unsigned long long y = n.train[v];
        int b = min(D, 1 + (int)((float)k * scale));
        while (w_off[b] <= k) ++b;        // bucket D ends at m > k
        while (w_off[b - 1] > k) --b;     // w_off[0] = 0 <= k
        int32_t delta = row_ltp(w_q, b, y & posts);
        if (ns <= kFewSpikes) {
            const int before = (int)(y >> kWinBits);
            for (int i = 0; i < ns; ++i) {
                const int a = (int)w_j[i] + b;
                if (a < a_min || a >= steps) continue;
                const unsigned long long z = y & ((1ull << a) - 1ull);      // post spikes before a (< kWinBits)
                const int lag = z ? a - 63 + __clzll((long long)z) : a + before;
                delta -= s_lutm[min(lag, kLut - 1)];
            }
        } else {
            delta -= many_ltd(w_x[b] & arrivals, y, s_lutm);
        }
        if (kDeriv) {
            n.w[base + k] = deriv_w(n, w, sd + delta);
            n.sd[base + k] = deriv_sd(n, sd + delta);
        } else if (delta) {
            n.sd[base + k] = sd + delta;
        }
    }
}

// the last block of the pass closes the window: nothing is owed
__device__ __forceinline__ void close_pass(const DevNet &n, uint32_t blocks)
{
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        DevWindow *win = n.win;
        if (atomicAdd(&win->done, 1u) == blocks - 1) {
            // every block has read the window
            win->p1 = win->p0 - 1;
            win->defer_from = kNoDefer;
            win->cursor = 0;
            win->done = 0;
            n.ctr->ltp_pending = kNoPending;
            n.ctr->fold_cursor = 0;
        }
    }
}

__device__ __forceinline__ void stdp_body(const DevNet &n, const Part &g)
{
    extern __shared__ int4 smem_i4[];
    if (!n.win) return;
    DevWindow *win = n.win;
    const int t = win->p1 + 1;             // the step after the window
    if (win->defer_from > win->p1) {
        if (g.bid == 0 && threadIdx.x == 0) win->p1 = win->p0 - 1;   // closed, nothing was left to it
        return;
    }
    const uint32_t npc = n.npc, nwarps = blockDim.x >> 5;
    int32_t *s_q = reinterpret_cast<int32_t *>(smem_i4);                            // [nwarps][kAmounts]
    unsigned long long *s_y = reinterpret_cast<unsigned long long *>(s_q + nwarps * kAmounts);   // [kSlots * npc]
    unsigned long long *s_x = s_y + kSlots * npc;                                   // [nwarps][32]
    int32_t *s_off = reinterpret_cast<int32_t *>(s_x + nwarps * 32);                // [nwarps][64]
    int32_t *s_lutp = s_off + nwarps * 64;
    int32_t *s_lutm = s_lutp + kLut;
    signed char *s_j = reinterpret_cast<signed char *>(s_lutm + kLut);              // [nwarps][kSpikeCap]
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
    int32_t *w_off = s_off + warp * 64;
    signed char *w_j = s_j + warp * kSpikeCap;
    for (int i = threadIdx.x; i < kLut; i += blockDim.x) {
        s_lutp[i] = n.lut_p[i];
        s_lutm[i] = n.lut_m[i];
    }
    int32_t *w_q = s_q + warp * kAmounts;
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
        // the warp's rows, 32 at a time: a lane finds out whether its row has
        // anything to do, the next such row's bucket ends are read ahead
        for (uint32_t q0 = r0 + warp; q0 < r1; q0 += 32 * nwarps) {
            const uint32_t q = q0 + lane * nwarps;
            const uint2 hq = q < r1 ? n.hl0[col * npc + q] : make_uint2(0, 0);
            uint32_t rows = __ballot_sync(0xffffffffu, q < r1 && (closes || row_live(s_y[q] & kTrainMask, hq, p0, D)));
            auto ends = [&](int at) {
                return lane <= D ? (int)n.doff[(size_t)(col * npc + q0 + at * nwarps) * kDoffStride + lane] : 0;
            };
            int next = rows ? ends(__ffs(rows) - 1) : 0;
            while (rows) {
                const int at = __ffs(rows) - 1, end = next;
                rows &= rows - 1u;
                if (rows) next = ends(__ffs(rows) - 1);
                const uint32_t r = q0 + at * nwarps;
                const uint2 h = make_uint2(__shfl_sync(0xffffffffu, hq.x, at), __shfl_sync(0xffffffffu, hq.y, at));
                int ns;
                row_spikes(s_y[r] & kTrainMask, h, end, D, p0, lane, w_off, w_x, w_j, w_q, s_lutp, ns);   // slot 0: own column
                const int m = __shfl_sync(0xffffffffu, end, D);
                __syncwarp();
                if (ns > kFewSpikes) {
                    if (lane >= 1 && lane <= D)
                        w_off[32 + lane] = row_ltp(w_q, lane, saturated_train(t - p0) & posts) -
                                           s_lutm[1] * __popcll(w_x[lane] & arrivals);
                    __syncwarp();
                }
                auto row = [&](auto deriv, auto few) {
                    stdp_row<decltype(deriv)::value, decltype(few)::value>(n, row_base(n, col * npc + r), m, D, w_off, w_x,
                                                                          w_j, ns, s_y, w_q, s_lutm, t - p0, posts,
                                                                          arrivals, lane);
                };
                if (ns <= kFewSpikes) {
                    if (closes) row(std::true_type{}, std::true_type{});
                    else row(std::false_type{}, std::true_type{});
                } else {
                    if (closes) row(std::true_type{}, std::false_type{});
                    else row(std::false_type{}, std::false_type{});
                }
                __syncwarp();
            }
        }
        if (threadIdx.x == 0) s_unit = g.nblk + atomicAdd(&win->cursor, 1u);
        __syncthreads();
        unit = s_unit;
        __syncthreads();
    }
    close_pass(n, g.nblk);
}

__device__ __forceinline__ void stdp_lists_body(const DevNet &n)
{
    extern __shared__ int4 smem_i4[];
    if (!n.win) return;
    DevWindow *win = n.win;
    const int t = win->p1 + 1;             // the step after the window
    if (win->defer_from > win->p1) return; // (a resident grid defers all steps of a window or ran none)
    const int nwarps = (int)(blockDim.x >> 5), lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int32_t *s_q = reinterpret_cast<int32_t *>(smem_i4), *w_q = s_q + warp * kAmounts;   // as stdp_body, without trains
    unsigned long long *s_x = reinterpret_cast<unsigned long long *>(s_q + nwarps * kAmounts), *w_x = s_x + warp * 32;
    int32_t *s_off = reinterpret_cast<int32_t *>(s_x + nwarps * 32), *w_off = s_off + warp * 64;
    int32_t *s_lutp = s_off + nwarps * 64, *s_lutm = s_lutp + kLut;
    signed char *w_j = reinterpret_cast<signed char *>(s_lutm + kLut) + warp * kSpikeCap;
    const int p0 = win->p0, from = win->defer_from;
    const unsigned long long arrivals = ((1ull << (t - p0)) - 1ull) & ~((1ull << (from - p0)) - 1ull);
    const unsigned long long posts = kTrainMask & ~((1ull << max(0, from - 1 - p0)) - 1ull);
    const bool closes = n.deriv_period && (t % (int)n.deriv_period) == 0;
    for (int i = threadIdx.x; i < kLut; i += blockDim.x) {
        s_lutp[i] = n.lut_p[i];
        s_lutm[i] = n.lut_m[i];
    }
    __syncthreads();
    for (uint32_t r = blockIdx.x * nwarps + warp; r < n.C * n.ne; r += gridDim.x * nwarps) {
        const uint32_t col = r / n.ne, p = col * n.npc + (r - col * n.ne);
        const unsigned long long own = n.train[p] & kTrainMask;
        const uint2 h = n.hl0[p];
        if (closes || row_live(own, h, p0, (int)n.D)) {
            const int end = lane <= (int)n.D ? (int)n.doff[(size_t)p * kDoffStride + lane] : 0;
            const int m = __shfl_sync(0xffffffffu, end, (int)n.D);
            int ns;
            row_spikes(own, h, end, (int)n.D, p0, lane, w_off, w_x, w_j, w_q, s_lutp, ns);
            __syncwarp();
            auto row = [&](auto deriv) {
                stdp_row_lists<decltype(deriv)::value>(n, row_base(n, p), m, (int)n.D, w_off, w_x, w_j, ns, w_q, s_lutm,
                                                       t - p0, posts, arrivals, lane);
            };
            if (closes) row(std::true_type{});
            else row(std::false_type{});
        }
        __syncwarp();
    }
    close_pass(n, gridDim.x);
}

__global__ void __launch_bounds__(1024) k_win_open(DevNet n, const int *t_now, int steps)
{
    win_open_body(n, t_now, steps, whole_grid());
}

__global__ void __launch_bounds__(256) k_train(DevNet n) { train_body(n, whole_grid()); }

__global__ void __launch_bounds__(kStdpBlock) k_stdp(DevNet n) { stdp_body(n, whole_grid()); }

__global__ void __launch_bounds__(kStdpListsBlock) k_stdp_lists(DevNet n) { stdp_lists_body(n); }

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
    train_body(n, x.part);
}

__global__ void __launch_bounds__(kStdpBlock) k_stdp_b(BatchLaunch b)
{
    const BatchBlock x = batch_block(b);
    const DevNet n = b.nets[x.net];
    stdp_body(n, x.part);
}

}  // namespace snn
