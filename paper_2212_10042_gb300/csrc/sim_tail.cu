// sim_tail.cu -- the z-test simulation without a histogram over every trial: counts
// of the rejections alone (k_sim_count), and the order statistic from a small tail
// of the trials (k_sim_tail).
//
// The cell-histogram kernel (sim_ztest.cu) increments a shared-memory cell for
// every trial, then reads the tile's box of ~1,700 cells off: about twelve thread
// instructions a trial at K = 16,384, half of them the read-off.
//
// k_sim_count.  S(x_0, x_1) < lambda iff x_1 >= b(x_0), b(x_0) the least such x_1
// (every row of S falls in x_1).  The count table carries b(x_0) in a row of its own
// beside arm 0's counts (k_counts), so four trials are one word: bit 7 of byte
// x_1 + (0x80 - b) is the rejection, no carry crossing a byte while counts and cuts
// stay below 128.  R and the successes of the rejecting trials follow by byte dot
// products: 2.3 thread instructions a trial, no branch, no shared memory.
//
// k_sim_tail (two arms).  The k_i-th smallest S of a tile lies near a known quantile: S is
// nearly normal with mean and variance from the tile's point, and k_i / K_i is
// given.  cap = that quantile at k_i + 3 sqrt(k_i) + 1, and the trials with S < cap are
// among those with x_1 - x_0 >= d, where d is the least cut(x_0) - x_0 over the tile's
// reachable x_0 (the axis box) whose row holds such a trial; four trials a word again.
// Each warp queues these candidates in shared memory and evaluates them 32 at a time:
// the cell's rank (rank = number of cells with a smaller statistic), the rejections,
// the rank as a key in global memory (the warp's own stretch) and in 256 bins.  Then
// the bin of the k_i-th key and its rank within the bin.  Trials left out have S >= cap,
// so the result is exact when it is at most cap and there are k_i keys.  Otherwise it
// is compared with sigma, the least S of a trial left out, and the pass is repeated
// with a lower d: one past the trials that the result asks for, or one, two, three
// less where there were too few candidates, then every trial.  Randomised test: when
// the result lies below cap (or sigma) the candidates hold every trial of the tying
// rank (at cap itself they need not: cells of one statistic differ in x_1 - x_0), so
// their words are gathered from the keys and the m-th smallest taken; no second pass
// over the count rows.
//
// Where lambda is above cap (alternatives, small alpha) the rejections are counted by
// bytes as in k_sim_count and are no candidates.  A box of few cells (rates near 0 or 1,
// few patients, where the quantile misses) is counted cell by cell, as the cell kernel
// does: in the 512 words of the bins and no more, since shared memory is taken from
// L1, which the candidates' reads live on (28 KB a block: 79 -> 91 us at 8,192 tiles).
// Both sides at 8,192 tiles, n = 100, K = 16,384, of the cell kernel's time: theta = 0 0.75,
// theta = -2 and 2 1.5 (one trial in five is a candidate), 3 and beyond 1.2 to 1.3 (by
// candidates 3.5 to 7); theta_1 = theta_0 + 2 1.5 (rejections as candidates 6).
//
// What bounds it: issue slots (67 % issue; 10 to 12 thread instructions a trial, of
// which the test and the queueing take half, the 7 % candidates a third) and the
// latency of the scattered count reads.
// 256^2 grid, K = 16,384 (32,896 tiles): 323 -> 261 us; 2^18 batch: 3.34 -> 2.56 ms;
// randomised calibration of the 128^2 grid, the whole call: 276 -> 187 us.  Five blocks an
// SM at 48 registers were no faster than four at 56.
//
// Tiles: a group of TT threads per tile, G tiles a block: 64 threads with many
// tiles (a warp per tile: 32,896 tiles 20 us a step slower, 8,256 randomised tiles
// 33, 2^18 level, and twice the keys in memory), 128 below 32 tiles an SM, a block
// of 256 below 8 an SM, for the latency of one tile.
#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>

#include "cse_internal.cuh"

namespace {

constexpr int kQueue = 288;   // a warp's candidate queue (up to 31 left over, at least 8 lanes' trials a round)
constexpr int kList = 256;    // words of a tying rank ranked in shared memory
constexpr int kTailThreads = 256;

// Largest box whose cells are counted one by one (k_sim_tail): with words, whose
// gathering is a second pass over the rows, only where candidates fail.
template <bool WORDS>
constexpr int tail_hist()
{
    return WORDS ? 256 : 512;
}

__device__ __forceinline__ int tail_warp_sum(int v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Rejections x >= b among trials k = k0, k0 + 1, .. k0 + 15, then step on, below K: adds
// their number, the sum of their x and (TWO) of their y.  x: the tested counts, y: the
// other arm's, b: each trial's cut (one arm: b1 in every byte).
template <bool TWO = true>
__device__ __forceinline__ void count_rejections(const uint8_t* __restrict__ x, const uint8_t* __restrict__ y,
                                                 const uint8_t* __restrict__ b, int K, int k0, int step, int* R,
                                                 int* X, int* Y, uint32_t b1 = 0u)
{
    uint32_t r = 0u, sx = 0u, sy = 0u;
#pragma unroll 2
    for (int k = k0; k < K; k += step) {   // k + 16 <= k_stride
        const uint4 u = *reinterpret_cast<const uint4*>(x + k);
        uint4 v = make_uint4(0u, 0u, 0u, 0u), c = make_uint4(b1, b1, b1, b1);
        if (TWO) {
            v = *reinterpret_cast<const uint4*>(y + k);
            c = *reinterpret_cast<const uint4*>(b + k);
        }
        const uint32_t xw[4] = {u.x, u.y, u.z, u.w}, yw[4] = {v.x, v.y, v.z, v.w}, bw[4] = {c.x, c.y, c.z, c.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            uint32_t m = ((xw[q] - bw[q] + 0x80808080u) >> 7) & 0x01010101u;   // one per rejecting trial
            const int rem = K - k - 4 * q;
            if (rem < 4) m &= rem > 0 ? (1u << (8 * rem)) - 1u : 0u;
            const uint32_t full = m * 255u;
            r = __dp4a(m, 0x01010101u, r);
            sx = __dp4a(xw[q] & full, 0x01010101u, sx);
            if (TWO) sy = __dp4a(yw[q] & full, 0x01010101u, sy);
        }
    }
    *R += (int)r;
    *X += (int)sx;
    *Y += (int)sy;
}

// A selection key: the rank, or (with the randomised test's words) rank << 17 | the
// trial's place among its warp's.  Ranks lie below 129^2 < 2^15.
template <bool WORDS>
struct tail_key {
    using type = uint16_t;
};
template <>
struct tail_key<true> {
    using type = uint32_t;
};

template <bool WORDS, int G>
__global__ void __launch_bounds__(kTailThreads, 4)
    k_sim_tail(TileArgs T, int32_t n_max, const uint8_t* __restrict__ cnt, int32_t NA, int32_t k_stride,
               int32_t K_tiles, const uint16_t* __restrict__ rank_g, const float* __restrict__ S_g,
               const float* __restrict__ vor_g, const int32_t* __restrict__ pos_g, int32_t n_cells, int32_t n1p,
               int32_t bin_shift, const uint32_t* __restrict__ bb, const int32_t* __restrict__ zpar,
               const uint8_t* __restrict__ zcut, float lambda_up,
               const uint32_t* __restrict__ W, SimOut o, uint32_t* __restrict__ c_tile, void* __restrict__ keys,
               int32_t key_seg, int32_t* __restrict__ counter, int32_t* __restrict__ err)
{
    pdl_entry();
    constexpr int TT = kTailThreads / G, NW = TT / 32;
    using Key = typename tail_key<WORDS>::type;
    constexpr int HW = tail_hist<WORDS>();
    __shared__ uint32_t s_hist[G][HW];   // 256 bins, or a small box's cells
    __shared__ uint32_t s_list[WORDS ? G : 1][kList];
    __shared__ uint16_t s_queue[kTailThreads / 32][kQueue];
    __shared__ int s_tile[G], s_next[G], s_pick[G], s_before[G], s_nlist[G], s_nk[G][NW];
    __shared__ uint32_t s_res[G];
    __shared__ int s_red[G][3][NW];
    __shared__ unsigned long long s_min[G];   // order key of the least lambda_i of the group's tiles
    const int tid = threadIdx.x, lane = tid & 31;
    const int g = tid / TT, lt = tid - g * TT, warp = lt >> 5;
    uint32_t* const hist = s_hist[g];
    uint32_t* const list = s_list[WORDS ? g : 0];
    uint16_t* const queue = s_queue[tid >> 5];
    // each warp appends its keys to its own stretch
    Key* const kbuf = reinterpret_cast<Key*>(keys) + ((int64_t)(blockIdx.x * G + g) * NW + warp) * key_seg;
    constexpr int d = 2;

    for (int b = tid; b < G * HW; b += kTailThreads) (&s_hist[0][0])[b] = 0u;
    if (tid < G) s_min[tid] = ~0ull;
    __syncthreads();
    const int rho = zpar[0];   // S < lambda iff rank < rho

    // least x_1 - x_0 over a box's trials with S < c (one past its largest: none)
    auto least_diff = [&](float c, int lo0, int hi0, int lo1, int hi1) {
        int dl = hi1 - lo0 + 1;
        for (int x0 = lo0 + lane; x0 <= hi0; x0 += 32) {
            const float* row = S_g + x0 * n1p;
            int lo = 0, hi = n_max + 1;   // least x_1 with S < c
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if (row[mid] < c) hi = mid;
                else lo = mid + 1;
            }
            if (lo <= hi1) dl = min(dl, max(lo, lo1) - x0);   // (a row without such trials leaves d alone)
        }
        return __reduce_min_sync(0xffffffffu, dl);
    };
    // the m-th smallest of the list's nl words
    auto word_of_list = [&](int nl, int m) {
        for (int j = lt; j < nl; j += TT) {
            const uint32_t w = list[j];
            int rank = 0;
            for (int q = 0; q < nl; ++q) {
                const uint32_t u = list[q];
                rank += (u < w || (u == w && q < j)) ? 1 : 0;
            }
            if (rank == m - 1) s_res[g] = w;
        }
        tile_sync<TT, G>(g);
        return s_res[g];
    };
    // the m-th smallest of the words that each(f) hands to f: four 8-bit digits
    auto word_by_digits = [&](int m, auto each) {
        uint32_t prefix = 0u, pmask = 0u;
        for (int sh = 24; sh >= 0; sh -= 8) {
            each([&](uint32_t x) {
                if ((x & pmask) == prefix) atomicAdd(&hist[(x >> sh) & 0xFFu], 1u);
            });
            tile_sync<TT, G>(g);
            if (warp == 0) {
                int before = 0;
                const int digit = warp_pick256<true>(hist, m, lane, &before);
                if (lane == 0) {
                    s_pick[g] = digit;
                    s_before[g] = before;
                }
            }
            tile_sync<TT, G>(g);
            prefix |= (uint32_t)s_pick[g] << sh;
            pmask |= 0xFFu << sh;
            m -= s_before[g];
        }
        return prefix;
    };

    if (lt == 0) s_next[g] = atomicAdd(counter, 1);
    for (;;) {
        if (lt == 0) {
            s_tile[g] = s_next[g];
            s_nlist[g] = 0;
        }
        tile_sync<TT, G>(g);
        const int64_t i = s_tile[g];
        if (i >= T.n_tiles) break;
        if (lt == 0) s_next[g] = atomicAdd(counter, 1);   // the next tile, fetched while this one runs
        const int K = T.K[i];
        const int v0 = T.center_idx[i * d + 0];
        const int v1 = T.center_idx[i * d + 1];
        // device-side argument checks: K_i in [1, K_max of the set], axis indices in range
        const bool bad = (K < 1) || (K > K_tiles) || v0 < 0 || v0 >= T.n_axis[0] || v1 < 0 ||
                         v1 >= T.n_axis[1];
        const int Kc = bad ? 0 : K;
        const int a0 = T.axis_off[0] + (bad ? 0 : v0);
        const int a1 = T.axis_off[1] + (bad ? 0 : v1);
        const int ks = bad ? 0 : o.ksel[i];
        const uint8_t* const c0 = cnt + (int64_t)a0 * k_stride;
        const uint8_t* const c1 = cnt + (int64_t)a1 * k_stride;
        int r_acc = 0, x0_acc = 0, x1_acc = 0;
        double lam_i = -INFINITY;
        uint32_t c_i = 0u;
        // the tile's reachable counts; differences of its trials.  Every byte 0x80 - d +
        // (x_1 - x_0) stays in 0 .. 255 for d = dmin + 1 .. dmax + 1
        const int lo0 = (int)min(bb[a0], (uint32_t)n_max), hi0 = (int)min(bb[NA + a0], (uint32_t)n_max);
        const int lo1 = (int)min(bb[a1], (uint32_t)n_max), hi1 = (int)min(bb[NA + a1], (uint32_t)n_max);
        const int w1 = hi1 - lo1 + 1, nbox = (hi0 - lo0 + 1) * w1;
        const int dmin = lo1 - hi0, dmax = hi1 - lo0;
        if (nbox <= HW) {   // count the box's cells; each thread then takes the ranks of its own
            constexpr int PER = HW / TT;
            uint32_t own_h[PER];
            int own_r[PER];
            const int base = lo0 * w1 + lo1;
            for (int k = lt * 16; k < Kc; k += TT * 16) {   // k + 16 <= k_stride
                const uint4 u0 = *reinterpret_cast<const uint4*>(c0 + k);
                const uint4 u1 = *reinterpret_cast<const uint4*>(c1 + k);
                const uint32_t y0[4] = {u0.x, u0.y, u0.z, u0.w}, y1[4] = {u1.x, u1.y, u1.z, u1.w};
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    const int x0 = (int)((y0[j >> 2] >> (8 * (j & 3))) & 0xFFu);
                    const int x1 = (int)((y1[j >> 2] >> (8 * (j & 3))) & 0xFFu);
                    if (k + j < Kc) atomicAdd(&hist[x0 * w1 + x1 - base], 1u);
                }
            }
            tile_sync<TT, G>(g);
#pragma unroll
            for (int t = 0; t < PER; ++t) {
                const int j = lt + t * TT, row = j / w1, x0 = lo0 + row, x1 = lo1 + j - row * w1;
                own_h[t] = hist[j];
                own_r[t] = own_h[t] ? (int)__ldg(rank_g + x0 * n1p + x1) : 0x7FFFFFFF;
                const int rej = own_r[t] < rho ? (int)own_h[t] : 0;
                r_acc += rej;
                x0_acc += rej * x0;
                x1_acc += rej * x1;
                hist[j] = 0u;
            }
            if (ks >= 1) {
                int B = 0, kr = ks;
#pragma unroll
                for (int phase = 0; phase < 2; ++phase) {   // the bin, then the rank in the bin
                    tile_sync<TT, G>(g);
#pragma unroll
                    for (int t = 0; t < PER; ++t)
                        if (own_h[t] && (phase == 0 || (own_r[t] >> bin_shift) == B))
                            atomicAdd(&hist[phase ? own_r[t] & ((1 << bin_shift) - 1) : own_r[t] >> bin_shift],
                                      own_h[t]);
                    tile_sync<TT, G>(g);
                    if (warp == 0) {
                        int before = 0;
                        const int b = warp_pick256<true>(hist, kr, lane, &before);
                        if (lane == 0) {
                            s_pick[g] = b;
                            s_before[g] = before;
                        }
                    }
                    tile_sync<TT, G>(g);
                    B = phase ? (B << bin_shift) + s_pick[g] : s_pick[g];
                    kr -= s_before[g];
                }
                lam_i = (double)vor_g[B];
                if (WORDS) {
                    // the words of the trials of rank B: those of its cells, one or two nearly
                    // always, which four trials' bytes are compared with at once
                    const int ntc = pos_g[n_cells + B], t0 = pos_g[B], t1 = ntc > 1 ? pos_g[B + 1] : t0;
                    const uint32_t p0 = (uint32_t)(t0 / n1p) * 0x01010101u, q0 = (uint32_t)(t0 % n1p) * 0x01010101u;
                    const uint32_t p1 = (uint32_t)(t1 / n1p) * 0x01010101u, q1 = (uint32_t)(t1 % n1p) * 0x01010101u;
                    uint32_t* const more = reinterpret_cast<uint32_t*>(kbuf - (int64_t)warp * key_seg);   // all warps'
                    for (int k = lt * 16; k < Kc; k += TT * 16) {
                        const uint4 u0 = *reinterpret_cast<const uint4*>(c0 + k);
                        const uint4 u1 = *reinterpret_cast<const uint4*>(c1 + k);
                        const uint32_t y0[4] = {u0.x, u0.y, u0.z, u0.w}, y1[4] = {u1.x, u1.y, u1.z, u1.w};
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            // a byte is zero where the trial lies in the cell
                            const uint32_t z0 = (y0[q] ^ p0) | (y1[q] ^ q0), z1 = (y0[q] ^ p1) | (y1[q] ^ q1);
                            const uint32_t hz = (((z0 - 0x01010101u) & ~z0) | ((z1 - 0x01010101u) & ~z1)) & 0x80808080u;
                            if (hz == 0u && ntc <= 2) continue;
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                const int cell = (int)((y0[q] >> (8 * j)) & 0xFFu) * n1p +
                                                 (int)((y1[q] >> (8 * j)) & 0xFFu);
                                const int kt = k + 4 * q + j;
                                const bool tie = ntc <= 2 ? cell == t0 || cell == t1
                                                          : (int)__ldg(rank_g + min(cell, n_cells - 1)) == B;
                                if (!tie || kt >= Kc) continue;
                                const int at = atomicAdd(&s_nlist[g], 1);
                                if (at < kList) list[at] = W[kt];
                                else more[at - kList] = W[kt];   // (a group's stretches hold all its trials)
                            }
                        }
                    }
                    tile_sync<TT, G>(g);
                    const int nl = s_nlist[g];
                    c_i = nl <= kList ? word_of_list(nl, kr) : word_by_digits(kr, [&](auto f) {
                        for (int k = lt; k < nl; k += TT) f(k < kList ? list[k] : more[k - kList]);
                    });
                }
            }
        } else {
            // d: the least difference of the trials with S < cap, the normal quantile (+inf: all)
            float cap = -INFINITY;
            int d_test = dmax + 1;
            if (ks >= 1) {
                const float share = ((float)ks + 3.0f * sqrtf((float)ks) + 1.0f) / (float)K;
                const float fn = (float)n_max, q0 = (float)o.sig[a0], q1 = (float)o.sig[a1];
                // S = (p_0 - p_1) / sqrt(2 pb (1 - pb) / n) to first order in the counts' shares
                // (below the diagonal the spread at a fixed pb does, and leaves fewer candidates)
                const float pb = 0.5f * (q0 + q1), v = pb * (1.0f - pb), den = rsqrtf(v * 2.0f / fn);
                const float e = q1 > q0 ? (q1 - q0) * (1.0f - 2.0f * pb) / (4.0f * v) : 0.0f;
                const float sd = den * sqrtf(((1.0f + e) * (1.0f + e) * q0 * (1.0f - q0) +
                                              (1.0f - e) * (1.0f - e) * q1 * (1.0f - q1)) / fn);
                cap = (q0 - q1) * den + normcdfinvf(fminf(share, 0.9f)) * sd + 0.05f;
                if (!(cap < INFINITY)) cap = INFINITY;   // NaN too
                d_test = max(least_diff(cap, lo0, hi0, lo1, hi1), dmin);
            }
            // rejections that are no candidates: counted by bytes, as k_sim_count does, or
            // (n_max > 126) made candidates
            int d_rej = dmax + 1;
            if (cap < lambda_up) {
                for (int x0 = lo0 + lane; x0 <= hi0; x0 += 32) {
                    const int cut = (int)zcut[x0];
                    if (cut <= hi1) d_rej = min(d_rej, max(cut, lo1) - x0);
                }
                d_rej = __reduce_min_sync(0xffffffffu, d_rej);
                if (n_max > 126) d_test = min(d_test, max(d_rej, dmin));
            }
            const bool bytes = d_rej < d_test;
            const int rho_c = bytes ? 0 : rho;   // ranks of the rejections among the candidates
            if (bytes)
                count_rejections(c1, c0, c0 + (int64_t)NA * k_stride, Kc, lt * 16, TT * 16, &r_acc, &x1_acc, &x0_acc);
            const bool wide = dmax - dmin > 126;
            for (int tries = 0;; ++tries) {
                const bool all = wide || d_test <= dmin;   // every trial, without the test
                const uint32_t zc = 0x80808080u - (uint32_t)d_test * 0x01010101u;
                int qn = 0, wk = 0;   // queued candidates, kept keys of this warp
                for (int st = 0; st * (TT * 32) < Kc; ++st) {   // group-uniform
                    // thirty-two consecutive trials per thread and step; bit 8 j + q of a
                    // thread's candidate word is trial 4 q + j.  kb: first trial of the warp
                    // in the queue's block of 64 steps
                    const int kb = (st & ~63) * (TT * 32) + warp * 1024, stq = st & 63;
                    const int kw = kb + stq * (TT * 32) + lane * 32;
                    uint32_t m = 0u;
                    if (kw < Kc) {
                            if (all) {
                            m = 0xFFFFFFFFu;
                        } else {
                            const bool two = kw + 16 < Kc;   // the second sixteen lie in the row
                            const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
                            const uint4 xa = *reinterpret_cast<const uint4*>(c1 + kw);
                            const uint4 xb = two ? *reinterpret_cast<const uint4*>(c1 + kw + 16) : zero;
                            uint32_t t[8] = {xa.x, xa.y, xa.z, xa.w, xb.x, xb.y, xb.z, xb.w};
                            const uint4 ya = *reinterpret_cast<const uint4*>(c0 + kw);
                            const uint4 yb = two ? *reinterpret_cast<const uint4*>(c0 + kw + 16) : zero;
                            const uint32_t y[8] = {ya.x, ya.y, ya.z, ya.w, yb.x, yb.y, yb.z, yb.w};
#pragma unroll
                            for (int q = 0; q < 8; ++q) t[q] = t[q] - y[q] + zc;
#pragma unroll
                            for (int q = 0; q < 8; ++q) m |= (t[q] >> (7 - q)) & (0x01010101u << q);
                        }
                        if (kw + 32 > Kc) m &= trials_below(Kc - kw);
                    }
                    const int nm = __popc(m);
                    int incl = nm;
#pragma unroll
                    for (int off = 1; off < 32; off <<= 1) {
                        const int y = __shfl_up_sync(0xffffffffu, incl, off);
                        if (lane >= off) incl += y;
                    }
                    const int total = __shfl_sync(0xffffffffu, incl, 31);
                    const bool flush = stq == 63 || (st + 1) * (TT * 32) >= Kc;
                    const int ent = (stq << 10) | (lane << 5);   // entry: step (6 bits), lane, bit
                    int done = 0;   // candidates of this step queued so far
                    do {
                        // the lanes whose candidates fit the queue (a prefix of those left)
                        const bool mine = incl - nm >= done && incl - done <= kQueue - qn;
                        const unsigned who = __ballot_sync(0xffffffffu, mine);
                        const int upto = __shfl_sync(0xffffffffu, incl, 31 - __clz(who));
                        if (mine) {
                            uint16_t* at = queue + qn + (incl - nm - done);
                            while (m) {
                                const int b = __ffs(m) - 1;
                                m &= m - 1u;
                                *at++ = (uint16_t)(ent | b);
                            }
                        }
                        qn += upto - done;
                        done = upto;
                        __syncwarp();
                        while (qn >= 32 || (flush && done == total && qn > 0)) {
                            const int n = min(qn, 32);
                            qn -= n;
                            const int ev = queue[qn + (lane < n ? lane : 0)];
                            const int k =
                                kb + (ev >> 10) * (TT * 32) + (ev & 0x3E0) + ((ev & 7) << 2) + ((ev >> 3) & 3);
                            const int x0 = (int)__ldg(c0 + k), x1 = (int)__ldg(c1 + k);
                            int r = (int)__ldg(rank_g + min(x0 * n1p + x1, n_cells - 1));
                            if (lane >= n) r = 0x7FFFFFFF;
                            const int rej = r < rho_c ? 1 : 0;
                            r_acc += rej;
                            x0_acc += rej ? x0 : 0;
                            x1_acc += rej ? x1 : 0;
                            if (ks >= 1) {
                                if (lane < n) {
                                    // WORDS: the trial by its place among the warp's (below 2^17)
                                    if (WORDS)
                                        kbuf[wk + lane] =
                                            (Key)(((uint32_t)r << 17) |
                                                  (uint32_t)(((st & ~63) + (ev >> 10)) * 1024 + ((k - kb) & 1023)));
                                    else kbuf[wk + lane] = (Key)r;
                                    atomicAdd(&hist[r >> bin_shift], 1u);
                                }
                                wk += n;
                            }
                            __syncwarp();   // the queue's entries read before the next round writes
                        }
                    } while (done < total);
                }
                if (ks < 1) break;
                if (lane == 0) s_nk[g][warp] = wk;
                tile_sync<TT, G>(g);
                int nk = 0;
#pragma unroll
                for (int w2 = 0; w2 < NW; ++w2) nk += s_nk[g][w2];
                if (nk < ks && !all) {   // fewer candidates than k_i: again from a lower difference
                    for (int b = lt; b < 256; b += TT) hist[b] = 0u;
                    d_test = tries < 3 ? max(d_test - 1 - tries, dmin) : dmin;
                    if (!bytes) r_acc = x0_acc = x1_acc = 0;
                    tile_sync<TT, G>(g);
                    continue;
                }
                // the ks-th smallest rank: its bin, then the rank within the bin
                auto key_rank = [&](int k) { return (uint32_t)kbuf[k] >> (WORDS ? 17 : 0); };
                auto key_word = [&](int k) {
                    const int at = (int)((uint32_t)kbuf[k] & 0x1FFFFu);
                    return W[(at >> 10) * (TT * 32) + warp * 1024 + (at & 1023)];
                };
                if (warp == 0) {
                    int before = 0;
                    const int b = warp_pick256<true>(hist, ks, lane, &before);
                    if (lane == 0) {
                        s_pick[g] = b;
                        s_before[g] = before;
                    }
                }
                tile_sync<TT, G>(g);
                const int B = s_pick[g], kr = ks - s_before[g];
                for (int k = lane; k < wk; k += 32) {
                    const uint32_t r = key_rank(k);
                    if ((int)(r >> bin_shift) == B) atomicAdd(&hist[r & ((1u << bin_shift) - 1u)], 1u);
                }
                tile_sync<TT, G>(g);
                if (warp == 0) {
                    int before = 0;
                    const int b = warp_pick256<true>(hist, kr, lane, &before);
                    if (lane == 0) {
                        s_pick[g] = (B << bin_shift) + b;
                        s_before[g] = kr - before;   // order of the ks-th trial among the rank's trials
                    }
                }
                tile_sync<TT, G>(g);
                const int rstar = s_pick[g], mrem = s_before[g];
                const float lam = vor_g[rstar];
                lam_i = (double)lam;
                // a trial left out might be smaller, or (words) of the same rank: again with every
                // trial up to this one
                if (!all && !(tries == 0 && (WORDS ? lam < cap : lam <= cap))) {   // (S >= cap left out at first)
                    float sigma = INFINITY;   // the least S of a trial left out
                    for (int x0 = lo0 + lane; x0 <= hi0; x0 += 32) {
                        const int x1 = min(x0 + d_test - 1, hi1);
                        if (x1 >= lo1) sigma = fminf(sigma, S_g[x0 * n1p + x1]);
                    }
#pragma unroll
                    for (int o2 = 16; o2 > 0; o2 >>= 1) sigma = fminf(sigma, __shfl_xor_sync(0xffffffffu, sigma, o2));
                    if (!(WORDS ? lam < sigma : lam <= sigma)) {
                        d_test = max(least_diff(WORDS ? nextafterf(lam, INFINITY) : lam, lo0, hi0, lo1, hi1), dmin);
                        if (!bytes) r_acc = x0_acc = x1_acc = 0;
                        tile_sync<TT, G>(g);
                        continue;
                    }
                }
                if (WORDS) {
                    // the mrem-th smallest word among the trials of rank rstar
                    for (int k = lane; k < wk; k += 32)
                        if ((int)key_rank(k) == rstar) {
                            const int at = atomicAdd(&s_nlist[g], 1);
                            if (at < kList) list[at] = key_word(k);
                        }
                    tile_sync<TT, G>(g);
                    const int nl = s_nlist[g];
                    c_i = nl <= kList ? word_of_list(nl, mrem) : word_by_digits(mrem, [&](auto f) {
                        for (int k = lane; k < wk; k += 32)
                            if ((int)key_rank(k) == rstar) f(key_word(k));
                    });
                }
                break;
            }
        }
        r_acc = tail_warp_sum(r_acc);
        x0_acc = tail_warp_sum(x0_acc);
        x1_acc = tail_warp_sum(x1_acc);
        if (lane == 0) {
            s_red[g][0][warp] = r_acc;
            s_red[g][1][warp] = x0_acc;
            s_red[g][2][warp] = x1_acc;
        }
        tile_sync<TT, G>(g);
        if (lt < d) {   // lane a: arm a's outputs, lane 0 the tile's
            int64_t Rt = 0, X = 0;
            for (int w2 = 0; w2 < NW; ++w2) {
                Rt += s_red[g][0][w2];
                X += s_red[g][1 + lt][w2];
            }
            if (o.Xrej) o.Xrej[i * d + lt] = X;
            if (o.score) {
                const double sg = bad ? NAN : o.sig[lt == 0 ? a0 : a1];
                o.score[i * d + lt] = (double)X - (double)n_max * sg * (double)Rt;
            }
            if (lt == 0) {
                if (bad) atomicOr(err, CSE_ERR_BAD_K);
                if (o.R) o.R[i] = Rt;
                if (o.cp_key)   // the tile's (K, R) in the Clopper-Pearson memo, as k_cp_mark would
                    o.cp_slot[i] = cp_memo_insert(((unsigned long long)(uint32_t)K << 32) | (uint32_t)Rt, o.cp_key,
                                                  o.cp_cap, o.cp_list, o.cp_nkeys);
                o.lam_tile[i] = lam_i;
                s_min[g] = min(s_min[g], order_key(lam_i));
                if (WORDS && c_tile) c_tile[i] = c_i;
            }
        }
        tile_sync<TT, G>(g);
    }
    __syncthreads();   // every group done before the queue is reset
    unsigned long long mine = ~0ull;
    if (tid == 0)
        for (int q = 0; q < G; ++q) mine = min(mine, s_min[q]);
    queue_reset_min(counter, o.min_key, mine, o.min_out, (int)gridDim.x);
}

// A warp's keys: its 1,024 trials of every step.
template <int G>
int32_t tail_key_seg(int32_t K_tiles)
{
    constexpr int TT = kTailThreads / G;
    return (K_tiles + TT * 32 - 1) / (TT * 32) * 1024;
}

template <bool WORDS, int G>
int reserve_tail(cse_ctx* c, const TileArgs& T, int32_t K_tiles, cudaStream_t s)
{
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_sim_tail<WORDS, G>, kTailThreads, 0) != cudaSuccess ||
        per_sm < 1) {
        cudaGetLastError();
        return CSE_CUDA_ERROR;
    }
    c->tail_grid = std::min<int64_t>((int64_t)per_sm * c->num_sms, (T.n_tiles + G - 1) / G);
    const size_t bytes =
        sizeof(typename tail_key<WORDS>::type) * (kTailThreads / 32) * (size_t)tail_key_seg<G>(K_tiles);
    return cse_reserve_keys(c, bytes, &c->tail_grid, s);
}

template <bool WORDS, int G>
int launch_tail(cse_ctx* c, const TileArgs& T, int32_t NA, int32_t k_stride, int32_t K_tiles, const SimOut& o,
                uint32_t* c_tile, cudaStream_t s)
{
    auto kern = k_sim_tail<WORDS, G>;
    const int32_t key_seg = tail_key_seg<G>(K_tiles);
    int sh = 0;   // ranks per bin: at most 256 bins, at most 128 ranks a bin (n_cells <= 129^2)
    while (((c->n_cells - 1) >> sh) > 255) ++sh;
    if (o.min_out) c->min_folded = true;
    if (o.cp_key) c->cp_marked = true;
    cse_prof_begin(c, KID_SIM_ZTEST, s);
    cse_launch(c->pdl, kern, dim3((unsigned)c->tail_grid), dim3(kTailThreads), 0, s, T, c->D.n_max, c->cnt, NA,
               k_stride, K_tiles, c->rank_tab, c->S_tab, c->val_of_rank, c->cell_of_pos, c->n_cells, c->n1p, sh, c->bb,
               c->zpar, c->zcut, c->z_lambda, c->tb, o, c_tile, c->keys, key_seg, c->counter, c->err);
    cse_prof_end(c, s);
    c->launches += 1;
    return cudaGetLastError() == cudaSuccess ? CSE_OK : CSE_CUDA_ERROR;
}

// Tiles a block (wider groups for the largest K: fewer keys, and a trial's place within a
// warp below 2^17).
template <bool WORDS>
int tail_groups(const cse_ctx* c, const TileArgs& T, int32_t K_tiles)
{
    const int64_t key_bytes = (int64_t)K_tiles * (WORDS ? 4 : 2);
    if (T.n_tiles < 8 * (int64_t)c->num_sms || K_tiles > (1 << 18)) return 1;
    if (T.n_tiles < 32 * (int64_t)c->num_sms || key_bytes > (1 << 17)) return 2;
    return 4;
}

template <bool WORDS>
int launch_groups(cse_ctx* c, const TileArgs& T, int32_t NA, int32_t k_stride, int32_t K_tiles, const SimOut& o,
                  uint32_t* c_tile, cudaStream_t s)
{
    switch (tail_groups<WORDS>(c, T, K_tiles)) {
    case 1: return launch_tail<WORDS, 1>(c, T, NA, k_stride, K_tiles, o, c_tile, s);
    case 2: return launch_tail<WORDS, 2>(c, T, NA, k_stride, K_tiles, o, c_tile, s);
    default: return launch_tail<WORDS, 4>(c, T, NA, k_stride, K_tiles, o, c_tile, s);
    }
}

template <bool WORDS>
int reserve_groups(cse_ctx* c, const TileArgs& T, int32_t K_tiles, cudaStream_t s)
{
    switch (tail_groups<WORDS>(c, T, K_tiles)) {
    case 1: return reserve_tail<WORDS, 1>(c, T, K_tiles, s);
    case 2: return reserve_tail<WORDS, 2>(c, T, K_tiles, s);
    default: return reserve_tail<WORDS, 4>(c, T, K_tiles, s);
    }
}

// Rejections alone: a group of TT threads per tile, sixteen trials a thread and step.
template <bool TWO, int TT>
__global__ void __launch_bounds__(256)
    k_sim_count(TileArgs T, int32_t n_max, const uint8_t* __restrict__ cnt, int32_t NA, int32_t k_stride,
                int32_t K_tiles, const uint8_t* __restrict__ zcut, SimOut o, int32_t* __restrict__ err)
{
    pdl_entry();
    constexpr int NW = TT / 32, G = 256 / TT, d = TWO ? 2 : 1;
    __shared__ int s_red[G][3][NW];
    const int tid = threadIdx.x, lane = tid & 31, g = tid / TT, lt = tid - g * TT, warp = lt >> 5;
    const uint32_t b1 = TWO ? 0u : (uint32_t)zcut[0] * 0x01010101u;
    for (int64_t i0 = (int64_t)blockIdx.x * G; i0 < T.n_tiles; i0 += (int64_t)gridDim.x * G) {   // block-uniform
        const int64_t i = i0 + g;
        const bool live = i < T.n_tiles;
        const int K = live ? T.K[i] : 0;
        const int v0 = live ? T.center_idx[i * d] : 0, v1 = (TWO && live) ? T.center_idx[i * d + 1] : 0;
        // device-side argument checks: K_i in [1, K_max of the set], axis indices in range
        const bool bad = (K < 1) || (K > K_tiles) || v0 < 0 || v0 >= T.n_axis[0] ||
                         (TWO && (v1 < 0 || v1 >= T.n_axis[1]));
        const int Kc = bad ? 0 : K;
        const int a0 = T.axis_off[0] + (bad ? 0 : v0), a1 = TWO ? T.axis_off[1] + (bad ? 0 : v1) : a0;
        const uint8_t* const c0 = cnt + (int64_t)a0 * k_stride;
        const uint8_t* const c1 = cnt + (int64_t)a1 * k_stride;   // the tested row
        const uint8_t* const cb = c0 + (int64_t)NA * k_stride;    // b(x_0) (two arms)
        int R = 0, X0 = 0, X1 = 0;
        count_rejections<TWO>(c1, c0, cb, Kc, lt * 16, TT * 16, &R, &X1, &X0, b1);
        const int r = tail_warp_sum(R), x1 = tail_warp_sum(X1), x0 = TWO ? tail_warp_sum(X0) : x1;
        if (lane == 0) {
            s_red[g][0][warp] = r;
            s_red[g][1][warp] = x0;
            s_red[g][2][warp] = x1;
        }
        if (TT == 32) __syncwarp();
        else __syncthreads();
        if (live && lt < d) {   // lane a: arm a's outputs, lane 0 the tile's
            int64_t Rt = 0, X = 0;
            for (int w2 = 0; w2 < NW; ++w2) {
                Rt += s_red[g][0][w2];
                X += s_red[g][1 + lt][w2];
            }
            if (lt == 0) {
                if (bad) atomicOr(err, CSE_ERR_BAD_K);
                if (o.R) o.R[i] = Rt;
            }
            if (o.Xrej) o.Xrej[i * d + lt] = X;
            if (o.score) {
                const double sg = bad ? NAN : o.sig[lt == 0 ? a0 : a1];
                o.score[i * d + lt] = (double)X - (double)n_max * sg * (double)Rt;
            }
        }
        if (TT == 32) __syncwarp();
        else __syncthreads();
    }
}

template <bool TWO, int TT>
int launch_count(cse_ctx* c, const TileArgs& T, int32_t NA, int32_t k_stride, int32_t K_tiles, const SimOut& o,
                 cudaStream_t s)
{
    auto kern = k_sim_count<TWO, TT>;
    constexpr int G = 256 / TT;
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 256, 0) != cudaSuccess || per_sm < 1) {
        cudaGetLastError();
        return CSE_CUDA_ERROR;
    }
    // blocks in turn over the tiles: several rounds each, so that ragged K evens out
    int64_t grid = (T.n_tiles + G - 1) / G;
    if (grid > 8 * (int64_t)per_sm * c->num_sms) grid = 8 * (int64_t)per_sm * c->num_sms;
    cse_prof_begin(c, KID_SIM_ZTEST, s);
    cse_launch(c->pdl, kern, dim3((unsigned)grid), dim3(256), 0, s, T, c->D.n_max, c->cnt, NA, k_stride, K_tiles,
               c->zcut, o, c->err);
    cse_prof_end(c, s);
    c->launches += 1;
    return cudaGetLastError() == cudaSuccess ? CSE_OK : CSE_CUDA_ERROR;
}

}  // namespace

int cse_launch_sim_count(cse_ctx* c, const TileArgs& T, int32_t NA, int32_t k_stride, int32_t K_tiles, const SimOut& o,
                         cudaStream_t s)
{
    // a warp per tile once every resident warp has one, else a block of 256
    const bool many = T.n_tiles >= 32 * (int64_t)c->num_sms;
    if (c->D.stat == CSE_STAT_TWO_ARM_POOLED_Z)
        return many ? launch_count<true, 32>(c, T, NA, k_stride, K_tiles, o, s)
                    : launch_count<true, 256>(c, T, NA, k_stride, K_tiles, o, s);
    return many ? launch_count<false, 32>(c, T, NA, k_stride, K_tiles, o, s)
                : launch_count<false, 256>(c, T, NA, k_stride, K_tiles, o, s);
}

int cse_launch_sim_tail(cse_ctx* c, const TileArgs& T, int32_t NA, int32_t k_stride, int32_t K_tiles, const SimOut& o,
                        bool words, uint32_t* c_tile, cudaStream_t s)
{
    return words ? launch_groups<true>(c, T, NA, k_stride, K_tiles, o, c_tile, s)
                 : launch_groups<false>(c, T, NA, k_stride, K_tiles, o, c_tile, s);
}

int cse_tail_reserve(cse_ctx* c, const TileArgs& T, int32_t K_tiles, bool words, cudaStream_t s)
{
    return words ? reserve_groups<true>(c, T, K_tiles, s) : reserve_groups<false>(c, T, K_tiles, s);
}
