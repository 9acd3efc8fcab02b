// uniforms.cu -- common random numbers, success thresholds, axis count tables
// and statistic tables.
//
// CRN (Sec. 7.3 of the paper: simulations may be shared across tiles as long
// as each tile's own simulations are i.i.d.): sim k, arm a, patient j uses word
// j mod 4 of Philox4x32-10(counter (k, a, j/4, 0), key = seed), and the patient
// succeeds iff u < t(theta).  The count tables draw the words themselves
// (k_counts); the plain z-test path keeps each (sim, arm) row sorted in memory
// (k_uniforms), where a success count is a binary search.
#include <cuda_runtime.h>

#include <cstring>

#include "cse_internal.cuh"

namespace {

// what a count table holds (see k_counts)
constexpr int kCountsRaw = 0, kCountsNib = 1, kCountsMapped = 2;

// Success threshold and sigmoid of axis value i of a tile set (flattened over
// the arms' axes).
__device__ __forceinline__ void threshold_of(int i, uint32_t* __restrict__ thr, double* __restrict__ sig,
                                             const TileArgs& T)
{
    int a = 0;
    while (a + 1 < T.d && i >= T.axis_off[a + 1]) ++a;
    const double th = T.axis[a][i - T.axis_off[a]];
    thr[i] = success_threshold(th);
    if (sig) sig[i] = 1.0 / (1.0 + exp(-th));
}

// One warp per (arm, sim) row: lane L generates and holds elements L*E .. L*E+E-1
// (E = 32-padded power of two / 32), and a bitonic network over the 32*E keys
// (in-register pairs when the partner distance is below E, warp shuffles above)
// sorts the row; pad keys (all ones) sort last and are not written.
//
// The randomised test's tie-break word of every sim rides on the first blocks, one
// thread each (tb; word 0 of Philox4x32-10(counter (k, 0, 0, 1), key = seed), the
// patients' draws using counter word 3 = 0).
template <int E>
__global__ void __launch_bounds__(256) k_uniforms(uint32_t* __restrict__ U, int32_t K_max, int32_t d,
                                                  int32_t n_max, uint32_t key0, uint32_t key1,
                                                  uint32_t* __restrict__ tb)
{
    pdl_entry();
    const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (tb && g < K_max) {
        u32x4 c = {(uint32_t)g, 0u, 0u, 1u};
        tb[g] = philox4x32_10(c, key0, key1).x;
    }
    constexpr int NP = 32 * E;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t row = (int64_t)blockIdx.x * 8 + warp;   // row = a * K_max + k
    if (row >= (int64_t)d * K_max) return;                  // the whole warp leaves together
    const uint32_t a = (uint32_t)(row / K_max), k = (uint32_t)(row % K_max);
    uint32_t v[E];
    u32x4 w = {0u, 0u, 0u, 0u};
#pragma unroll
    for (int i = 0; i < E; ++i) {
        const int e = lane * E + i;
        if (i == 0 || (e & 3) == 0) {   // word j/4 of Philox(k, a, j/4, 0) holds element j
            u32x4 c = {k, a, (uint32_t)(e >> 2), 0u};
            w = philox4x32_10(c, key0, key1);
        }
        const uint32_t u = ((e & 3) == 0) ? w.x : ((e & 3) == 1) ? w.y : ((e & 3) == 2) ? w.z : w.w;
        v[i] = (e < n_max) ? u : 0xFFFFFFFFu;
    }
#pragma unroll
    for (int kk = 2; kk <= NP; kk <<= 1) {
#pragma unroll
        for (int j = kk >> 1; j > 0; j >>= 1) {
            if (j >= E) {
#pragma unroll
                for (int i = 0; i < E; ++i) {
                    const int e = lane * E + i;
                    const uint32_t p = __shfl_xor_sync(0xffffffffu, v[i], j / E);
                    const bool keep_min = ((e & kk) == 0) == ((e & j) == 0);
                    v[i] = keep_min ? (p < v[i] ? p : v[i]) : (p > v[i] ? p : v[i]);
                }
            } else {
#pragma unroll
                for (int i = 0; i < E; ++i) {
                    if ((i & j) == 0) {
                        const int i2 = i | j;
                        const bool up = ((lane * E + i) & kk) == 0;
                        const uint32_t x = v[i], y = v[i2];
                        const uint32_t lo = x < y ? x : y, hi = x < y ? y : x;
                        v[i] = up ? lo : hi;
                        v[i2] = up ? hi : lo;
                    }
                }
            }
        }
    }
    uint32_t* out = U + row * n_max;
#pragma unroll
    for (int i = 0; i < E; ++i) {
        const int e = lane * E + i;
        if (e < n_max) out[e] = v[i];
    }
}

// Success threshold and sigmoid (for the score's grad A) of every axis value.  With
// Z.S set (z-test calls that do not run the cell histogram) the last block finds
// the call's constants: the number of cells with S < lambda (Z.pos), and per x_0 the least
// x_1 with S < lambda (n_max + 1: none; each row of S falls in x_1).
struct TailArgs {
    const float* S;
    int32_t n_cells, n1p, n_max;   // row length n1p: n_max + 1, or 1 for one arm
    float lambda_up;
    const int32_t* pos;   // the cells sorted by S, or NULL
    int32_t* zpar;
    uint8_t* zcut;        // or NULL
};

__global__ void __launch_bounds__(256) k_thresholds(uint32_t* __restrict__ thr, double* __restrict__ sig, TileArgs T,
                                                    int32_t n_total, TailArgs Z)
{
    pdl_entry();
    if (Z.S && blockIdx.x == gridDim.x - 1) {
        if (Z.pos) {   // the sorted cells (pos): the block's threads search in two rounds
            const int step = (Z.n_cells + (int)blockDim.x - 1) / (int)blockDim.x;
            auto below = [&](int p) { return p < Z.n_cells && Z.S[Z.pos[p]] < Z.lambda_up; };
            const int c1 = __syncthreads_count(below(threadIdx.x * step));   // positions 0, step, ... below lambda
            const int base = c1 > 0 ? (c1 - 1) * step + 1 : 0;
            const int c2 = __syncthreads_count(c1 > 0 && (int)threadIdx.x < step - 1 && below(base + threadIdx.x));
            if (threadIdx.x == 0) Z.zpar[0] = base + c2;
        }
        if (Z.zcut && threadIdx.x < (Z.n1p > 1 ? Z.n1p : 1)) {
            const float* row = Z.S + threadIdx.x * Z.n1p;   // one arm: the table itself is the row
            int lo = 0, hi = Z.n_max + 1;
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if (row[mid] < Z.lambda_up) hi = mid;
                else lo = mid + 1;
            }
            Z.zcut[threadIdx.x] = (uint8_t)lo;
        }
        return;
    }
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_total) return;
    threshold_of(i, thr, sig, T);
}

// Axis count table: cnt[(l * NA + off_a + v) * k_stride + k] = number of the
// first look_n[l] patients of (sim k, arm a) whose uniform is below t(axis_a[v]).
//
// Counts along an arm's rising thresholds are the running sums of a histogram: a
// uniform u counts for every value with t > u, so it adds one at the position
// p(u) = #{t <= u} and the counts are prefix sums.  A block takes 128 sims of one
// arm and a chunk of its values: it draws the sims' Philox words (no sorted rows of
// uniforms in memory), finds p(u) by a table over the top 12 bits and a short binary
// search, adds into a shared-memory histogram of four sims a word (byte lanes: a
// count is at most 128; lane l of every warp owns column l, so no bank conflicts),
// and writes the prefix sums four sims a store.  Per count that is ~2 thread
// instructions instead of a merge step's ~10 on byte loads and stores, and per
// uniform ~30 instead of the 28-step sorting network.  Axis values in any order:
// a chunk whose thresholds do not rise is sorted first.
//
// Bound by issue slots.  With the uniforms' pass and its sort, the count pass they
// replace took: two arms, 256 values each, K = 16,384 26 + 24 us, now 15 us in all; 2^18
// batch (959 values, K = 65,536) 92 + 99, now 49; one arm, 1,500 values, K = 65,536
// 28 + 115, now 54; 4,096 values in random order, K = 8,192 15 + 244, now 44.
//
// MODE kCountsNib (the packed four-arm form): two planes instead of three, plane 0
// the two interim segments' counts in the two halves of a byte (first segment << 4
// | second segment; both at most 15), plane 1 map[final count].  kCountsMapped: a
// second plane holds map[count] for arm 0's values.
constexpr int kCntSims = 128, kCntThreads = 512;

// top bits of a word that index the position table: with three histograms fewer,
// so that two blocks fit an SM's shared memory
template <int SEGS>
constexpr int cnt_lut_bits()
{
    return SEGS > 1 ? 11 : 12;
}

template <int SEGS, int MODE>
__global__ void __launch_bounds__(kCntThreads) k_counts(uint8_t* __restrict__ cnt, const uint32_t* __restrict__ thr,
                                                        TileArgs T, int32_t NA, int32_t K_tiles, int32_t k_stride,
                                                        int2 looks, int32_t n_max, uint32_t key0, uint32_t key1,
                                                        uint32_t* __restrict__ tb, int32_t chunk, int32_t pow2,
                                                        int32_t v_base, const uint8_t* __restrict__ map)
{
    pdl_entry();
    constexpr int NW = kCntThreads / 32, LB = cnt_lut_bits<SEGS>(), LUT = 1 << LB;
    extern __shared__ __align__(16) uint32_t smem[];
    // histogram [SEGS][chunk][32], thresholds [chunk], table, order, then (sorting
    // only, before the histogram is in use) 64-bit keys over the histogram
    uint32_t* delta = smem;
    uint32_t* st = smem + SEGS * chunk * 32;
    uint16_t* perm = reinterpret_cast<uint16_t*>(st + chunk);
    __shared__ __align__(16) uint32_t lut[LUT];   // a bucket's thresholds: those below it | its own << 16
    __shared__ uint32_t s_scan[NW];
    __shared__ uint8_t s_map[MODE != kCountsRaw ? CSE_MAX_NMAX + 1 : 1];
    __shared__ uint32_t s_part[SEGS][NW][32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int a = blockIdx.y, k0 = blockIdx.x * kCntSims, v0 = v_base + blockIdx.z * chunk;
    int na = T.n_axis[0], off = T.axis_off[0];
#pragma unroll
    for (int b = 1; b < CSE_MAX_ARMS; ++b)   // by selection: no runtime index into the argument
        if (a == b) {
            na = T.n_axis[b];
            off = T.axis_off[b];
        }
    // the randomised test's tie-break words (word 0 of Philox(counter (k, 0, 0, 1)))
    if (tb && a == 0 && v0 == 0 && tid < kCntSims && k0 + tid < K_tiles) {
        u32x4 c = {(uint32_t)(k0 + tid), 0u, 0u, 1u};
        tb[k0 + tid] = philox4x32_10(c, key0, key1).x;
    }
    const int nv = min(chunk, na - v0);
    if (nv <= 0) return;   // an arm with fewer chunks
    if (MODE != kCountsRaw)
        for (int i = tid; i <= n_max; i += kCntThreads) s_map[i] = map[i];
    // the chunk's thresholds in rising order
    bool falls = false;
    for (int i = tid; i < nv; i += kCntThreads) {
        const uint32_t t = thr[off + v0 + i];
        st[i] = t;
        perm[i] = (uint16_t)i;
        falls |= i > 0 && thr[off + v0 + i - 1] > t;
    }
    if (__syncthreads_or(falls)) {   // bitonic sort of (threshold, index), padded with all ones
        unsigned long long* key = reinterpret_cast<unsigned long long*>(delta);
        for (int i = tid; i < pow2; i += kCntThreads)
            key[i] = i < nv ? ((unsigned long long)st[i] << 32) | (unsigned)i : ~0ull;
        for (int size = 2; size <= pow2; size <<= 1)
            for (int j = size >> 1; j > 0; j >>= 1) {
                __syncthreads();
                for (int i = tid; i < pow2 / 2; i += kCntThreads) {
                    const int lo = 2 * i - (i & (j - 1)), hi = lo + j;
                    const unsigned long long x = key[lo], y = key[hi];
                    if ((x > y) == ((lo & size) == 0)) {
                        key[lo] = y;
                        key[hi] = x;
                    }
                }
            }
        __syncthreads();
        for (int i = tid; i < nv; i += kCntThreads) {
            st[i] = (uint32_t)(key[i] >> 32);
            perm[i] = (uint16_t)(uint32_t)key[i];
        }
        __syncthreads();
    }
    // the table over the words' top bits: thresholds counted per bucket, then scanned
    constexpr int PER = LUT / kCntThreads;
    for (int i = tid; i < LUT / 4; i += kCntThreads) reinterpret_cast<uint4*>(lut)[i] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
    for (int i = tid; i < nv; i += kCntThreads) atomicAdd(&lut[st[i] >> (32 - LB)], 1u);
    __syncthreads();
    uint32_t own[PER], local = 0u;
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        own[i] = lut[tid * PER + i];
        local += own[i];
    }
    uint32_t incl = local;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) s_scan[warp] = incl;
    __syncthreads();
    uint32_t start = incl - local;
    for (int w = 0; w < warp; ++w) start += s_scan[w];
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        lut[tid * PER + i] = start | (own[i] << 16);
        start += own[i];
    }
    for (int i = tid; i < SEGS * chunk * 8; i += kCntThreads)
        reinterpret_cast<uint4*>(delta)[i] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
    // Philox blocks: lane l draws for sims 4 l + r of the block
    const int nq = (n_max + 3) >> 2;
    for (int t = warp; t < 4 * nq; t += NW) {
        const int r = t & 3, q = t >> 2, k = k0 + 4 * lane + r;
        if (k >= K_tiles) continue;
        const u32x4 c = {(uint32_t)k, (uint32_t)a, (uint32_t)q, 0u};
        const u32x4 w = philox4x32_10(c, key0, key1);
        const uint32_t u4[4] = {w.x, w.y, w.z, w.w};
        int lo[4], hi[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint32_t x = lut[u4[j] >> (32 - LB)];
            lo[j] = (int)(x & 0xFFFFu);
            hi[j] = lo[j] + (int)(x >> 16);
        }
        // one step settles the buckets of at most one threshold, nearly all of them
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int mid = (lo[j] + hi[j]) >> 1;
            const bool up = lo[j] < hi[j] && st[min(mid, nv - 1)] <= u4[j];
            hi[j] = up ? hi[j] : min(hi[j], mid);
            lo[j] = up ? mid + 1 : lo[j];
        }
#pragma unroll
        for (int j = 0; j < 4; ++j)
            while (lo[j] < hi[j]) {
                const int mid = (lo[j] + hi[j]) >> 1;
                if (st[mid] <= u4[j]) lo[j] = mid + 1;
                else hi[j] = mid;
            }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int e = 4 * q + j;
            const int seg = SEGS > 1 ? (e >= looks.x ? 1 : 0) + (e >= looks.y ? 1 : 0) : 0;
            if (e < n_max && lo[j] < nv) atomicAdd(&delta[(seg * chunk + lo[j]) * 32 + lane], 1u << (8 * r));
        }
    }
    __syncthreads();
    // prefix sums down the rows: each warp its stretch, from the sums of those above
    const int per = (nv + NW - 1) / NW, j0 = min(warp * per, nv), j1 = min(j0 + per, nv);
    uint32_t acc[SEGS];
#pragma unroll
    for (int g = 0; g < SEGS; ++g) {
        uint32_t x = 0u;
#pragma unroll 4
        for (int j = j0; j < j1; ++j) x += delta[(g * chunk + j) * 32 + lane];
        s_part[g][warp][lane] = x;
    }
    __syncthreads();
#pragma unroll
    for (int g = 0; g < SEGS; ++g) {
        acc[g] = 0u;
        for (int w = 0; w < warp; ++w) acc[g] += s_part[g][w][lane];
    }
    const int k = k0 + 4 * lane;
    if (k >= k_stride) return;   // k_stride is a multiple of 16
    auto mapped = [&](uint32_t x) {
        return (uint32_t)s_map[x & 0xFFu] | ((uint32_t)s_map[(x >> 8) & 0xFFu] << 8) |
               ((uint32_t)s_map[(x >> 16) & 0xFFu] << 16) | ((uint32_t)s_map[x >> 24] << 24);
    };
    const int64_t plane = (int64_t)NA * k_stride;
#pragma unroll 4
    for (int j = j0; j < j1; ++j) {
        uint8_t* row = cnt + (int64_t)(off + v0 + perm[j]) * k_stride + k;
        uint32_t sum = 0u;
#pragma unroll
        for (int g = 0; g < SEGS; ++g) {
            acc[g] += delta[(g * chunk + j) * 32 + lane];
            sum += acc[g];
            if (MODE != kCountsNib) *reinterpret_cast<uint32_t*>(row + g * plane) = sum;
        }
        if (MODE == kCountsNib) {
            *reinterpret_cast<uint32_t*>(row) = (acc[0] << 4) | acc[SEGS > 1 ? 1 : 0];
            *reinterpret_cast<uint32_t*>(row + plane) = mapped(sum);
        }
        if (MODE == kCountsMapped && a == 0) *reinterpret_cast<uint32_t*>(row + plane) = mapped(sum);
    }
}

// Least and greatest final-look count of each axis value over its first
// K_tiles sims: bb[v] and bb[NA + v].  One block per axis value, 16-byte loads
// folded with byte-wise min / max; the row's padding bytes past K_tiles (never
// written) are masked to the neutral values.
__global__ void __launch_bounds__(256) k_axis_box(const uint8_t* __restrict__ cnt, int32_t NA, int32_t k_stride,
                                                 int32_t K_tiles, int32_t last, uint32_t* __restrict__ bb)
{
    pdl_entry();
    const int v = blockIdx.x;
    const uint8_t* row = cnt + ((int64_t)last * NA + v) * k_stride;
    unsigned lo = 0xFFFFFFFFu, hi = 0u;
    for (int k16 = threadIdx.x * 16; k16 < K_tiles; k16 += blockDim.x * 16) {
        const uint4 w = *reinterpret_cast<const uint4*>(row + k16);
        const uint32_t q[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            // bytes at or past K_tiles take the neutral values
            const int valid = min(max(K_tiles - (k16 + 4 * b), 0), 4);
            const uint32_t keep = valid >= 4 ? 0xFFFFFFFFu : ((1u << (8 * valid)) - 1u);
            lo = __vminu4(lo, q[b] | ~keep);
            hi = __vmaxu4(hi, q[b] & keep);
        }
    }
    // bytes to one value, then the block
    lo = min(min(lo & 0xFFu, (lo >> 8) & 0xFFu), min((lo >> 16) & 0xFFu, lo >> 24));
    hi = max(max(hi & 0xFFu, (hi >> 8) & 0xFFu), max((hi >> 16) & 0xFFu, hi >> 24));
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    __shared__ unsigned s_lo[8], s_hi[8];
    const int warp = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) {
        s_lo[warp] = lo;
        s_hi[warp] = hi;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < (int)(blockDim.x >> 5); ++w) {
            lo = min(lo, s_lo[w]);
            hi = max(hi, s_hi[w]);
        }
        bb[v] = lo;
        bb[NA + v] = hi;
    }
}

// FP32 statistics with correctly rounded operations in a fixed order (no FMA
// contraction: every step is an explicit __f*_rn intrinsic).
__device__ float stat_one_arm(int x, int n, double p0d)
{
    const float p0 = (float)p0d;
    const float fn = (float)n;
    const float num = __fsub_rn((float)x, __fmul_rn(fn, p0));
    float var = __fmul_rn(fn, p0);
    var = __fmul_rn(var, __fsub_rn(1.0f, p0));
    const float z = __fdiv_rn(num, __fsqrt_rn(var));
    return -z;
}

__device__ float stat_two_arm(int x0, int x1, int n0, int n1)
{
    const float fn0 = (float)n0, fn1 = (float)n1;
    const float p0 = __fdiv_rn((float)x0, fn0);
    const float p1 = __fdiv_rn((float)x1, fn1);
    const float pb = __fdiv_rn((float)(x0 + x1), __fadd_rn(fn0, fn1));
    const float inv = __fadd_rn(__fdiv_rn(1.0f, fn0), __fdiv_rn(1.0f, fn1));
    float var = __fmul_rn(pb, __fsub_rn(1.0f, pb));
    var = __fmul_rn(var, inv);
    float z = 0.0f;
    if (var > 0.0f) z = __fdiv_rn(__fsub_rn(p1, p0), __fsqrt_rn(var));
    return -z;
}

__global__ void k_stat_table(float* __restrict__ S, DesignArgs D, int32_t n_cells, int32_t n1p)
{
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= n_cells) return;
    if (D.stat == CSE_STAT_ONE_ARM_Z) {
        S[c] = stat_one_arm(c, D.n_max, D.p0);
    } else {
        S[c] = stat_two_arm(c / n1p, c % n1p, D.n_max, D.n_max);
    }
}

// rank[c] = #{c' : S[c'] < S[c]}; val_of_rank[rank[c]] = S[c] (equal S share a rank).
// With pos and ntie (may be NULL): pos[rank[c] + #{c' < c : S[c'] = S[c]}] = c,
// the cells sorted by (S, index), so the cells of rank r sit at positions r,
// r + 1, ..., r + ntie[r] - 1, ntie[r] = #{c' : S[c'] = S[c]}.
// A warp a cell: bound by the n_cells^2 comparisons (a thread a cell left most of the
// SMs without a block: 10,201 cells 306 us, so 41).
__global__ void __launch_bounds__(256) k_rank_table(const float* __restrict__ S, uint16_t* __restrict__ rank,
                                                    float* __restrict__ vor, int32_t* __restrict__ pos,
                                                    int32_t* __restrict__ ntie, int32_t n_cells)
{
    const int c = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (c >= n_cells) return;
    const float s = S[c];
    int r = 0, e = 0, t = 0;
    for (int j = lane; j < n_cells; j += 32) {
        const float v = S[j];
        r += (v < s);
        e += (j < c && v == s);
        t += (v == s);
    }
    r = __reduce_add_sync(0xffffffffu, r);
    e = __reduce_add_sync(0xffffffffu, e);
    t = __reduce_add_sync(0xffffffffu, t);
    if (lane != 0) return;
    rank[c] = (uint16_t)r;
    vor[r] = s;
    if (pos) {
        pos[r + e] = c;
        if (e == 0) ntie[r] = t;
    }
}

}  // namespace

int cse_launch_uniforms(cse_ctx* c, cudaStream_t s)
{
    const int64_t rows = (int64_t)c->D.d * c->K_max;
    const int blocks = (int)((rows + 7) / 8);
    const int n = c->D.n_max;
    const uint32_t k0 = (uint32_t)c->seed, k1 = (uint32_t)(c->seed >> 32);
    cse_prof_begin(c, KID_UNIFORMS, s);
#define CSE_UNIFORMS(E) \
    cse_launch(c->pdl, k_uniforms<E>, dim3(blocks), dim3(256), 0, s, c->U, c->K_max, c->D.d, n, k0, k1, c->tb)
    if (n <= 32) CSE_UNIFORMS(1);
    else if (n <= 64) CSE_UNIFORMS(2);
    else CSE_UNIFORMS(4);
#undef CSE_UNIFORMS
    cse_prof_end(c, s);
    c->launches += 1;
    return cudaGetLastError() == cudaSuccess ? CSE_OK : CSE_CUDA_ERROR;
}

int cse_launch_tables(cse_ctx* c, cudaStream_t s)
{
    if (cse_posterior_design(c->D.stat)) return CSE_OK;
    const int n = c->n_cells;
    cse_prof_begin(c, KID_TABLES, s);
    k_stat_table<<<(n + 255) / 256, 256, 0, s>>>(c->S_tab, c->D, n, c->n1p);
    k_rank_table<<<(n + 7) / 8, 256, 0, s>>>(c->S_tab, c->rank_tab, c->val_of_rank, c->cell_of_pos,
                                                c->cell_of_pos ? c->cell_of_pos + n : nullptr, n);
    cse_prof_end(c, s);
    c->launches += 2;
    return cudaGetLastError() == cudaSuccess ? CSE_OK : CSE_CUDA_ERROR;
}

int cse_launch_thresholds(cse_ctx* c, const TileArgs& T, int32_t n_axis_total, cudaStream_t s)
{
    TailArgs Z = {};
    if (c->zmode != ZMODE_CELLS)
        Z = {c->S_tab, c->n_cells, c->n1p, c->D.n_max, c->z_lambda, nullptr, nullptr, nullptr};
    if (c->zmode == ZMODE_TAIL) {
        Z.pos = c->cell_of_pos;
        Z.zpar = c->zpar;
    }
    Z.zcut = c->zcut;
    cse_prof_begin(c, KID_THRESHOLDS, s);
    cse_launch(c->pdl, k_thresholds, dim3((n_axis_total + 255) / 256 + (Z.S ? 1 : 0)), dim3(256), 0, s, c->thr, c->sig,
               T, n_axis_total, Z);
    cse_prof_end(c, s);
    c->launches += 1;
    return cudaGetLastError() == cudaSuccess ? CSE_OK : CSE_CUDA_ERROR;
}

template <int SEGS, int MODE>
static int launch_counts(cse_ctx* c, const TileArgs& T, int32_t NA, int32_t K_tiles, int32_t k_stride,
                         const uint8_t* map, cudaStream_t s)
{
    // chunks of at most 512 values (256 with three segments: 2 to 3 blocks an SM),
    // equal in size, a multiple of 32
    constexpr int CH_MAX = SEGS > 1 ? 256 : 512;
    int na = 0;
    for (int a = 0; a < T.d; ++a) na = T.n_axis[a] > na ? T.n_axis[a] : na;
    const int64_t nz = ((int64_t)na + CH_MAX - 1) / CH_MAX;
    const int chunk = (int)(((na + nz - 1) / nz + 31) / 32 * 32);
    int pow2 = 32;
    while (pow2 < chunk) pow2 <<= 1;
    auto kern = k_counts<SEGS, MODE>;
    const size_t smem = (size_t)chunk * (SEGS * 128 + 4 + 2);
    // the limit of the largest chunk, whatever this call's: it belongs to the kernel, and another
    // thread may be launching with a larger chunk (with the static arrays, up to 23 KB, it passes 48 KB)
    if (smem > 20 * 1024 && cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 CH_MAX * (SEGS * 128 + 4 + 2)) != cudaSuccess) {
        cudaGetLastError();
        return CSE_CUDA_ERROR;
    }
    cse_prof_begin(c, KID_AXIS_COUNTS, s);
    const int64_t z_max = 65535;   // chunks of one launch
    for (int64_t v = 0; v < na; v += z_max * chunk) {
        const int64_t nzc = ((int64_t)na - v + chunk - 1) / chunk;
        const dim3 grid((unsigned)((K_tiles + kCntSims - 1) / kCntSims), (unsigned)T.d,
                        (unsigned)(nzc < z_max ? nzc : z_max));
        cse_launch(c->pdl, kern, grid, dim3(kCntThreads), smem, s, c->cnt, c->thr, T, NA, K_tiles, k_stride,
                   make_int2(c->D.look_n[0], c->D.look_n[1]), c->D.n_max, (uint32_t)c->seed,
                   (uint32_t)(c->seed >> 32), c->tb, chunk, pow2, (int32_t)v, map);
        c->launches += 1;
    }
    cse_prof_end(c, s);
    return cudaGetLastError() == cudaSuccess ? CSE_OK : CSE_CUDA_ERROR;
}

int cse_launch_axis_counts(cse_ctx* c, const TileArgs& T, int32_t n_axis_total, int32_t K_tiles,
                           int32_t k_stride, cudaStream_t s)
{
    if (cse_count_nibbles(c))
        return launch_counts<3, kCountsNib>(c, T, n_axis_total, K_tiles, k_stride, c->bt_score, s);
    if (c->D.n_looks > 1) return launch_counts<3, kCountsRaw>(c, T, n_axis_total, K_tiles, k_stride, nullptr, s);
    // (b(x_0) beside arm 0's counts: where the kernel counts rejections by bytes)
    const bool map = c->zmode == ZMODE_COUNT ||
                     (c->zmode == ZMODE_TAIL && c->D.n_max <= 126 && c->z_lambda > -INFINITY);
    if (map && T.d == 2)
        return launch_counts<1, kCountsMapped>(c, T, n_axis_total, K_tiles, k_stride, c->zcut, s);
    return launch_counts<1, kCountsRaw>(c, T, n_axis_total, K_tiles, k_stride, nullptr, s);
}

int cse_launch_axis_box(cse_ctx* c, int32_t n_axis_total, int32_t K_tiles, int32_t k_stride, cudaStream_t s)
{
    cse_prof_begin(c, KID_AXIS_COUNTS, s);
    cse_launch(c->pdl, k_axis_box, dim3(n_axis_total), dim3(256), 0, s, c->cnt, n_axis_total, k_stride, K_tiles,
               c->D.n_looks - 1, c->bb);
    cse_prof_end(c, s);
    c->launches += 1;
    return cudaGetLastError() == cudaSuccess ? CSE_OK : CSE_CUDA_ERROR;
}
