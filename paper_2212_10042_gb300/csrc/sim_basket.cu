// sim_basket.cu -- the Bayesian basket trial of Sec. 10.1: four arms of n patients
// (n = 35 in the paper), one analysis, and the hierarchical model
//   theta_i ~ N(mu, s2), mu ~ N(-1.34, 100), s2 ~ InvGamma(0.0005, 0.000005)
// on the offset log-odds theta_i = logit(p_i) - t_i, where t_i is the logit of
// arm i's null response rate.  Each arm's likelihood is replaced by the normal
// approximation of its empirical logit (x + 1/2 successes, n - x + 1/2
// failures), s2 is integrated on the 16 log-spaced nodes shared with the
// four-arm selection design, mu and the thetas exactly.  Arm i is rejected when
// P(theta_i > 0 | x) > 1 - lambda (lambda = 0.15: the 85% rule); the FWER
// statistic of a tile is S = min over the tile's null arms of 1 - P_i.
//
// The posterior depends on a trial only through its four success counts, so the
// context tabulates Q_i = 1 - P_i in FP32 over all (n + 1)^4 count states once
// (a float4 per state, 27 MB for n = 35, L2-resident) and, from it, the trials
// that cannot decide anything (k_sim_basket).  The direct mode (plain path)
// evaluates the same FP32 function for every trial instead.
#include <cuda_runtime.h>
#include <math.h>

#include "cse_internal.cuh"

namespace {

constexpr int BT = 256;          // threads of the simulation kernel
constexpr int BWARP = BT / 32;
constexpr int SPT = 8;           // direct mode: consecutive sims per thread and step (one 8-byte count load per arm)

struct Basket {
    int n;        // patients per arm
    int m;        // n + 1: count states per arm
    float t[4];   // null logits t_i
};

// Q_i = 1 - P(theta_i > 0 | x) for the four arms, FP32.  Not inlined, so the
// table builder and the direct mode run the same instruction sequence.
__device__ __noinline__ void basket_q_f32(const int* x, const Basket& B, const NodeConst& C, float* Q)
{
    const float MU0 = -1.34f, TAU2 = 100.0f;
    float th[4], s2[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float xs = (float)x[i] + 0.5f, fs = (float)(B.n - x[i]) + 0.5f;
        th[i] = logf(xs / fs) - B.t[i];
        s2[i] = 1.0f / xs + 1.0f / fs;
    }
    float lw[kBayesNodes], qj[kBayesNodes][4];
    float mx = -INFINITY;
#pragma unroll 4
    for (int j = 0; j < kBayesNodes; ++j) {
        const float sg = C.sig2[j];
        float W = 0.f, Sr = 0.f, Srr = 0.f, Sth = 0.f, prod = 1.f;
        float w[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float den = sg + s2[i];
            w[i] = 1.0f / den;
            const float r = th[i] - MU0;
            W += w[i];
            Sr += w[i] * r;
            Srr += w[i] * r * r;
            Sth += w[i] * th[i];
            prod *= den;
        }
        // N(theta_hat; mu0 1, s2 I + diag(s_i^2) + 100 11') by the rank-one update
        const float prec = 1.0f / TAU2 + W;
        const float quad = Srr - Sr * Sr / prec;
        const float logdet = logf(prod * (1.0f + TAU2 * W));
        lw[j] = C.lprior[j] - 0.5f * logdet - 0.5f * quad;
        mx = fmaxf(mx, lw[j]);
        const float mmu = (MU0 / TAU2 + Sth) / prec;
        const float vmu = 1.0f / prec;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            // theta_i | mu, s2, x ~ N((1 - c) th_i + c mu, s_i^2 s2 / (s_i^2 + s2)), c = s_i^2 / (s_i^2 + s2);
            // mu integrated over N(mmu, vmu)
            const float c = s2[i] * w[i];
            const float v = s2[i] * sg * w[i] + c * c * vmu;
            const float e = (1.0f - c) * th[i] + c * mmu;
            qj[j][i] = normcdff(-e * rsqrtf(v));   // 1 - P(theta_i > 0) without the cancellation
        }
    }
    float Z = 0.f, a[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int j = 0; j < kBayesNodes; ++j) {
        const float wj = expf(lw[j] - mx);
        Z += wj;
#pragma unroll
        for (int i = 0; i < 4; ++i) a[i] += wj * qj[j][i];
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) Q[i] = a[i] / Z;
}

__global__ void k_table_basket(float4* __restrict__ Qt, Basket B)
{
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    const int m = B.m;
    __shared__ NodeConst C;
    node_const_block(C);
    if (s >= m * m * m * m) return;
    const int x[4] = {s / (m * m * m), (s / (m * m)) % m, (s / m) % m, s % m};
    float Q[4];
    basket_q_f32(x, B, C, Q);
    Qt[s] = make_float4(Q[0], Q[1], Q[2], Q[3]);
}

// S of one trial: min over the null arms in `mask` of Q_i (+inf when none).
__device__ __forceinline__ float masked_min(const float4& q, uint32_t mask)
{
    float S = INFINITY;
    if (mask & 1u) S = fminf(S, q.x);
    if (mask & 2u) S = fminf(S, q.y);
    if (mask & 4u) S = fminf(S, q.z);
    if (mask & 8u) S = fminf(S, q.w);
    return S;
}

template <bool TABLE>
__device__ __forceinline__ float4 state_q(const float4* __restrict__ Qt, const Basket& B, const NodeConst& C,
                                          const int* x)
{
    if (TABLE) return __ldg(Qt + ((x[0] * B.m + x[1]) * B.m + x[2]) * B.m + x[3]);
    float Q[4];
    basket_q_f32(x, B, C, Q);
    return make_float4(Q[0], Q[1], Q[2], Q[3]);
}

__device__ __forceinline__ int basket_warp_sum(int v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// One thread: the tile's outputs from the warps' sums.
__device__ __forceinline__ void basket_store(const TileArgs& T, const Basket& B, const SimOut& o, int64_t i, int K,
                                             bool bad, const int* v, const int (*red)[BWARP], int warps,
                                             bool select, double lam_i, int32_t* err)
{
    if (bad) atomicOr(err, CSE_ERR_BAD_K);
    int64_t Rt = 0, X[4] = {0, 0, 0, 0};
    for (int w = 0; w < warps; ++w) {
        Rt += red[0][w];
        for (int a = 0; a < 4; ++a) X[a] += red[1 + a][w];
    }
    if (o.R) o.R[i] = Rt;
    if (o.cp_key)   // the tile's (K, R) in the Clopper-Pearson memo, as k_cp_mark would
        o.cp_slot[i] = cp_memo_insert(((unsigned long long)(uint32_t)K << 32) | (uint32_t)Rt, o.cp_key, o.cp_cap,
                                      o.cp_list, o.cp_nkeys);
    for (int a = 0; a < 4; ++a) {
        if (o.Xrej) o.Xrej[i * 4 + a] = X[a];
        if (o.score) {
            const double sg = bad ? NAN : o.sig[T.axis_off[a] + v[a]];
            o.score[i * 4 + a] = (double)X[a] - (double)B.n * sg * (double)Rt;
        }
    }
    if (select && o.lam_tile) o.lam_tile[i] = lam_i;
}

// ---------------------------------------------------------------------------
// The tabulated simulation: counting by bits, evaluating only the trials that can
// decide the order statistic.
//
// A 16-byte gather from the state table touches a line of L1 per trial, and L1
// looks up one line a clock: one clock a trial and SM whatever else the kernel does
// (3.1 of the 3.67 ms of the 16^4 grid at K = 2^14).  Whether a trial rejects, and
// whether it can be among the k_i smallest S, is a bit of its count state.  Before
// the launch k_basket_bits packs "Q_a < lambda" over all states, a bit per x_3 in a
// word per (arm, x_0, x_1, x_2); the context keeps the same for kLevels fixed levels
// of S.  A tile takes the states within kWindow standard deviations of its expected
// counts (w_a counts of arm a), ORs the words of its null arms and puts them in
// shared memory: w_0 w_1 w_2 words (~2,000), against K trials that each read one.
// A trial's four counts are the bytes of one word P (byte transposes); two additions
// and a mask tell whether all lie in the window, a dot product and a multiply-add
// give its word, and the rotation by P brings its bit to the top.  The sign bits of
// four trials become a byte mask, and one dot product per arm adds their counts.
//
// Evaluated from the state table, queued per warp and 32 at a time: trials outside
// the window (4 in a hundred) and, with a selection, those below the tile's level L_c,
// the least one above the k_i smallest S as far as the first kSample trials (all
// evaluated) tell, with a margin of 2.5 standard deviations.  Keys below L_c go to
// the warp's stretch of global memory and into 256 bins; the k_i-th is ranked within
// its bin.  It is exact when it is at most L_c.
//
// Otherwise, and where the sample shows a large share of the trials below L_c (rates far
// from the null rates: every S near 0 or near 1, which the levels do not resolve), the
// tile goes to a list for k_sim_basket_all, which evaluates every trial: there the counts
// hardly vary and its gathers meet in few lines.  8^4 grid, K = 16,384, a step over logits
// [1, 4] 837 -> 334 us (every trial through the queue before; 366 with the gathers alone),
// [-1, 2] 1,080 -> 540 (567), [-6, -4] 612 -> 338 (409), [-3.5, 1] 358 -> 346 (812).
// The share: a quarter against a half 536 / 612 us over [-1, 2], but n = 20 313 / 291.
// 256 threads a tile below 4 tiles an SM: 150 tiles of 2^18 trials 1,565 -> 700 us.
//
// What bounds it: issue slots (71 %) and the integer pipe (65 %): per 32 trials ~17
// warp instructions of test and count, ~10 of queue and scan, ~7 of evaluation, and
// ~20 of the tile's own work (building the window, setup, selection).  16^4 grid,
// K = 2^14, with a selection (59,992 tiles): 3.67 -> 1.90 ms; 6,036 tiles of 1,000 to
// 30,000 trials without one: 152 -> 112 us, plus 10 for the bits of lambda.  Measured
// on the way: one bit per state at a fixed level and every rejection evaluated 3.28 ms
// (the candidates' own work), lambda's and the level's bits in separate words 2.58,
// in one 2.34; 128 threads a tile instead of 256 1.98 (more tiles in flight to cover
// the window's loads and the barriers); the sample and the tiles without a test a trial a
// lane, unqueued: 1.95.
// ---------------------------------------------------------------------------
constexpr int kLevels = 32;        // levels of S for selections: 2^((c + 1) / 4 - 8), the last +inf
constexpr int kMaxM = 64;          // count states of an arm: two 32-bit words of x_3
constexpr int kSample = 512;       // first trials of a tile, all evaluated to place c
// up to this K every trial is evaluated, a trial a lane: 19,056 tiles, a step at K = 1,500 509 us
// against 580 by bits, at 2,000 587 against 593
constexpr int kAllK = 2048;
// up to this K a tile that turns out dense is finished here, every trial evaluated, instead of
// starting again in the kernel over the list (8^4 grid, a step at K = 4,096: 231 us against 241)
constexpr int kHereK = 8192;
constexpr int kQueue = 288;        // a warp's candidate queue (up to 31 left over, at least 16 lanes' trials a round)
constexpr int kList = 256;         // keys of the selected bin ranked in shared memory
constexpr int kSpan3 = 16;         // most counts of arm 3 in the window: the bits of half a word
constexpr float kWindow = 2.6f;    // half-width of the window in standard deviations

__host__ __device__ inline float basket_level(int c)
{
    return c >= kLevels - 1 ? INFINITY : exp2f(0.25f * (float)(c + 1) - 8.0f);
}

// most counts of an arm in the window (p = 1/2; of arm 3 at most kSpan3)
inline int basket_span(int n)
{
    const int w = (int)(kWindow * sqrtf((float)n)) + 2;
    return w < n + 1 ? w : n + 1;
}

// bits[(l 4 + a) rows + row] of levels l = first .. first + count - 1: bit 31 - (x_3 & 31) of half
// x_3 >> 5 is Q_a(row, x_3) < level (lambda_up for l = kLevels).  A warp per row: the table's row is
// read once for all arms and levels: bound by its loads (the lambda level of n = 35: 10 us, 27 MB read).
__global__ void __launch_bounds__(256) k_basket_bits(uint2* __restrict__ bits, const float4* __restrict__ Qt, int m,
                                                     int rows, int first, int count, float lambda_up)
{
    const int row = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (row >= rows) return;
    const int x0 = 31 - lane, x1 = 63 - lane;
    const float4 none = make_float4(INFINITY, INFINITY, INFINITY, INFINITY);
    const float4 q0 = x0 < m ? __ldg(Qt + (int64_t)row * m + x0) : none;
    const float4 q1 = x1 < m ? __ldg(Qt + (int64_t)row * m + x1) : none;
    for (int l = first; l < first + count; ++l) {
        const float lev = l == kLevels ? lambda_up : basket_level(l);
        const uint32_t b[8] = {__ballot_sync(0xffffffffu, q0.x < lev), __ballot_sync(0xffffffffu, q1.x < lev),
                               __ballot_sync(0xffffffffu, q0.y < lev), __ballot_sync(0xffffffffu, q1.y < lev),
                               __ballot_sync(0xffffffffu, q0.z < lev), __ballot_sync(0xffffffffu, q1.z < lev),
                               __ballot_sync(0xffffffffu, q0.w < lev), __ballot_sync(0xffffffffu, q1.w < lev)};
        if (lane < 4) {
            uint2 h = make_uint2(b[0], b[1]);
            if (lane == 1) h = make_uint2(b[2], b[3]);
            if (lane == 2) h = make_uint2(b[4], b[5]);
            if (lane == 3) h = make_uint2(b[6], b[7]);
            bits[((int64_t)l * 4 + lane) * rows + row] = h;
        }
    }
}

// Bits 31 .. 32 - s cleared (s in 0 .. 32).
__device__ __forceinline__ uint32_t bits_from(int s) { return s >= 32 ? 0u : 0xFFFFFFFFu >> s; }

// Bits 31 (HIGH) or 15 of f[0..3] as bytes 0xFF / 0x00 (prmt's replicated sign: selector bit 3).
template <bool HIGH>
__device__ __forceinline__ uint32_t sign_bytes(const uint32_t* f)
{
    uint32_t a, b;
    if (HIGH) {
        asm("prmt.b32 %0, %1, %2, 0x00FB;" : "=r"(a) : "r"(f[0]), "r"(f[1]));
        asm("prmt.b32 %0, %1, %2, 0xFB00;" : "=r"(b) : "r"(f[2]), "r"(f[3]));
    } else {
        asm("prmt.b32 %0, %1, %2, 0x00D9;" : "=r"(a) : "r"(f[0]), "r"(f[1]));
        asm("prmt.b32 %0, %1, %2, 0xD900;" : "=r"(b) : "r"(f[2]), "r"(f[3]));
    }
    return __byte_perm(a, b, 0x7610);
}

// The window's bits of a row, x_3 = lo .. hi - 1 (at most 16), at 15 - (x_3 & 15): m[j] selects the
// window's part of states 16 j .. 16 j + 15.
__device__ __forceinline__ uint32_t fold16(const uint2& h, const uint2& mk)
{
    const uint32_t t = (h.x & mk.x) | (h.y & mk.y);
    return (t | (t >> 16)) & 0xFFFFu;
}

template <bool SELECT, int NT>
__global__ void __launch_bounds__(NT, 1024 / NT)
    k_sim_basket(TileArgs T, Basket B, const uint8_t* __restrict__ cnt, int32_t k_stride, int32_t K_tiles,
                 const float4* __restrict__ Qt, const uint2* __restrict__ planes, int32_t span, float lambda_up,
                 bool want_R, SimOut o, uint32_t* __restrict__ keys, int32_t key_seg, int32_t* __restrict__ left,
                 int32_t* __restrict__ counter, int32_t* __restrict__ err)
{
    constexpr int NW = NT / 32;
    constexpr int ALL = kLevels - 1;   // every trial evaluated
    // word 0: a trial outside the window (evaluated, not counted); then w_0 w_1 w_2 words: lambda's bits
    // in the upper half, those of the level in the lower
    extern __shared__ uint32_t bits[];
    __shared__ uint16_t s_queue[NW][kQueue];
    __shared__ uint32_t hist[SELECT ? 256 : 1];
    __shared__ uint32_t list[SELECT ? kList : 1];
    __shared__ int s_tile, s_next, s_pick, s_before, s_nlist, s_nk[NW];
    __shared__ uint32_t s_res;
    __shared__ int s_red[5][BWARP];
    __shared__ unsigned long long s_min;   // order key of the least lambda_i of this CTA's tiles
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint16_t* const queue = s_queue[warp];
    // each warp appends its keys to its own stretch of key_seg words
    uint32_t* const kbuf = keys + ((int64_t)blockIdx.x * NW + warp) * key_seg;
    const unsigned below = (1u << lane) - 1u;
    const int m = B.m;
    const int dense = B.n > 24 ? kSample / 4 : kSample / 2;   // (few patients: few values of S, so large steps)
    if (SELECT)
        for (int b = tid; b < 256; b += NT) hist[b] = 0u;
    if (tid == 0) {
        s_min = ~0ull;
        s_next = atomicAdd(counter, 1);
        bits[0] = 0xFFFFu;
    }

    for (;;) {
        __syncthreads();
        if (tid == 0) {
            s_tile = s_next;
            s_nlist = 0;
        }
        __syncthreads();
        const int64_t i = s_tile;
        if (i >= T.n_tiles) break;
        if (tid == 0) s_next = atomicAdd(counter, 1);   // the next tile, fetched while this one runs
        const int K = T.K[i];
        // each lane one arm's index and window, then shared: counts lo .. lo + w - 1, within 0 .. n
        const int la = lane & 3;
        const int vl = T.center_idx[i * 4 + la];
        int na = T.n_axis[0], ao = T.axis_off[0];
#pragma unroll
        for (int a = 1; a < 4; ++a)   // by selection: no runtime index into the argument
            if (la == a) na = T.n_axis[a], ao = T.axis_off[a];
        const bool bad = __any_sync(0xffffffffu, vl < 0 || vl >= na) || K < 1 || K > K_tiles;
        const int atl = ao + (bad ? 0 : vl);
        const float pl = bad ? 0.5f : (float)o.sig[atl], mu = (float)B.n * pl;
        const int wl = min((int)(2.0f * kWindow * sqrtf(mu * (1.0f - pl))) + 2, la == 3 ? min(span, kSpan3) : span);
        const int ll = min(max((int)(mu + 0.5f - 0.5f * (float)(wl - 1)), 0), m - wl);
        const uint32_t mask = T.null_mask[i] & 15u;   // null arms (none: S = +inf throughout)
        const int Kc = (bad || mask == 0u) ? 0 : K;
        const uint8_t* rowp[4];
        int lo[4], w[4], v[4];
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            v[a] = __shfl_sync(0xffffffffu, vl, a);
            rowp[a] = cnt + (int64_t)__shfl_sync(0xffffffffu, atl, a) * k_stride;
            w[a] = __shfl_sync(0xffffffffu, wl, a);
            lo[a] = __shfl_sync(0xffffffffu, ll, a);
        }
        const int ks = (SELECT && !bad) ? o.ksel[i] : 0;
        const bool sel = SELECT && ks >= 1;
        // A selection starts with a sample, every trial of it evaluated.  c: the level of the
        // trials to come (-1: none is needed)
        bool sample = sel && Kc > kAllK;
        int c = (sel || Kc <= kAllK) ? ALL : -1;
        int r_neg = 0, x_neg[4] = {0, 0, 0, 0};   // minus the rejections and their counts
        double lam_i = -INFINITY;
        bool found = false, leave = false;   // leave: to the kernel that evaluates every trial
        do {
            int qn = 0, wk = 0;   // queued candidates, kept keys of this warp
            const int k0 = sample ? kSample : 0;
            // bytes of P: x_3, x_2, x_1, x_0.  C1: bit 7 of a byte set iff x >= lo; C2: iff
            // x >= lo + w (bytes up to 127: no carry)
            const uint32_t C1 = 0x80808080u - (uint32_t)(lo[3] | (lo[2] << 8) | (lo[1] << 16) | (lo[0] << 24));
            const uint32_t C2 = C1 - (uint32_t)(w[3] | (w[2] << 8) | (w[1] << 16) | (w[0] << 24));
            // byte address of a trial's word: 4 ((x_0 w_1 + x_1) w_2 + x_2) + base
            const uint32_t W0 = 4u * (uint32_t)(w[1] * w[2]), WD = (4u << 8) | ((uint32_t)(4 * w[2]) << 16);
            const uint32_t base = 4u - 4u * (uint32_t)((lo[0] * w[1] + lo[1]) * w[2] + lo[2]);
            float level = c < 0 ? 0.0f : basket_level(c);
            // one trial a lane
            auto eval = [&](int k, bool live) {
                int x[4];
                bool count = c == ALL;   // a rejection inside the window is counted by its bit
#pragma unroll
                for (int a = 0; a < 4; ++a) {
                    x[a] = min((int)__ldg(rowp[a] + k), B.n);
                    count |= (uint32_t)(x[a] - lo[a]) >= (uint32_t)w[a];
                }
                const float4 q = __ldg(Qt + ((x[0] * m + x[1]) * m + x[2]) * m + x[3]);
                const float S = live ? masked_min(q, mask) : INFINITY;
                const int rej = (S < lambda_up && live && count) ? 1 : 0;
                r_neg -= rej;
#pragma unroll
                for (int a = 0; a < 4; ++a) x_neg[a] -= rej ? x[a] : 0;
                if (sel) {
                    const bool keep = S < level;
                    const unsigned kept = __ballot_sync(0xffffffffu, keep);
                    if (keep) {
                        kbuf[wk + __popc(kept & below)] = __float_as_uint(S);
                        atomicAdd(&hist[key_bin(__float_as_uint(S))], 1u);
                    }
                    wk += __popc(kept);
                }
            };
            if (sample) {   // the sample, spread over the warps, and the level of the trials to come
                for (int k = warp * (kSample / NW) + lane; k < (warp + 1) * (kSample / NW); k += 32) eval(k, true);
                __syncthreads();
                if (warp == 0) {
                    // the least level with the keys below it so far, scaled to all K trials and
                    // less 2.5 standard deviations, reaching k_i
                    const float f = ((float)Kc - (float)kSample) / (float)kSample, d = 2.5f * sqrtf(f * (1.0f + f));
                    const float r = (d + sqrtf(d * d + 4.0f * (1.0f + f) * (float)ks)) / (2.0f * (1.0f + f));
                    int before = 0;
                    const int b = warp_pick256<false>(hist, (int)ceilf(r * r) + 1, lane, &before);
                    const bool above = b >= 0 && (lane == ALL || key_bin(__float_as_uint(basket_level(lane))) > b);
                    const unsigned who = __ballot_sync(0xffffffffu, above);   // a lane a level
                    const int cl = who ? __ffs(who) - 1 : ALL;
                    // the sample's keys below it: with more than dense of the trials among them the
                    // test saves nothing
                    const int kb = key_bin(__float_as_uint(basket_level(cl)));
                    int nb = 0;
#pragma unroll
                    for (int j = 0; j < 8; ++j) nb += lane * 8 + j < kb ? (int)hist[lane * 8 + j] : 0;
                    nb = basket_warp_sum(nb);
                    if (lane == 0) s_pick = cl == ALL || nb > dense ? ALL : cl;
                }
                __syncthreads();
                c = s_pick;
                leave = c == ALL && Kc > kHereK;
                if (leave) break;
                level = basket_level(c);
            }
            if (c == ALL)   // no test: a trial a lane (k - lane is the warp's)
                for (int k = k0 + tid; k - lane < Kc; k += NT) eval(min(k, Kc - 1), k < Kc);
            // sixteen consecutive trials per thread and step from k0 on
            for (int st = 0; c != ALL && k0 + st * (NT * 16) < Kc; ++st) {
                if (st == 0) {
                    // a thread a word; its place steps by NT words
                    const int hi3 = lo[3] + w[3], w12 = w[1] * w[2], rows = w[0] * w12, rm = m * m * m;
                    const uint2 mk = make_uint2(bits_from(lo[3]) & ~bits_from(min(hi3, 32)),
                                                bits_from(max(lo[3] - 32, 0)) & ~bits_from(max(hi3 - 32, 0)));
                    const int d0 = NT / w12, e0 = NT - d0 * w12, d1 = e0 / w[2], d2 = e0 - d1 * w[2];
                    int y1 = tid % w12, src = tid / w12;
                    int y2 = y1 % w[2];
                    y1 /= w[2];
                    src = ((lo[0] + src) * m + lo[1] + y1) * m + lo[2] + y2;
                    const int step = (d0 * m + d1) * m + d2, c2 = m - w[2], c1 = (m - w[1]) * m;
                    const uint2* const pl = planes + (int64_t)kLevels * 4 * rm;
                    const uint2* const pc = planes + (int64_t)max(c, 0) * 4 * rm;
#pragma unroll 2
                    for (int r = tid; r < rows; r += NT) {
                        uint2 hl = make_uint2(0u, 0u), hc = make_uint2(0u, 0u);
#pragma unroll
                        for (int a = 0; a < 4; ++a)
                            if ((mask >> a) & 1u) {
                                if (want_R) {
                                    const uint2 h = __ldg(pl + a * rm + src);
                                    hl.x |= h.x, hl.y |= h.y;
                                }
                                if (SELECT && c >= 0) {
                                    const uint2 h = __ldg(pc + a * rm + src);
                                    hc.x |= h.x, hc.y |= h.y;
                                }
                            }
                        bits[1 + r] = (fold16(hl, mk) << 16) | (SELECT ? fold16(hc, mk) : 0u);
                        y2 += d2, y1 += d1, src += step;
                        if (y2 >= w[2]) y2 -= w[2], y1 += 1, src += c2;
                        if (y1 >= w[1]) y1 -= w[1], src += c1;
                    }
                    __syncthreads();
                }
                // first trial of the warp at the start of the queue's block of 64 steps
                const int kb = k0 + (st & ~63) * (NT * 16) + warp * 512;
                const int stq = st & 63;
                const int kw = kb + stq * (NT * 16) + lane * 16;
                uint32_t cm = 0u;   // bit t: trial kw + t is evaluated
                if (kw < Kc) {
                    uint32_t A[4][4];
#pragma unroll
                    for (int a = 0; a < 4; ++a) {   // kw + 16 <= k_stride (a multiple of 16)
                        const uint4 x = __ldg(reinterpret_cast<const uint4*>(rowp[a] + kw));
                        A[a][0] = x.x, A[a][1] = x.y, A[a][2] = x.z, A[a][3] = x.w;
                    }
                    if (kw + 16 > Kc) {   // trials at or past K: outside the window (lo + w <= 64 < 127)
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            const int left = Kc - kw - 4 * q;
                            const uint32_t past = left >= 4 ? 0u : left <= 0 ? ~0u : ~0u << (8 * left);
#pragma unroll
                            for (int a = 0; a < 4; ++a) A[a][q] = (A[a][q] & ~past) | (0x7F7F7F7Fu & past);
                        }
                    }
                    int cneg = 0;   // minus the candidates' bits
#pragma unroll
                    for (int q = 3; q >= 0; --q) {
                        const uint32_t l01 = __byte_perm(A[3][q], A[2][q], 0x5140);
                        const uint32_t l23 = __byte_perm(A[3][q], A[2][q], 0x7362);
                        const uint32_t h01 = __byte_perm(A[1][q], A[0][q], 0x5140);
                        const uint32_t h23 = __byte_perm(A[1][q], A[0][q], 0x7362);
                        const uint32_t P[4] = {__byte_perm(l01, h01, 0x5410), __byte_perm(l01, h01, 0x7632),
                                               __byte_perm(l23, h23, 0x5410), __byte_perm(l23, h23, 0x7632)};
                        uint32_t f[4];
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const uint32_t out = (~(P[j] + C1) | (P[j] + C2)) & 0x80808080u;
                            uint32_t at = (P[j] >> 24) * W0 + __dp4a(P[j], WD, base);
                            at = out ? 0u : at;
                            f[j] = *reinterpret_cast<const uint32_t*>(reinterpret_cast<const char*>(bits) + at)
                                   << (P[j] & 15u);
                        }
                        const int M = (int)sign_bytes<true>(f), C = (int)sign_bytes<false>(f);
                        r_neg = __dp4a(M, 0x01010101, r_neg);
#pragma unroll
                        for (int a = 0; a < 4; ++a) x_neg[a] = __dp4a(M, (int)A[a][q], x_neg[a]);
                        cneg = __dp4a(C, 0x08040201, cneg * 16);
                    }
                    cm = (uint32_t)(-cneg);
                    if (kw + 16 > Kc) cm &= (1u << (Kc - kw)) - 1u;   // trials at or past K
                }
                const int nm = __popc(cm);
                int incl = nm;
#pragma unroll
                for (int off = 1; off < 32; off <<= 1) {
                    const int y = __shfl_up_sync(0xffffffffu, incl, off);
                    if (lane >= off) incl += y;
                }
                const int total = __shfl_sync(0xffffffffu, incl, 31);
                const bool flush = (st & 63) == 63 || k0 + (st + 1) * (NT * 16) >= Kc;
                const int ent = (stq << 9) | (lane << 4);   // entry: step (6 bits), lane, trial
                int done = 0;   // candidates of this step queued so far
                do {
                    // the lanes whose candidates fit the queue (a prefix of those left)
                    const bool mine = incl - nm >= done && incl - done <= kQueue - qn;
                    const unsigned who = __ballot_sync(0xffffffffu, mine);
                    const int upto = __shfl_sync(0xffffffffu, incl, 31 - __clz(who));
                    if (mine) {
                        uint16_t* at = queue + qn + (incl - nm - done);
                        while (cm) {
                            const int b = __ffs(cm) - 1;
                            cm &= cm - 1u;
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
                        const int k = kb + (ev >> 9) * (NT * 16) + (ev & 511);
                        eval(k, lane < n);
                        __syncwarp();   // the queue's entries read before the next round writes
                    }
                } while (done < total);
            }
            if (!sel) break;
            if (lane == 0) s_nk[warp] = wk;
            __syncthreads();
            // the ks-th smallest key: its bin, then its rank among the bin's keys
            int nk = 0;
#pragma unroll
            for (int w2 = 0; w2 < NW; ++w2) nk += s_nk[w2];
            found = nk >= ks;
            if (found) {
                if (warp == 0) {
                    int before = 0;
                    const int b = warp_pick256<true>(hist, ks, lane, &before);
                    if (lane == 0) {
                        s_pick = b;
                        s_before = before;
                    }
                }
                __syncthreads();
                const int b = s_pick, kr = ks - s_before;
                for (int k = lane; k < wk; k += 32) {   // each warp its own keys
                    const uint32_t key = kbuf[k];
                    if (key_bin(key) == b) {
                        const int at = atomicAdd(&s_nlist, 1);
                        if (at < kList) list[at] = key;
                    }
                }
                __syncthreads();
                const int nl = s_nlist;
                if (nl <= kList) {
                    for (int j = tid; j < nl; j += NT) {
                        const uint32_t key = list[j];
                        int rank = 0;
                        for (int q = 0; q < nl; ++q) {
                            const uint32_t u = list[q];
                            rank += (u < key || (u == key && q < j)) ? 1 : 0;
                        }
                        if (rank == kr - 1) s_res = key;
                    }
                    __syncthreads();
                } else {   // radix select over the bin's keys: digits of 8, 8, 8 and 7 bits (S >= 0)
                    uint32_t prefix = 0u, pmask = 0u;
                    int kq = kr;
                    for (int pass = 0; pass < 4; ++pass) {
                        const int sh = pass < 3 ? 23 - 8 * pass : 0;
                        const uint32_t dm = pass < 3 ? 0xFFu : 0x7Fu;
                        for (int k = lane; k < wk; k += 32) {
                            const uint32_t key = kbuf[k];
                            if (key_bin(key) == b && (key & pmask) == prefix) atomicAdd(&hist[(key >> sh) & dm], 1u);
                        }
                        __syncthreads();
                        if (warp == 0) {
                            int before = 0;
                            const int digit = warp_pick256<true>(hist, kq, lane, &before);
                            if (lane == 0) {
                                s_pick = digit;
                                s_before = before;
                            }
                        }
                        __syncthreads();
                        prefix |= (uint32_t)s_pick << sh;
                        pmask |= dm << sh;
                        kq -= s_before;
                    }
                    if (tid == 0) s_res = prefix;
                    __syncthreads();
                }
                lam_i = (double)__uint_as_float(s_res);
                // exact unless it lies above the level of the trials left out
                leave = !(lam_i <= (double)basket_level(c));
            } else {
                lam_i = INFINITY;   // with every trial evaluated, the k_i-th smallest S is +inf
                leave = c != ALL;   // too few keys below the level
            }
        } while (false);
        if (SELECT && sel && !found) {   // (the selection clears the bins)
            __syncthreads();   // every thread has read the counts
            for (int b = tid; b < 256; b += NT) hist[b] = 0u;
        }
        if (leave) {
            if (tid == 0) left[atomicAdd(counter + 2, 1)] = (int32_t)i;
            continue;
        }
        const int Rw = -basket_warp_sum(r_neg);
        int Xw[4];
#pragma unroll
        for (int a = 0; a < 4; ++a) Xw[a] = -basket_warp_sum(x_neg[a]);
        if (lane == 0) {
            s_red[0][warp] = Rw;
            for (int a = 0; a < 4; ++a) s_red[1 + a][warp] = Xw[a];
        }
        __syncthreads();
        if (tid == 0) {
            basket_store(T, B, o, i, K, bad, v, s_red, NW, SELECT, lam_i, err);
            if (SELECT) s_min = min(s_min, order_key(lam_i));
        }
    }
    queue_reset_min(counter, o.min_key, s_min, SELECT ? o.min_out : nullptr, (int)gridDim.x, left != nullptr);
}

// Every trial evaluated, from the state table (the tiles that k_sim_basket leaves: one
// 16-byte gather a trial, which costs little where the counts hardly vary) or, the
// plain path's form, through the posterior function.  SELECT adds
// the per-tile order statistic lambda_i = S_(ksel_i) by a three-digit radix select
// (11, 11, 10 bits of the FP32 keys, which order like the non-negative S) over the
// keys the CTA stored.
template <bool TABLE, bool SELECT>
__global__ void __launch_bounds__(BT, 4)
    k_sim_basket_all(TileArgs T, Basket B, const uint8_t* __restrict__ cnt, int32_t k_stride, int32_t K_tiles,
                     const float4* __restrict__ Qt, float lambda_up, SimOut o, uint32_t* __restrict__ keys,
                     const int32_t* __restrict__ list, int32_t* __restrict__ counter, int32_t* __restrict__ err)
{
    pdl_entry();
    int blocks;
    const int64_t n_todo = queue_tiles(list, counter, T.n_tiles, &blocks);
    if ((int)blockIdx.x >= blocks) return;
    __shared__ uint32_t hist[2048];
    __shared__ int s_tile, s_scan[BWARP], s_res[2];
    __shared__ int s_red[5][BWARP];
    __shared__ unsigned long long s_min;   // order key of the least lambda_i of this CTA's tiles
    if (threadIdx.x == 0) s_min = ~0ull;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    NodeConst C;
    if (!TABLE) C = node_const();
    uint32_t* kbuf = keys + (int64_t)blockIdx.x * k_stride;
    for (;;) {
        if (tid == 0) s_tile = atomicAdd(counter, 1);
        if (SELECT)
            for (int b = tid; b < 2048; b += BT) hist[b] = 0u;
        __syncthreads();
        const int64_t turn = s_tile;
        if (turn >= n_todo) break;
        const int64_t i = list ? (int64_t)list[turn] : turn;
        const int K = T.K[i];
        bool bad = (K < 1) || (K > K_tiles);
        int v[4];
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            v[a] = T.center_idx[i * 4 + a];
            bad |= (v[a] < 0) || (v[a] >= T.n_axis[a]);
        }
        const int Kc = bad ? 0 : K;
        const uint32_t mask = T.null_mask[i];
        const uint8_t* rowp[4];
#pragma unroll
        for (int a = 0; a < 4; ++a) rowp[a] = cnt + (int64_t)(T.axis_off[a] + (bad ? 0 : v[a])) * k_stride;
        int r_acc = 0, xs[4] = {0, 0, 0, 0};
        for (int k8 = tid * SPT; k8 < Kc; k8 += BT * SPT) {
            // k8 + SPT <= k_stride (k_stride is a multiple of 16): the loads stay in the row
            uint2 w[4];
#pragma unroll
            for (int a = 0; a < 4; ++a) w[a] = __ldg(reinterpret_cast<const uint2*>(rowp[a] + k8));
            float4 q[SPT];
#pragma unroll
            for (int j = 0; j < SPT; ++j) {
                q[j] = make_float4(INFINITY, INFINITY, INFINITY, INFINITY);
                if (k8 + j < Kc) {
                    int x[4];
#pragma unroll
                    for (int a = 0; a < 4; ++a)
                        x[a] = min((int)(((j < 4 ? w[a].x : w[a].y) >> (8 * (j & 3))) & 0xFFu), B.n);
                    q[j] = state_q<TABLE>(Qt, B, C, x);
                }
            }
            uint32_t kq[SPT];
#pragma unroll
            for (int j = 0; j < SPT; ++j) {
                float S = INFINITY;
                if (k8 + j < Kc) {
                    S = masked_min(q[j], mask);
                    const int rej = (S < lambda_up) ? 1 : 0;
                    r_acc += rej;
#pragma unroll
                    for (int a = 0; a < 4; ++a) {
                        const int x = min((int)(((j < 4 ? w[a].x : w[a].y) >> (8 * (j & 3))) & 0xFFu), B.n);
                        xs[a] += rej ? x : 0;
                    }
                    if (SELECT) atomicAdd(&hist[__float_as_uint(S) >> 21], 1u);
                }
                kq[j] = __float_as_uint(S);
            }
            if (SELECT) {
                *reinterpret_cast<uint4*>(kbuf + k8) = make_uint4(kq[0], kq[1], kq[2], kq[3]);
                *reinterpret_cast<uint4*>(kbuf + k8 + 4) = make_uint4(kq[4], kq[5], kq[6], kq[7]);
            }
        }
        r_acc = basket_warp_sum(r_acc);
#pragma unroll
        for (int a = 0; a < 4; ++a) xs[a] = basket_warp_sum(xs[a]);
        if (lane == 0) {
            s_red[0][warp] = r_acc;
            for (int a = 0; a < 4; ++a) s_red[1 + a][warp] = xs[a];
        }
        __syncthreads();
        double lam_i = -INFINITY;
        if (SELECT) {
            const int ks = bad ? 0 : o.ksel[i];
            if (ks >= 1) {
                int before1, before2, before3;
                const int b1 = block_find_kth<BT>(hist, 2048, ks, s_scan, s_res, &before1);
                for (int b = tid; b < 2048; b += BT) hist[b] = 0u;
                __syncthreads();
                for (int k = tid; k < Kc; k += BT) {
                    const uint32_t key = kbuf[k];
                    if ((int)(key >> 21) == b1) atomicAdd(&hist[(key >> 10) & 0x7FF], 1u);
                }
                const int b2 = block_find_kth<BT>(hist, 2048, ks - before1, s_scan, s_res, &before2);
                for (int b = tid; b < 1024; b += BT) hist[b] = 0u;
                __syncthreads();
                const uint32_t pre = ((uint32_t)b1 << 11) | (uint32_t)b2;
                for (int k = tid; k < Kc; k += BT) {
                    const uint32_t key = kbuf[k];
                    if ((key >> 10) == pre) atomicAdd(&hist[key & 0x3FF], 1u);
                }
                const int b3 = block_find_kth<BT>(hist, 1024, ks - before1 - before2, s_scan, s_res, &before3);
                lam_i = (double)__uint_as_float((pre << 10) | (uint32_t)b3);
            }
        }
        if (tid == 0) {
            basket_store(T, B, o, i, K, bad, v, s_red, BWARP, SELECT, lam_i, err);
            if (SELECT) s_min = min(s_min, order_key(lam_i));
        }
        __syncthreads();
    }
    queue_reset_min(counter, o.min_key, s_min, SELECT ? o.min_out : nullptr, blocks, false, list != nullptr);
}

template <bool TABLE>
__global__ void k_emit_basket(TileArgs T, Basket B, const uint8_t* __restrict__ cnt, int32_t k_stride,
                              int32_t K_tiles, const float4* __restrict__ Qt, const int64_t* __restrict__ off,
                              float* __restrict__ S_out, int32_t* __restrict__ err)
{
    NodeConst C;
    if (!TABLE) C = node_const();
    for (int64_t i = blockIdx.x; i < T.n_tiles; i += gridDim.x) {
        const int K = T.K[i];
        bool bad = (K < 1) || (K > K_tiles);
        int v[4];
        for (int a = 0; a < 4; ++a) {
            v[a] = T.center_idx[i * 4 + a];
            bad |= (v[a] < 0) || (v[a] >= T.n_axis[a]);
        }
        if (bad) {
            if (threadIdx.x == 0) atomicOr(err, CSE_ERR_BAD_K);
            continue;
        }
        const uint32_t mask = T.null_mask[i];
        for (int k = threadIdx.x; k < K; k += blockDim.x) {
            int x[4];
            for (int a = 0; a < 4; ++a)
                x[a] = min((int)cnt[(int64_t)(T.axis_off[a] + v[a]) * k_stride + k], B.n);
            S_out[off[i] + k] = masked_min(state_q<TABLE>(Qt, B, C, x), mask);
        }
    }
}

Basket make_basket(const DesignArgs& D)
{
    Basket B;
    B.n = D.look_n[0];
    B.m = B.n + 1;
    for (int a = 0; a < 4; ++a) B.t[a] = (float)D.tnull[a];
    return B;
}

// Blocks of a launch, and the key buffer for `words` words a block.
template <typename Kern>
int basket_grid(cse_ctx* c, Kern kern, int nt, size_t smem, int64_t tiles, int64_t words, int64_t* grid,
                cudaStream_t s)
{
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, nt, smem) != cudaSuccess || per_sm < 1) {
        cudaGetLastError();
        return CSE_CUDA_ERROR;
    }
    *grid = (int64_t)per_sm * c->num_sms;
    if (*grid > tiles) *grid = tiles;
    return words ? cse_reserve_keys(c, sizeof(uint32_t) * (size_t)words, grid, s) : CSE_OK;
}

template <bool SEL, int NT>
int launch_basket(cse_ctx* c, const TileArgs& T, int32_t k_stride, int32_t K_tiles, double lambda, const SimOut& o,
                  cudaStream_t s)
{
    // a warp's keys: its share of the sample and its 512 trials of every step
    const int32_t key_seg = kSample / (NT / 32) + (K_tiles + NT * 16 - 1) / (NT * 16) * 512;
    int64_t grid = 0;
    const Basket B = make_basket(c->D);
    const int span = basket_span(B.n), rows = B.m * B.m * B.m;
    // the words of the widest window, w_0 w_1 w_2 <= span^3, and word 0: at most 42,596 bytes (n = 63:
    // span 22), with the static arrays of 128 threads below the default limit of 48 KB, of 256 above
    const size_t smem = ((size_t)span * span * span + 1) * sizeof(uint32_t);
    if (NT > 128 && smem > 40 * 1024 &&   // one limit for every design: it belongs to the kernel
        cudaFuncSetAttribute(k_sim_basket<SEL, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, 42 * 1024) !=
            cudaSuccess) {
        cudaGetLastError();
        return CSE_CUDA_ERROR;
    }
    const float lam = lambda_float_up(lambda);
    const bool want_R = o.R || o.Xrej || o.score || o.cp_key;
    const int st = basket_grid(c, k_sim_basket<SEL, NT>, NT, smem, T.n_tiles, SEL ? (int64_t)(NT / 32) * key_seg : 0,
                               &grid, s);
    if (st != CSE_OK) return st;
    if (SEL && o.min_out) c->min_folded = true;
    if (o.cp_key) c->cp_marked = true;
    cse_prof_begin(c, KID_SIM_BASKET, s);
    if (want_R && K_tiles > kAllK) {   // the bits of this call's lambda
        k_basket_bits<<<(unsigned)((rows + 7) / 8), 256, 0, s>>>(c->bk_bits, c->bk_q, B.m, rows, kLevels, 1, lam);
        c->launches += 1;
    }
    // selections over more than kAllK trials leave the tiles without use for a test
    int32_t* left = SEL && K_tiles > kAllK ? c->left : nullptr;
    k_sim_basket<SEL, NT><<<(unsigned)grid, NT, smem, s>>>(T, B, c->cnt, k_stride, K_tiles, c->bk_q, c->bk_bits, span,
                                                          lam, want_R, o, c->keys, key_seg, left, c->counter, c->err);
    c->launches += 1;
    if (left) {   // a block's keys hold at least k_stride words
        int per_sm = 0;
        auto all = k_sim_basket_all<true, SEL>;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, all, BT, 0) != cudaSuccess || per_sm < 1) {
            cudaGetLastError();
            return CSE_CUDA_ERROR;
        }
        if (grid > (int64_t)per_sm * c->num_sms) grid = (int64_t)per_sm * c->num_sms;
        cse_launch(true, all, dim3((unsigned)grid), dim3(BT), 0, s, T, B, c->cnt, k_stride, K_tiles, c->bk_q, lam, o,
                   c->keys, left, c->counter, c->err);
        c->launches += 1;
    }
    cse_prof_end(c, s);
    return cudaGetLastError() == cudaSuccess ? CSE_OK : CSE_CUDA_ERROR;
}

template <bool SEL>
int launch_basket_direct(cse_ctx* c, const TileArgs& T, int32_t k_stride, int32_t K_tiles, double lambda,
                         const SimOut& o, cudaStream_t s)
{
    int64_t grid = 0;
    const int st = basket_grid(c, k_sim_basket_all<false, SEL>, BT, 0, T.n_tiles, SEL ? k_stride : 0, &grid, s);
    if (st != CSE_OK) return st;
    if (SEL && o.min_out) c->min_folded = true;
    if (o.cp_key) c->cp_marked = true;
    cse_prof_begin(c, KID_SIM_BASKET, s);
    k_sim_basket_all<false, SEL><<<(unsigned)grid, BT, 0, s>>>(T, make_basket(c->D), c->cnt, k_stride, K_tiles, nullptr,
                                                              lambda_float_up(lambda), o, c->keys, nullptr, c->counter,
                                                              c->err);
    cse_prof_end(c, s);
    c->launches += 1;
    return cudaGetLastError() == cudaSuccess ? CSE_OK : CSE_CUDA_ERROR;
}

}  // namespace

int cse_basket_setup(cse_ctx* c, cudaStream_t s)
{
    const Basket B = make_basket(c->D);
    const int64_t states = (int64_t)B.m * B.m * B.m * B.m;
    c->bt_tables = states <= CSE_BAYES_TABLE_MAX && B.m <= kMaxM;
    if (!c->bt_tables) return CSE_OK;   // direct evaluation per simulation
    const int rows = B.m * B.m * B.m;
    const size_t bits_bytes = (size_t)(kLevels + 1) * 4 * (size_t)rows * sizeof(uint2);
    if (cudaMalloc(&c->bk_q, (size_t)states * sizeof(float4)) != cudaSuccess ||
        cudaMalloc(&c->bk_bits, bits_bytes) != cudaSuccess) {
        cudaGetLastError();
        return CSE_OOM;
    }
    cse_prof_begin(c, KID_BASKET_TABLE, s);
    k_table_basket<<<(unsigned)((states + 255) / 256), 256, 0, s>>>(c->bk_q, B);
    cse_prof_end(c, s);
    // level +inf (kLevels - 1) is never read
    k_basket_bits<<<(unsigned)((rows + 7) / 8), 256, 0, s>>>(c->bk_bits, c->bk_q, B.m, rows, 0, kLevels - 1, 0.0f);
    c->launches += 2;
    return cudaGetLastError() == cudaSuccess ? CSE_OK : CSE_CUDA_ERROR;
}

int cse_launch_emit_basket(cse_ctx* c, const TileArgs& T, int32_t NA, int32_t k_stride, int32_t K_tiles,
                           const int64_t* off, float* S_out, cudaStream_t s)
{
    (void)NA;
    const int64_t grid = T.n_tiles < 4096 ? T.n_tiles : 4096;
    const Basket B = make_basket(c->D);
    if (c->bt_tables && !c->bt_direct)
        k_emit_basket<true><<<(unsigned)grid, 256, 0, s>>>(T, B, c->cnt, k_stride, K_tiles, c->bk_q, off, S_out,
                                                           c->err);
    else
        k_emit_basket<false><<<(unsigned)grid, 256, 0, s>>>(T, B, c->cnt, k_stride, K_tiles, c->bk_q, off, S_out,
                                                            c->err);
    c->launches += 1;
    return cudaGetLastError() == cudaSuccess ? CSE_OK : CSE_CUDA_ERROR;
}

int cse_launch_sim_basket(cse_ctx* c, const TileArgs& T, int32_t NA, int32_t k_stride, int32_t K_tiles,
                          double lambda, const SimOut& o, cudaStream_t s)
{
    (void)NA;
    const bool sel = (o.lam_tile != nullptr && o.ksel != nullptr);
    if (c->bt_tables && !c->bt_direct) {
        // 256 threads a tile while there are too few tiles to fill the SMs with blocks of 128
        if (T.n_tiles <= 4 * (int64_t)c->num_sms)
            return sel ? launch_basket<true, 256>(c, T, k_stride, K_tiles, lambda, o, s)
                       : launch_basket<false, 256>(c, T, k_stride, K_tiles, lambda, o, s);
        return sel ? launch_basket<true, 128>(c, T, k_stride, K_tiles, lambda, o, s)
                   : launch_basket<false, 128>(c, T, k_stride, K_tiles, lambda, o, s);
    }
    return sel ? launch_basket_direct<true>(c, T, k_stride, K_tiles, lambda, o, s)
               : launch_basket_direct<false>(c, T, k_stride, K_tiles, lambda, o, s);
}
