// sim_bayes4.cu -- the four-arm Bayesian selection design (control + 3
// treatments, interim analyses after look_n[0] and look_n[1] patients per arm,
// final analysis after look_n[2]) with the hierarchical model of Sec. 10.1:
//   theta_i ~ N(mu, s2), mu ~ N(-1.34, 100), s2 ~ InvGamma(0.0005, 0.000005),
// each arm's likelihood replaced by the normal approximation of its empirical
// logit, s2 integrated on 16 log-spaced nodes in [1e-6, 1e3] (trapezoid in
// log s2, weights normalised by log-sum-exp), mu and theta integrated exactly.
// Interim: drop treatment i when P(theta_i > theta_0 | data) < drop (its data
// stay in the model, frozen).  Final: S = min over active true-null arms of
// 1 - P_i; reject iff S < lambda.  The posterior runs in FP32.
//
// The design depends on a simulated trial only through its success counts, so
// the posterior is tabulated once per context over every reachable count state
// (interim drop decisions and final-look probabilities); a simulation then costs
// count reads and a few table reads.  Treatments are exchangeable in the model,
// so the final-look table holds, per control count and sorted triple of
// treatment codes, the three P(theta_self > theta_0) side by side (one float4:
// one 16-byte read per trial), each evaluated with the arms in the canonical
// order (control, self, the other two ascending).  A direct mode evaluates the
// same FP32 posterior function per simulation instead of reading tables.
#include <cuda_runtime.h>
#include <math.h>

#include <type_traits>

#include "cse_internal.cuh"

namespace {

constexpr int NODES = kBayesNodes;   // quadrature nodes of s2 (node_const)
constexpr int BT = 256;          // threads of the simulation kernel
constexpr int BWARP = BT / 32;

// P(theta_i > theta_0 | data) for i = 1..3 in FP32.  Not inlined, so every caller
// runs the same instruction sequence (identical results for identical inputs).
__device__ __noinline__ void posterior4_f32(const int* x, const int* n, const NodeConst& C, float* P)
{
    const float MU0 = -1.34f, TAU2 = 100.0f;
    float th[4], s2[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float xs = (float)x[i] + 0.5f, fs = (float)(n[i] - x[i]) + 0.5f;
        th[i] = logf(xs / fs);
        s2[i] = 1.0f / xs + 1.0f / fs;
    }
    float lw[NODES], pj[NODES][3];
    float mx = -INFINITY;
#pragma unroll 4
    for (int j = 0; j < NODES; ++j) {
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
        const float prec = 1.0f / TAU2 + W;
        const float quad = Srr - Sr * Sr / prec;
        const float logdet = logf(prod * (1.0f + TAU2 * W));
        lw[j] = C.lprior[j] - 0.5f * logdet - 0.5f * quad;
        mx = fmaxf(mx, lw[j]);
        const float mmu = (MU0 / TAU2 + Sth) / prec;
        const float vmu = 1.0f / prec;
        float c[4], v[4], e[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            c[i] = s2[i] * w[i];
            v[i] = s2[i] * sg * w[i];
            e[i] = (1.0f - c[i]) * th[i] + c[i] * mmu;
        }
#pragma unroll
        for (int i = 1; i < 4; ++i) {
            const float md = e[i] - e[0];
            const float dc = c[i] - c[0];
            const float vd = v[i] + v[0] + dc * dc * vmu;
            pj[j][i - 1] = normcdff(md * rsqrtf(vd));
        }
    }
    float Z = 0.f, a0 = 0.f, a1 = 0.f, a2 = 0.f;
#pragma unroll
    for (int j = 0; j < NODES; ++j) {
        const float wj = expf(lw[j] - mx);
        Z += wj;
        a0 += wj * pj[j][0];
        a1 += wj * pj[j][1];
        a2 += wj * pj[j][2];
    }
    P[0] = a0 / Z;
    P[1] = a1 / Z;
    P[2] = a2 / Z;
}

// Treatment-state codes: at the second analysis, code < n1+1 is "dropped at the
// first analysis with x successes of n1", else "active with x = code-(n1+1) of
// n2"; at the final analysis codes < n1+1 and < n1+1+n2+1 are dropped at the
// first / second analysis, the rest active with x = code-(n1+1)-(n2+1) of n3.
struct Looks {
    int n1, n2, n3, S2, S3, NP;   // NP = S3 (S3 + 1) / 2 unordered pairs
    int NT;                       // S3 (S3 + 1) (S3 + 2) / 6 sorted triples
};

// Position of the sorted triple a <= b <= c among all sorted triples of codes
// (combinatorial number system).
__device__ __forceinline__ int triple_index(int a, int b, int c)
{
    return c * (c + 1) * (c + 2) / 6 + b * (b + 1) / 2 + a;
}

__device__ __forceinline__ void decode3(const Looks& L, int code, int* x, int* n)
{
    if (code <= L.n1) {
        *x = code;
        *n = L.n1;
    } else if (code <= L.n1 + 1 + L.n2) {
        *x = code - (L.n1 + 1);
        *n = L.n2;
    } else {
        *x = code - (L.n1 + 1) - (L.n2 + 1);
        *n = L.n3;
    }
}

__global__ void k_table_d1(uint8_t* __restrict__ D1, Looks L, float drop)
{
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    const int m = L.n1 + 1;
    __shared__ NodeConst C;
    node_const_block(C);
    if (s >= m * m * m * m) return;
    int x[4] = {s / (m * m * m), (s / (m * m)) % m, (s / m) % m, s % m};
    int n[4] = {L.n1, L.n1, L.n1, L.n1};
    float P[3];
    posterior4_f32(x, n, C, P);
    D1[s] = (uint8_t)((P[0] < drop ? 1 : 0) | (P[1] < drop ? 2 : 0) | (P[2] < drop ? 4 : 0));
}

// Drop bits at the second analysis of the three treatments with codes t[0..2]
// (control: c successes of n2).  The posterior is evaluated with the treatments
// in ascending code order and the bits mapped back, so the result depends on the
// codes only as a multiset, permuted with them: treatments with equal codes hold
// equal data, and the FP32 evaluation gives them equal probabilities in either
// order.  Both the tables and the direct mode use this function.
__device__ __forceinline__ int d2_bits(const Looks& L, const NodeConst& C, float drop, int c, const int t[3])
{
    int v[3] = {4 * t[0], 4 * t[1] + 1, 4 * t[2] + 2};   // code, then treatment
    int lo = min(v[0], v[1]);
    v[1] = max(v[0], v[1]);
    v[0] = lo;
    lo = min(v[1], v[2]);
    v[2] = max(v[1], v[2]);
    v[1] = lo;
    lo = min(v[0], v[1]);
    v[1] = max(v[0], v[1]);
    v[0] = lo;
    int x[4], n[4];
    x[0] = c;
    n[0] = L.n2;
    for (int k = 0; k < 3; ++k) {
        const int code = v[k] >> 2;
        if (code <= L.n1) {
            x[k + 1] = code;
            n[k + 1] = L.n1;
        } else {
            x[k + 1] = code - (L.n1 + 1);
            n[k + 1] = L.n2;
        }
    }
    float P[3];
    posterior4_f32(x, n, C, P);
    int bits = 0;
    for (int k = 0; k < 3; ++k)
        if (P[k] < drop) bits |= 1 << (v[k] & 3);
    return bits;
}

__global__ void k_table_d2(uint8_t* __restrict__ D2, Looks L, float drop)
{
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    const int S2 = L.S2;
    __shared__ NodeConst C;
    node_const_block(C);
    if (s >= (L.n2 + 1) * S2 * S2 * S2) return;
    const int c = s / (S2 * S2 * S2);
    const int t[3] = {(s / (S2 * S2)) % S2, (s / S2) % S2, s % S2};
    D2[s] = (uint8_t)d2_bits(L, C, drop, c, t);
}

// (a, b, z) with a <= b <= z and z (z + 1) (z + 2) / 6 + b (b + 1) / 2 + a = r.
__device__ __forceinline__ void decode_triple(int r, int* a, int* b, int* z)
{
    int zz = (int)cbrtf(6.0f * (float)r);   // largest z with z (z + 1) (z + 2) / 6 <= r
    while (zz > 0 && zz * (zz + 1) * (zz + 2) / 6 > r) --zz;
    while ((zz + 1) * (zz + 2) * (zz + 3) / 6 <= r) ++zz;
    const int r2 = r - zz * (zz + 1) * (zz + 2) / 6;
    int bb = (int)floorf((sqrtf(8.0f * r2 + 1.0f) - 1.0f) * 0.5f);   // largest b with b (b + 1) / 2 <= r2
    while (bb > 0 && bb * (bb + 1) / 2 > r2) --bb;
    while ((bb + 1) * (bb + 2) / 2 <= r2) ++bb;
    *a = r2 - bb * (bb + 1) / 2;
    *b = bb;
    *z = zz;
}

// The second-analysis drop bits over sorted code triples only, three bits an
// entry, ten entries a 32-bit word: entry e = c * NT2 + tri(a, b, z) (a <= b <= z
// < S2, NT2 = S2 (S2 + 1) (S2 + 2) / 6) sits in word e / 10 at bit 3 (e % 10)
// and holds D2[c][a][b][z], whose bit k belongs to the treatment at sorted
// position k.  By the symmetry of d2_bits this is all of D2.
__global__ void k_table_d2s(uint32_t* __restrict__ D2s, const uint8_t* __restrict__ D2, Looks L, int32_t nt2)
{
    const int64_t word = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t tot = (int64_t)(L.n2 + 1) * nt2;
    if (10 * word >= tot) return;
    const int S2 = L.S2;
    uint32_t out = 0u;
    for (int h = 0; h < 10; ++h) {
        const int64_t e = 10 * word + h;
        if (e >= tot) break;
        const int c = (int)(e / nt2);
        int a, b, z;
        decode_triple((int)(e % nt2), &a, &b, &z);
        out |= (uint32_t)(D2[((c * S2 + a) * S2 + b) * S2 + z] & 7) << (3 * h);
    }
    D2s[word] = out;
}

// F4[c * NT + triple_index(A, B, Z)] = (P_A, P_B, P_Z, 0) for the sorted codes
// A <= B <= Z: P_A = P(theta_A > theta_0) with the arms ordered (control, A, B, Z),
// P_B with (control, B, A, Z), P_Z with (control, Z, A, B).
__global__ void k_table_f4(float4* __restrict__ F4, Looks L)
{
    const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t tot = (int64_t)(L.n3 + 1) * L.NT;
    __shared__ NodeConst C;
    node_const_block(C);
    if (s >= tot) return;
    const int c = (int)(s / L.NT);
    int a, b, z;
    decode_triple((int)(s % L.NT), &a, &b, &z);
    const int self[3] = {a, b, z}, lo[3] = {b, a, a}, hi[3] = {z, z, b};
    float out[3];
    for (int k = 0; k < 3; ++k) {
        int x[4], n[4];
        x[0] = c;
        n[0] = L.n3;
        decode3(L, self[k], &x[1], &n[1]);
        decode3(L, lo[k], &x[2], &n[2]);
        decode3(L, hi[k], &x[3], &n[3]);
        float P[3];
        posterior4_f32(x, n, C, P);
        out[k] = P[0];
    }
    F4[s] = make_float4(out[0], out[1], out[2], 0.0f);
}

// P_self at the final analysis evaluated directly, with the canonical arm order.
__device__ __forceinline__ float final_p_direct(const Looks& L, const NodeConst& C, int c, int self, int o1, int o2)
{
    const int ta = min(o1, o2), tb = max(o1, o2);
    int x[4], n[4];
    x[0] = c;
    n[0] = L.n3;
    decode3(L, self, &x[1], &n[1]);
    decode3(L, ta, &x[2], &n[2]);
    decode3(L, tb, &x[3], &n[3]);
    float P[3];
    posterior4_f32(x, n, C, P);
    return P[0];
}

// Statistic S of one simulated trial from its cumulative counts xl[look][arm].
template <bool TABLES>
__device__ __forceinline__ float design_stat(const Looks& L, const uint8_t* __restrict__ D1,
                                             const uint8_t* __restrict__ D2, const float4* __restrict__ F4,
                                             const NodeConst& C, float drop, const int xl[3][4], uint32_t mask)
{
    // first analysis: every arm at n1
    int bits;
    if (TABLES) {
        const int m = L.n1 + 1;
        // D1 may live in shared memory: a generic load (not the global-only __ldg)
        bits = D1[((xl[0][0] * m + xl[0][1]) * m + xl[0][2]) * m + xl[0][3]];
    } else {
        int x[4] = {xl[0][0], xl[0][1], xl[0][2], xl[0][3]};
        int n[4] = {L.n1, L.n1, L.n1, L.n1};
        float P[3];
        posterior4_f32(x, n, C, P);
        bits = (P[0] < drop ? 1 : 0) | (P[1] < drop ? 2 : 0) | (P[2] < drop ? 4 : 0);
    }
    int drop1 = bits & 7;                       // dropped at the first analysis
    if (drop1 == 7) return INFINITY;
    int t2[3];
#pragma unroll
    for (int i = 0; i < 3; ++i)
        t2[i] = ((drop1 >> i) & 1) ? xl[0][i + 1] : (L.n1 + 1) + xl[1][i + 1];
    if (TABLES) {
        bits = __ldg(D2 + ((xl[1][0] * L.S2 + t2[0]) * L.S2 + t2[1]) * L.S2 + t2[2]);
    } else {
        bits = d2_bits(L, C, drop, xl[1][0], t2);
    }
    const int drop2 = bits & 7 & ~drop1;        // dropped at the second analysis
    if ((drop1 | drop2) == 7) return INFINITY;
    int t3[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        if ((drop1 >> i) & 1) t3[i] = xl[0][i + 1];
        else if ((drop2 >> i) & 1) t3[i] = (L.n1 + 1) + xl[1][i + 1];
        else t3[i] = (L.n1 + 1) + (L.n2 + 1) + xl[2][i + 1];
    }
    const int use = 7 & ~(drop1 | drop2) & (int)mask;   // active true-null treatments
    float S = INFINITY;
    if (TABLES) {
        if (use) {
            // sort the three codes with each treatment's bit of `use` below them
            // (2 code + bit): equal codes have equal table entries, so the order
            // between them does not matter, and each sorted position carries its
            // own bit, so no permutation is tracked
            int v0 = 2 * t3[0] + (use & 1), v1 = 2 * t3[1] + ((use >> 1) & 1), v2 = 2 * t3[2] + ((use >> 2) & 1);
            int lo = min(v0, v1);
            v1 = max(v0, v1);
            v0 = lo;
            lo = min(v1, v2);
            v2 = max(v1, v2);
            v1 = lo;
            lo = min(v0, v1);
            v1 = max(v0, v1);
            v0 = lo;
            // the tables exist only when they hold at most 2^27 floats: a 32-bit index
            const float4 q = __ldg(F4 + (xl[2][0] * L.NT + triple_index(v0 >> 1, v1 >> 1, v2 >> 1)));
            // min over the counted treatments of 1 - P_i, as 1 - max P_i: x -> 1 - x
            // rounds monotonically, so the two agree bit for bit
            float pm = -1.0f;
            if (v0 & 1) pm = fmaxf(pm, q.x);
            if (v1 & 1) pm = fmaxf(pm, q.y);
            if (v2 & 1) pm = fmaxf(pm, q.z);
            S = 1.0f - pm;
        }
    } else {
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            if ((use >> i) & 1) {
                const float p = final_p_direct(L, C, xl[2][0], t3[i], t3[(i + 1) % 3], t3[(i + 2) % 3]);
                S = fminf(S, 1.0f - p);
            }
        }
    }
    return S;
}

// The tabulated statistic with one trial's counts packed one arm per byte,
// Pl = [x_l0, x_l1, x_l2, x_l3] for look l (valid while every final-look code
// fits seven bits: S3 <= 128).  The same table reads as design_stat<true>, with
// the index and code arithmetic done on whole words:
// - the first-look index ((x0 m + x1) m + x2) m + x3 as (x0 m + x1) m^2 +
//   (x2 m + x3), m = n1 + 1, by two dot products of the packed bytes with packed
//   radix weights (dp4a);
// - the second-look drop bits from a table over sorted code triples held in
//   shared memory (the per-trial global gather of the full table was a fifth of
//   the kernel's time), three bits an entry, and the first-look bits four bits an
//   entry: the less shared memory the two CTAs of an SM take, the more is left
//   to L1 for the final-table gathers;
// - the codes of the next look chosen per treatment by one byte permutation:
//   byte i + 1 comes from the previous codes if treatment i was dropped, else
//   from this look's counts plus the code offset (n1 + 1, then S2).  The
//   permutation's selector is 0x7654 with bit 2 of nibble i + 1 cleared for each
//   dropped treatment: the three drop bits spread to bits 6, 10, 14 by one
//   multiply (d * 0x1240) and mask (0x4440).
struct PackedConst {
    uint32_t w1hi, w1lo, m1sq;   // first-look index weights: [m, 1, 0, 0], [0, 0, m, 1], m^2
    uint32_t off1, off2;         // code offsets on bytes 1..3: n1 + 1, S2
    int32_t nt2;                 // sorted code triples of the second analysis
};

__device__ __forceinline__ float design_stat_packed(const Looks& L, const PackedConst& Q, const uint8_t* D1,
                                                    const uint32_t* D2s, const float4* __restrict__ F4, const int* tri,
                                                    const uint32_t* perm, uint32_t P0, uint32_t P1, uint32_t P2,
                                                    uint32_t mask)
{
    // Branch-free: a trial with every treatment dropped (or none counted) runs
    // the whole sequence, every index staying within its table for any counts,
    // and gets +inf at the end; the trials of a step then form one straight
    // block that the compiler interleaves (measured: 26.8 -> 25.6 ms on the
    // refined-platten sample, with the step's bounds checks only in the tail)
    const uint32_t i1 = __dp4a(P0, Q.w1hi, 0u) * Q.m1sq + __dp4a(P0, Q.w1lo, 0u);
    const uint32_t drop1 = ((uint32_t)D1[i1 >> 1] >> ((i1 & 1u) << 2)) & 7u;   // two entries a byte
    // [x_10, codes of the three treatments at the second analysis]
    const uint32_t T2 = __byte_perm(P0, P1 + Q.off1, ((drop1 * 0x1240u) & 0x4440u) ^ 0x7654u);
    // second analysis: the codes sorted with the treatment index below them
    // (4 code + i), the sorted-triple table (k_table_d2s) in shared memory, and
    // the bits of the sorted positions mapped back to the treatments by perm
    const uint32_t V2 = ((T2 << 2) & 0xFCFCFC00u) | 0x02010000u;
    int u0 = (int)((V2 >> 8) & 0xFFu), u1 = (int)((V2 >> 16) & 0xFFu), u2 = (int)(V2 >> 24);
    int lo2 = min(u0, u1);
    u1 = max(u0, u1);
    u0 = lo2;
    lo2 = min(u1, u2);
    u2 = max(u1, u2);
    u1 = lo2;
    lo2 = min(u0, u1);
    u1 = max(u0, u1);
    u0 = lo2;
    const int e2 = (int)(T2 & 0xFFu) * Q.nt2 + tri[768 + u2] + tri[512 + u1] + (u0 >> 2);
    const uint32_t w2 = __umulhi((uint32_t)e2, 0xCCCCCCCDu) >> 3;   // e2 / 10 (exact below 2^32)
    const uint32_t nib = (D2s[w2] >> (3u * ((uint32_t)e2 - 10u * w2))) & 7u;
    const uint32_t dd = drop1 | ((perm[((u0 & 3) << 2) | (u1 & 3)] >> (3u * nib)) & 7u);
    // [x_20, codes at the final analysis]
    const uint32_t T3 = __byte_perm(T2, P2 + Q.off2, ((dd * 0x1240u) & 0x4440u) ^ 0x7654u);
    const uint32_t use = 7u & ~dd & mask;   // active true-null treatments
    // bytes 1..3: 2 code + the treatment's bit of `use`, sorted as in design_stat
    const uint32_t V = ((T3 << 1) & 0xFEFEFE00u) | ((use * 0x408100u) & 0x01010100u);
    int v0 = (int)((V >> 8) & 0xFFu), v1 = (int)((V >> 16) & 0xFFu), v2 = (int)(V >> 24);
    int lo = min(v0, v1);
    v1 = max(v0, v1);
    v0 = lo;
    lo = min(v1, v2);
    v2 = max(v1, v2);
    v1 = lo;
    lo = min(v0, v1);
    v1 = max(v0, v1);
    v0 = lo;
    // tri[v] = b (b + 1) / 2 and tri[256 + v] = c (c + 1) (c + 2) / 6 for b, c = v >> 1
    const float4 q = __ldg(F4 + ((int)(T3 & 0xFFu) * L.NT + tri[256 + v2] + tri[v1] + (v0 >> 1)));
    float pm = -1.0f;
    if (v0 & 1) pm = fmaxf(pm, q.x);
    if (v1 & 1) pm = fmaxf(pm, q.y);
    if (v2 & 1) pm = fmaxf(pm, q.z);
    return use == 0u ? INFINITY : 1.0f - pm;
}

// Four words of four trials each, an arm a word, to a word a trial, an arm a byte.
__device__ __forceinline__ void transpose4(const uint32_t in[4], uint32_t out[4])
{
    const uint32_t t0 = __byte_perm(in[0], in[1], 0x5140u), t1 = __byte_perm(in[2], in[3], 0x5140u);
    const uint32_t t2 = __byte_perm(in[0], in[1], 0x7362u), t3 = __byte_perm(in[2], in[3], 0x7362u);
    out[0] = __byte_perm(t0, t1, 0x5410u);
    out[1] = __byte_perm(t0, t1, 0x7632u);
    out[2] = __byte_perm(t2, t3, 0x5410u);
    out[3] = __byte_perm(t2, t3, 0x7632u);
}

__device__ __forceinline__ int warp_sum_i(int v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Block-wide: index b of the bin holding the ks-th (1-indexed) element of
// hist[0..nb), and the count of elements in bins before b.  All threads call.
template <int NTH>
__device__ void find_kth(const uint32_t* hist, int nb, int ks, int* s_scan, int* s_res, int* out_b, int* out_before)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int CH = (nb + NTH - 1) / NTH;
    const int b0 = tid * CH, b1 = min(b0 + CH, nb);
    int local = 0;
    for (int b = b0; b < b1; ++b) local += (int)hist[b];
    int incl = local;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += y;
    }
    if (lane == 31) s_scan[warp] = incl;
    if (tid == 0) {
        s_res[0] = -1;
        s_res[1] = 0;
    }
    __syncthreads();
    int wpre = 0;
    for (int w = 0; w < warp; ++w) wpre += s_scan[w];
    incl += wpre;
    const int excl = incl - local;
    if (excl < ks && ks <= incl) {
        int cum = excl;
        for (int b = b0; b < b1; ++b) {
            const int h = (int)hist[b];
            if (cum + h >= ks) {
                s_res[0] = b;
                s_res[1] = cum;
                break;
            }
            cum += h;
        }
    }
    __syncthreads();
    *out_b = s_res[0];
    *out_before = s_res[1];
    __syncthreads();
}

// Shared memory of the packed form: tri[v] = c (c + 1) / 2 and tri[256 + v] =
// c (c + 1) (c + 2) / 6 for c = v >> 1 (final-look codes with their use bit),
// tri[512 + u], tri[768 + u] the same for c = u >> 2 (second-look codes with the
// treatment index); perm[(t0 << 2) | t1] maps the drop bits of the sorted
// positions to the treatments (t0, t1, 3 - t0 - t1) at those positions: bits B
// go to (perm >> 3 B) & 7.
__device__ __forceinline__ void packed_tables(int tid, int nth, int* tri, uint32_t* perm)
{
    for (int v = tid; v < 256; v += nth) {
        const int b = v >> 1, c = v >> 2;
        tri[v] = b * (b + 1) / 2;
        tri[256 + v] = b * (b + 1) * (b + 2) / 6;
        tri[512 + v] = c * (c + 1) / 2;
        tri[768 + v] = c * (c + 1) * (c + 2) / 6;
    }
    if (tid < 16) {
        const int t0 = tid >> 2, t1 = tid & 3, t2 = 3 - t0 - t1;
        uint32_t m = 0u;
        if (t0 < 3 && t1 < 3 && t0 != t1 && t2 >= 0 && t2 < 3 && t2 != t0 && t2 != t1)
            for (uint32_t B = 0; B < 8; ++B)
                m |= ((((B & 1u) << t0) | (((B >> 1) & 1u) << t1) | (((B >> 2) & 1u) << t2))) << (3u * B);
        perm[tid] = m;
    }
}

// ---------------------------------------------------------------------------
// The tabulated simulation: only the trials that can decide anything are
// evaluated.
//
// A tile's outputs depend on the trials with S < lambda (R, Xrej, score) and on
// the k_i smallest S (k_i / K_i <= alpha: about two in a hundred), yet the drop
// decisions and the final-table gather cost ~140 thread instructions a trial.
// A lower bound on S from the final counts alone settles the rest.  With a
// strictly rising score u of the final counts and D = max over the counted
// treatments of u(count) - u(control's count),
//   D < d  =>  S >= sigma(d) := min over the final-table entries of an active
//                               treatment with score difference at most d - 1,
// for any drop pattern, since every counted treatment's 1 - P is such an entry
// (k_table_dmin).  A pass at difference d therefore evaluates the candidates
// D >= d only: exact for R when lambda <= sigma(d), and for the order statistic
// when the k_i-th smallest S among the candidates is at most sigma(d) (checked;
// otherwise the pass is repeated at a lower d, down to every trial).
//
// The score is the angular transform asin(sqrt(.)), scaled to 0 .. 98: with raw
// counts one difference means a smaller S for counts near 0 or n than in the
// middle, and sigma(d) has to cover the worst (refined platten, d chosen with
// hindsight: 21 % of the trials are candidates by raw counts, 14 % by score, 10 %
// by the exact two-argument bound; 2.3 % are needed).
//
// The test D >= d runs on packed bytes, four trials a word: bit 7 of byte
// u_i + (0x80 - d - u_0), no carry crossing a byte for the d allowed: 1.5
// instructions a trial.  Each warp queues its candidates in shared memory and
// evaluates them 32 at a time.  A tile starts with its first kSample trials, all
// evaluated, and raises d after them and after 1, 2, 4, ... steps as far as the
// keys found so far allow with a margin that shrinks to zero towards the end.
// Keys go to the CTA's own stretch of global memory (4 % of the trials) and into
// 256 bins of 1/16 octave; the order statistic is ranked within its bin.
//
// A warp of whose 512 trials of a step more than kDense are candidates evaluates all of
// them, a lane four consecutive trials from whole count words: no queue, no scattered
// bytes (a candidate costs about twice a trial read that way).
//
// What bounds it: issue slots at the latency of the candidates' scattered reads (71 %
// issue, 64 % ALU pipe, 62 to 68 warp instructions per 32 trials of which the candidates,
// ~290 each, take four fifths).  262,144 refined tiles x 65,536 trials: 103 -> 36.8 ms; the
// 16^4 grid at K = 2^14: 5.6 -> 1.9 ms.  Measured on the way: evaluating every candidate
// by raw counts with a margin fixed by the sample 65 ms, with d raised along the pass
// 51 ms; final-table loads that skip L1 lost 10 %.  Levels that make most trials
// candidates, 8^4 grid at K = 2^14, the whole call (every trial in a straight line / all
// through the queue / now): validation at lambda = 1 570 / 616 / 475 us, calibration at
// alpha = 0.3 530 / 568 / 471, at 0.5 534 / 635 / 540.
//
// Tiles: a group of NT / G threads per tile (named barriers), G tiles a block;
// G = 1 only when there are too few tiles to give every group one.
// ---------------------------------------------------------------------------
constexpr double kScoreTop = 98.0;   // largest score (differences then span -29 .. 30 without carries)
constexpr int kSample = 512;     // first trials of a tile, all evaluated to place d
constexpr int kAllK = 1024;      // up to this K every trial is evaluated
constexpr int kQueue = 288;      // a warp's candidate queue (up to 31 left over, at least 16 lanes' trials a round)
constexpr int kList = 256;       // keys of the selected bin ranked in shared memory
constexpr int kDense = 320;      // candidates among a warp's 512 trials of a step from which all are evaluated

// dmin[D + u(n3)] (float bits, preset to +inf) = the least S an active treatment
// with final score difference D to the control can give, over every state of the
// final table.
__global__ void __launch_bounds__(256) k_table_dmin(const float4* __restrict__ F4, Looks L,
                                                    const uint8_t* __restrict__ score, uint32_t* __restrict__ dmin)
{
    __shared__ uint32_t m[2 * CSE_MAX_NMAX + 1];
    __shared__ int u[CSE_MAX_NMAX + 1];
    for (int j = threadIdx.x; j <= 2 * CSE_MAX_NMAX; j += blockDim.x) m[j] = 0x7F800000u;
    for (int j = threadIdx.x; j <= L.n3; j += blockDim.x) u[j] = score[j];
    __syncthreads();
    const int top = u[L.n3];
    const int64_t tot = (int64_t)(L.n3 + 1) * L.NT;
    for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < tot; s += (int64_t)gridDim.x * blockDim.x) {
        int t[3];
        decode_triple((int)(s % L.NT), &t[0], &t[1], &t[2]);
        const int c = (int)(s / L.NT);
        const float4 q = __ldg(F4 + s);
        const float p[3] = {q.x, q.y, q.z};
#pragma unroll
        for (int k = 0; k < 3; ++k)   // 0 <= P <= 1 (a0 <= Z term by term), so S's bits order as integers
            if (t[k] >= L.S2) atomicMin(&m[u[t[k] - L.S2] - u[c] + top], __float_as_uint(1.0f - fmaxf(-1.0f, p[k])));
    }
    __syncthreads();
    for (int j = threadIdx.x; j <= 2 * top; j += blockDim.x)
        if (m[j] != 0x7F800000u) atomicMin(&dmin[j], m[j]);
}

// Threads and blocks per SM: the packed form's shared-memory tables (57.6 KB)
// and queues leave room for two blocks of 512; the byte form reads its tables
// from global memory.
template <bool PACKED>
constexpr int b4_threads()
{
    return PACKED ? 512 : BT;
}

template <bool PACKED, int G>
constexpr int b4_group()
{
    return b4_threads<PACKED>() / G;
}

template <bool SELECT, bool PACKED, int G, typename Off>
__global__ void __launch_bounds__(b4_threads<PACKED>(), PACKED ? 2 : 4)
    k_sim_bayes4(TileArgs T, Looks L, const uint8_t* __restrict__ cnt, int32_t NA, int32_t k_stride, int32_t K_tiles,
                 const uint8_t* __restrict__ D1g, const uint8_t* __restrict__ D2, const float4* __restrict__ F4,
                 const uint8_t* __restrict__ score, const uint32_t* __restrict__ dmin, int32_t top, int32_t dlo,
                 int32_t nd, float lambda_up, bool want_R, SimOut o, uint32_t* __restrict__ keys, int32_t key_seg,
                 int32_t* __restrict__ counter, int32_t* __restrict__ err, const PackedConst Q,
                 const uint32_t* __restrict__ D2sg, int32_t d1_bytes, int32_t d2s_bytes)
{
    constexpr int NT = b4_threads<PACKED>();
    constexpr int TT = b4_group<PACKED, G>();
    constexpr int NW = TT / 32;
    __shared__ int s_tri[PACKED ? 1024 : 1];
    __shared__ uint32_t s_perm[PACKED ? 16 : 1];
    __shared__ uint8_t s_inv[PACKED ? 128 : 1];   // final count of each score
    __shared__ uint32_t s_raw[2 * CSE_MAX_NMAX + 1];
    __shared__ float s_sig[2 * CSE_MAX_NMAX + 2];   // sigma(dlo + e), e < nd; +inf at e = 0 (every trial)
    __shared__ int s_sbin[2 * CSE_MAX_NMAX + 2];    // its bin (256 at e = 0)
    __shared__ int s_tile[G], s_next[G], s_pick[G], s_before[G], s_nlist[G], s_nk[G][NW];
    __shared__ uint32_t s_res[G];
    __shared__ int s_red[G][5][NW];
    __shared__ unsigned long long s_min[G];   // order key of the least lambda_i of the group's tiles
    // first-analysis drop table (two entries a byte) and, at d1_bytes (a multiple
    // of 16), the sorted second-analysis table; then the warps' queues, the keys
    // and the digit histograms
    extern __shared__ __align__(16) uint8_t smem[];
    const int tid = threadIdx.x, lane = tid & 31;
    const int g = tid / TT, lt = tid - g * TT, warp = lt >> 5;   // group, thread and warp in the group
    const uint32_t* D2s = reinterpret_cast<const uint32_t*>(smem + d1_bytes);
    uint32_t* const hists = reinterpret_cast<uint32_t*>(smem + d1_bytes + d2s_bytes);
    uint32_t* const hist = hists + g * 256;
    uint32_t* const list = hists + G * 256 + (SELECT ? g * kList : 0);
    uint16_t* const queue =
        reinterpret_cast<uint16_t*>(hists + G * 256 + (SELECT ? G * kList : 0)) + (tid >> 5) * kQueue;
    // each warp appends its keys to its own stretch of key_seg words
    uint32_t* const kgrp = keys + (int64_t)(blockIdx.x * G + g) * NW * key_seg;
    uint32_t* const kbuf = kgrp + (int64_t)warp * key_seg;
    const unsigned below = (1u << lane) - 1u;

    if (PACKED) {
        const int m = L.n1 + 1, n1t = m * m * m * m;
        for (int b = tid; 2 * b < n1t; b += NT)
            smem[b] = (uint8_t)((D1g[2 * b] & 7) | ((2 * b + 1 < n1t ? D1g[2 * b + 1] & 7 : 0) << 4));
        packed_tables(tid, NT, s_tri, s_perm);
        // d2s_bytes: a multiple of 16, within the global table's allocation
        for (int b = tid; b < d2s_bytes / 16; b += NT)
            reinterpret_cast<uint4*>(smem + d1_bytes)[b] = __ldg(reinterpret_cast<const uint4*>(D2sg) + b);
    }
    if (PACKED)
        for (int x = tid; x <= L.n3; x += NT) s_inv[score[x]] = (uint8_t)x;   // the scores are distinct
    for (int j = tid; j <= 2 * top; j += NT) s_raw[j] = dmin[j];
    for (int b = tid; b < G * 256; b += NT) hists[b] = 0u;
    if (tid < G) s_min[tid] = ~0ull;
    __syncthreads();
    for (int e = tid; e < nd; e += NT) {
        uint32_t v = 0x7F800000u;   // difference values below d = dlo + e
        if (e > 0)
            for (int j = 0; j < dlo + e + top; ++j) v = min(v, s_raw[j]);
        s_sig[e] = __uint_as_float(v);
        s_sbin[e] = e > 0 ? key_bin(v) : 256;
    }
    __syncthreads();
    int e_lam = nd - 1;   // the highest d that is exact for the rejections
    if (want_R) {
        e_lam = 0;
        for (int e = nd - 1; e > 0; --e)
            if (s_sig[e] >= lambda_up) {
                e_lam = e;
                break;
            }
    }

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
        bool bad = (K < 1) || (K > K_tiles);
        int v[4];
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            v[a] = T.center_idx[i * 4 + a];
            bad |= (v[a] < 0) || (v[a] >= T.n_axis[a]);
        }
        const uint32_t mask = T.null_mask[i] & 7u;   // counted treatments (none: S = +inf throughout)
        const int Kc = (bad || mask == 0u) ? 0 : K;
        // offsets of each arm's row of final scores; its interim rows lie whole
        // planes before it
        Off row[4];
        const Off plane = (Off)NA * (Off)k_stride;
#pragma unroll
        for (int a = 0; a < 4; ++a)
            row[a] = (PACKED ? 1 : 2) * plane + (Off)(T.axis_off[a] + (bad ? 0 : v[a])) * (Off)k_stride;
        const int ks = (SELECT && !bad) ? o.ksel[i] : 0;
        int r_acc = 0, xs[4] = {0, 0, 0, 0};
        // a first pass starts with the sample (every trial) and moves d up as its
        // keys allow; a repeated pass runs at one d
        bool adapt = SELECT && ks >= 1 && Kc > kAllK;
        int e = (SELECT && ks >= 1) ? 0 : e_lam;   // e = 0: every trial
        double lam_i = -INFINITY;
        for (int tries = 1;; ++tries) {
            float sigma = s_sig[e];
            int qn = 0, wk = 0;   // queued candidates, kept keys of this warp
            uint32_t a02 = 0u, a13 = 0u, waves = 0u;
            // a trial's S, its final counts (bytes P2, or xf) and whether the lane has one
            auto account = [&](float S, uint32_t P2, const int* xf, bool live) {
                if (!live) S = INFINITY;
                const uint32_t rej = (S < lambda_up) ? 1u : 0u;
                r_acc += (int)rej;
                if (PACKED) {
                    a02 += (P2 & 0x00FF00FFu) * rej;
                    a13 += __byte_perm(P2, 0u, 0x4341u) * rej;
                    if ((++waves & 127u) == 0u) {   // 16-bit halves: 128 x 255 < 2^16
                        xs[0] += (int)(a02 & 0xFFFFu);
                        xs[2] += (int)(a02 >> 16);
                        xs[1] += (int)(a13 & 0xFFFFu);
                        xs[3] += (int)(a13 >> 16);
                        a02 = a13 = 0u;
                    }
                } else {
#pragma unroll
                    for (int a = 0; a < 4; ++a) xs[a] += (int)rej * xf[a];
                }
                if (SELECT) {
                    const bool keep = S < sigma;
                    const unsigned kept = __ballot_sync(0xffffffffu, keep);
                    if (ks >= 1) {
                        if (keep) {
                            kbuf[wk + __popc(kept & below)] = __float_as_uint(S);
                            atomicAdd(&hist[key_bin(__float_as_uint(S))], 1u);
                        }
                        wk += __popc(kept);
                    }
                }
            };
            // step -1 of a first pass: the sample, spread over the warps; then sixteen
            // consecutive trials per thread and step from k0 on.  Bit 8 j + q of a
            // thread's candidate word is trial 4 q + j.
            constexpr int SW = kSample / NW;   // sample trials of a warp, a multiple of 16
            const int k0 = adapt ? kSample : 0;
            int st = adapt ? -1 : 0;
            for (;; ++st) {
                if (st >= 0 && k0 + st * (TT * 16) >= Kc) break;   // group-uniform
                // first trial of the warp at the start of the queue's block of 64 steps
                const int kb = st < 0 ? warp * SW : k0 + (st & ~63) * (TT * 16) + warp * 512;
                const int stq = st < 0 ? 0 : st & 63;
                const int kw = kb + stq * (TT * 16) + lane * 16;
                const int kend = st < 0 ? (warp + 1) * SW : Kc;
                uint32_t m = 0u;
                if (kw < kend) {
                    if (e == 0) {
                        m = 0x0F0F0F0Fu;
                    } else {
                        const uint32_t zc = 0x80808080u - (uint32_t)(dlo + e) * 0x01010101u;
                        const uint4 c = *reinterpret_cast<const uint4*>(cnt + (Off)(row[0] + (Off)kw));
                        const uint32_t z[4] = {zc - c.x, zc - c.y, zc - c.z, zc - c.w};
                        uint32_t t[4] = {0u, 0u, 0u, 0u};
#pragma unroll
                        for (int a = 1; a < 4; ++a)
                            if ((mask >> (a - 1)) & 1u) {
                                const uint4 x = *reinterpret_cast<const uint4*>(cnt + (Off)(row[a] + (Off)kw));
                                t[0] |= x.x + z[0];
                                t[1] |= x.y + z[1];
                                t[2] |= x.z + z[2];
                                t[3] |= x.w + z[3];
                            }
                        m = ((t[0] >> 7) & 0x01010101u) | ((t[1] >> 6) & 0x02020202u) | ((t[2] >> 5) & 0x04040404u) |
                            ((t[3] >> 4) & 0x08080808u);
                    }
                    if (kw + 16 > kend) m &= trials_below(kend - kw);   // trials at or past K
                }
                int nm = __popc(m), incl = nm;
#pragma unroll
                for (int off = 1; off < 32; off <<= 1) {
                    const int y = __shfl_up_sync(0xffffffffu, incl, off);
                    if (lane >= off) incl += y;
                }
                int total = __shfl_sync(0xffffffffu, incl, 31);
                if (total > kDense) {   // most of the warp's trials: all of them, from whole count words
                    const int k0w = kw - lane * 16;
#pragma unroll 1
                    for (int k4 = k0w + lane * 4; k4 - lane * 4 < min(k0w + 512, kend); k4 += 128) {
                        const Off at = (Off)min(k4, (Kc - 1) & ~3);   // (its four lie in the row)
                        uint32_t wf[4], wi[PACKED ? 4 : 8];
#pragma unroll
                        for (int a = 0; a < 4; ++a) {
                            wf[a] = __ldg(reinterpret_cast<const uint32_t*>(cnt + (Off)(row[a] + at)));
                            wi[a] = __ldg(reinterpret_cast<const uint32_t*>(cnt + (Off)(row[a] + at - plane)));
                            if constexpr (!PACKED)
                                wi[4 + a] =
                                    __ldg(reinterpret_cast<const uint32_t*>(cnt + (Off)(row[a] + at - 2 * plane)));
                        }
                        if constexpr (PACKED) {
                            uint32_t E[4], F[4];
                            transpose4(wi, E);
                            transpose4(wf, F);
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                const uint32_t P0 = (E[j] >> 4) & 0x0F0F0F0Fu, P1 = P0 + (E[j] & 0x0F0F0F0Fu);
                                const uint32_t P2 = (uint32_t)s_inv[F[j] & 0x7Fu] |
                                                    (uint32_t)s_inv[(F[j] >> 8) & 0x7Fu] << 8 |
                                                    (uint32_t)s_inv[(F[j] >> 16) & 0x7Fu] << 16 |
                                                    (uint32_t)s_inv[(F[j] >> 24) & 0x7Fu] << 24;
                                account(design_stat_packed(L, Q, smem, D2s, F4, s_tri, s_perm, P0, P1, P2, mask), P2,
                                        nullptr, k4 + j < kend);
                            }
                        } else {
#pragma unroll 1
                            for (int j = 0; j < 4; ++j) {
                                int xl[3][4];
#pragma unroll
                                for (int a = 0; a < 4; ++a) {
                                    xl[0][a] = (int)((wi[4 + a] >> (8 * j)) & 0xFFu);
                                    xl[1][a] = (int)((wi[a] >> (8 * j)) & 0xFFu);
                                    xl[2][a] = (int)((wf[a] >> (8 * j)) & 0xFFu);
                                }
                                const NodeConst C{};   // not read by the tabulated form
                                account(design_stat<true>(L, D1g, D2, F4, C, 0.0f, xl, mask), 0u, xl[2], k4 + j < kend);
                            }
                        }
                    }
                    m = 0u;
                    nm = incl = total = 0;
                }
                const bool flush = (st & 63) == 63 || k0 + (st + 1) * (TT * 16) >= Kc;
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
                        const Off k = (Off)(kb + (ev >> 10) * (TT * 16) + ((ev & 0x3E0) >> 1) + ((ev & 7) << 2) +
                                            ((ev >> 3) & 3));
                        float S;
                        uint32_t P2 = 0u;
                        int xf[4];
                        if constexpr (PACKED) {
                            uint32_t E = 0u;
#pragma unroll
                            for (int a = 0; a < 4; ++a) {
                                P2 |= (uint32_t)s_inv[__ldg(cnt + (Off)(row[a] + k))] << (8 * a);
                                E |= (uint32_t)__ldg(cnt + (Off)(row[a] + k - plane)) << (8 * a);
                            }
                            const uint32_t P0 = (E >> 4) & 0x0F0F0F0Fu, P1 = P0 + (E & 0x0F0F0F0Fu);
                            S = design_stat_packed(L, Q, smem, D2s, F4, s_tri, s_perm, P0, P1, P2, mask);
                        } else {
                            int xl[3][4];
#pragma unroll
                            for (int l = 0; l < 3; ++l)
#pragma unroll
                                for (int a = 0; a < 4; ++a)
                                    xl[l][a] = (int)__ldg(cnt + (Off)(row[a] + k - (Off)(2 - l) * plane));
#pragma unroll
                            for (int a = 0; a < 4; ++a) xf[a] = xl[2][a];
                            const NodeConst C{};   // not read by the tabulated form
                            S = design_stat<true>(L, D1g, D2, F4, C, 0.0f, xl, mask);
                        }
                        account(S, P2, xf, lane < n);
                        __syncwarp();   // the queue's entries read before the next round writes
                    }
                } while (done < total);
                // after the sample and after 1, 2, 4, 8, ... steps of a first pass: d for
                // the trials to come
                if (SELECT && adapt && ((st + 1) & st) == 0) {
                    tile_sync<TT, G>(g);
                    if (warp == 0) {
                        // the highest d such that the keys below sigma(d) so far, scaled to
                        // all K trials and less 2.5 standard deviations, reach k_i
                        const float seen = (float)min(k0 + (st + 1) * (TT * 16), Kc);
                        const float f = ((float)Kc - seen) / seen, v = 2.5f * sqrtf(f * (1.0f + f));
                        const float r = (v + sqrtf(v * v + 4.0f * (1.0f + f) * (float)ks)) / (2.0f * (1.0f + f));
                        int before = 0;
                        const int B = warp_pick256<false>(hist, (int)ceilf(r * r) + 1, lane, &before);
                        int top = e;
                        if (B >= 0)
                            for (int j = lane; j <= e_lam; j += 32)
                                if (s_sbin[j] > B) top = max(top, j);
                        top = __reduce_max_sync(0xffffffffu, top);
                        if (lane == 0) s_pick[g] = top;
                    }
                    tile_sync<TT, G>(g);
                    e = s_pick[g];
                    sigma = s_sig[e];
                }
            }
            if (PACKED) {
                xs[0] += (int)(a02 & 0xFFFFu);
                xs[2] += (int)(a02 >> 16);
                xs[1] += (int)(a13 & 0xFFFFu);
                xs[3] += (int)(a13 >> 16);
            }
            if (!SELECT || ks < 1) break;
            if (lane == 0) s_nk[g][warp] = wk;
            tile_sync<TT, G>(g);
            // the ks-th smallest key: its bin, then its rank among the bin's keys
            int nk = 0;
#pragma unroll
            for (int w2 = 0; w2 < NW; ++w2) nk += s_nk[g][w2];
            bool found = nk >= ks;
            if (found) {
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
#pragma unroll 4
                for (int k = lane; k < wk; k += 32) {   // each warp its own keys
                    const uint32_t key = kbuf[k];
                    if (key_bin(key) == B) {
                        const int at = atomicAdd(&s_nlist[g], 1);
                        if (at < kList) list[at] = key;
                    }
                }
                tile_sync<TT, G>(g);
                const int nl = s_nlist[g];
                if (nl <= kList) {
                    for (int j = lt; j < nl; j += TT) {
                        const uint32_t key = list[j];
                        int rank = 0;
                        for (int q = 0; q < nl; ++q) {
                            const uint32_t u = list[q];
                            rank += (u < key || (u == key && q < j)) ? 1 : 0;
                        }
                        if (rank == kr - 1) s_res[g] = key;
                    }
                    tile_sync<TT, G>(g);
                } else {   // radix select over the bin's keys: digits of 8, 8, 8 and 7 bits (S >= 0)
                    uint32_t prefix = 0u, pmask = 0u;
                    int kq = kr;
                    for (int pass = 0; pass < 4; ++pass) {
                        const int sh = pass < 3 ? 23 - 8 * pass : 0;
                        const uint32_t dm = pass < 3 ? 0xFFu : 0x7Fu;
#pragma unroll 4
                        for (int k = lane; k < wk; k += 32) {
                            const uint32_t key = kbuf[k];
                            if (key_bin(key) == B && (key & pmask) == prefix) atomicAdd(&hist[(key >> sh) & dm], 1u);
                        }
                        tile_sync<TT, G>(g);
                        if (warp == 0) {
                            int before = 0;
                            const int digit = warp_pick256<true>(hist, kq, lane, &before);
                            if (lane == 0) {
                                s_pick[g] = digit;
                                s_before[g] = before;
                            }
                        }
                        tile_sync<TT, G>(g);
                        prefix |= (uint32_t)s_pick[g] << sh;
                        pmask |= dm << sh;
                        kq -= s_before[g];
                    }
                    if (lt == 0) s_res[g] = prefix;
                    tile_sync<TT, G>(g);
                }
                lam_i = (double)__uint_as_float(s_res[g]);
                // exact unless it lies above the bound of the trials left out
                found = lam_i <= (double)sigma;
            } else {
                for (int b = lt; b < 256; b += TT) hist[b] = 0u;
                lam_i = INFINITY;   // with every trial evaluated, the k_i-th smallest S is +inf
            }
            if (found || e == 0) break;
            // too few keys below sigma: the whole pass again at a lower d
            e = tries < 4 ? max(e - 2 * tries, 0) : 0;
            adapt = false;
            r_acc = 0;
#pragma unroll
            for (int a = 0; a < 4; ++a) xs[a] = 0;
            tile_sync<TT, G>(g);   // every thread has read the counts
            if (lt == 0) s_nlist[g] = 0;
            tile_sync<TT, G>(g);
        }
        r_acc = warp_sum_i(r_acc);
#pragma unroll
        for (int a = 0; a < 4; ++a) xs[a] = warp_sum_i(xs[a]);
        if (lane == 0) {
            s_red[g][0][warp] = r_acc;
            for (int a = 0; a < 4; ++a) s_red[g][1 + a][warp] = xs[a];
        }
        tile_sync<TT, G>(g);
        if (lt == 0) {
            if (bad) atomicOr(err, CSE_ERR_BAD_K);
            int64_t Rt = 0, X[4] = {0, 0, 0, 0};
            for (int w2 = 0; w2 < NW; ++w2) {
                Rt += s_red[g][0][w2];
                for (int a = 0; a < 4; ++a) X[a] += s_red[g][1 + a][w2];
            }
            if (o.R) o.R[i] = Rt;
            if (o.cp_key)   // the tile's (K, R) in the Clopper-Pearson memo, as k_cp_mark would
                o.cp_slot[i] = cp_memo_insert(((unsigned long long)(uint32_t)K << 32) | (uint32_t)Rt, o.cp_key,
                                              o.cp_cap, o.cp_list, o.cp_nkeys);
            for (int a = 0; a < 4; ++a) {
                if (o.Xrej) o.Xrej[i * 4 + a] = X[a];
                if (o.score) {
                    const double sg = bad ? NAN : o.sig[T.axis_off[a] + v[a]];
                    o.score[i * 4 + a] = (double)X[a] - (double)L.n3 * sg * (double)Rt;
                }
            }
            if (SELECT && o.lam_tile) o.lam_tile[i] = lam_i;
            if (SELECT) s_min[g] = min(s_min[g], order_key(lam_i));
        }
        tile_sync<TT, G>(g);
    }
    __syncthreads();   // every group done before the queue is reset
    unsigned long long mine = ~0ull;
    if (tid == 0)
        for (int q = 0; q < G; ++q) mine = min(mine, s_min[q]);
    queue_reset_min(counter, o.min_key, mine, SELECT ? o.min_out : nullptr, (int)gridDim.x);
}

// The direct form (plain path, CSE_OPT_BAYES_DIRECT, and designs whose tables
// would not fit): the posterior evaluated for every trial, one tile per block.
template <bool SELECT>
__global__ void __launch_bounds__(BT, 5)
    k_sim_bayes4_direct(TileArgs T, Looks L, float drop, const uint8_t* __restrict__ cnt, int32_t NA,
                        int32_t k_stride, int32_t K_tiles, float lambda_up, SimOut o, uint32_t* __restrict__ keys,
                        int32_t* __restrict__ counter, int32_t* __restrict__ err)
{
    constexpr int NTH = BT;
    constexpr int NW = BWARP;
    __shared__ uint32_t hist[2048];
    __shared__ int s_tile, s_scan[NW], s_res[2];
    __shared__ int s_red[5][NW];
    __shared__ unsigned long long s_min;   // order key of the least lambda_i of this CTA's tiles
    if (threadIdx.x == 0) s_min = ~0ull;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const NodeConst C = node_const();
    uint32_t* kbuf = keys + (int64_t)blockIdx.x * k_stride;
    for (;;) {
        if (tid == 0) s_tile = atomicAdd(counter, 1);
        if (SELECT)
            for (int b = tid; b < 2048; b += NTH) hist[b] = 0u;
        __syncthreads();
        const int64_t i = s_tile;
        if (i >= T.n_tiles) break;
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
        // row index of the count table for (analysis l, arm a)
        int row[3][4];
#pragma unroll
        for (int l = 0; l < 3; ++l)
#pragma unroll
            for (int a = 0; a < 4; ++a) row[l][a] = l * NA + T.axis_off[a] + (bad ? 0 : v[a]);
        int r_acc = 0, xs[4] = {0, 0, 0, 0};
        // four consecutive sims per thread and step: one 32-bit load per table row
        auto load_rows = [&](int k4, uint32_t w[3][4]) {
#pragma unroll
            for (int l = 0; l < 3; ++l)
#pragma unroll
                for (int a = 0; a < 4; ++a)
                    w[l][a] = __ldg(reinterpret_cast<const uint32_t*>(cnt + (int64_t)row[l][a] * k_stride + k4));
        };
        for (int k4 = tid * 4; k4 < Kc; k4 += NTH * 4) {
            uint32_t w[3][4], kq[4];
            load_rows(k4, w);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                float S = INFINITY;
                if (k4 + j < Kc) {
                    int xl[3][4];
#pragma unroll
                    for (int l = 0; l < 3; ++l)
#pragma unroll
                        for (int a = 0; a < 4; ++a) xl[l][a] = (w[l][a] >> (8 * j)) & 0xFF;
                    S = design_stat<false>(L, nullptr, nullptr, nullptr, C, drop, xl, mask);
                    const int rej = (S < lambda_up) ? 1 : 0;
                    r_acc += rej;
#pragma unroll
                    for (int a = 0; a < 4; ++a) xs[a] += rej * xl[2][a];   // integer multiply-add
                    if (SELECT) atomicAdd(&hist[__float_as_uint(S) >> 21], 1u);
                }
                kq[j] = __float_as_uint(S);
            }
            if (SELECT) *reinterpret_cast<uint4*>(kbuf + k4) = make_uint4(kq[0], kq[1], kq[2], kq[3]);
        }
        r_acc = warp_sum_i(r_acc);
#pragma unroll
        for (int a = 0; a < 4; ++a) xs[a] = warp_sum_i(xs[a]);
        if (lane == 0) {
            s_red[0][warp] = r_acc;
            for (int a = 0; a < 4; ++a) s_red[1 + a][warp] = xs[a];
        }
        __syncthreads();
        double lam_i = -INFINITY;
        if (SELECT) {
            const int ks = bad ? 0 : o.ksel[i];
            if (ks >= 1) {
                // three-digit radix select (11, 11, 10 bits) over the tile's keys
                int b1, before1, b2, before2, b3, before3;
                find_kth<NTH>(hist, 2048, ks, s_scan, s_res, &b1, &before1);
                for (int b = tid; b < 2048; b += NTH) hist[b] = 0u;
                __syncthreads();
                for (int k = tid; k < Kc; k += NTH) {
                    const uint32_t key = kbuf[k];
                    if ((int)(key >> 21) == b1) atomicAdd(&hist[(key >> 10) & 0x7FF], 1u);
                }
                __syncthreads();
                find_kth<NTH>(hist, 2048, ks - before1, s_scan, s_res, &b2, &before2);
                for (int b = tid; b < 1024; b += NTH) hist[b] = 0u;
                __syncthreads();
                const uint32_t pre = ((uint32_t)b1 << 11) | (uint32_t)b2;
                for (int k = tid; k < Kc; k += NTH) {
                    const uint32_t key = kbuf[k];
                    if ((key >> 10) == pre) atomicAdd(&hist[key & 0x3FF], 1u);
                }
                __syncthreads();
                find_kth<NTH>(hist, 1024, ks - before1 - before2, s_scan, s_res, &b3, &before3);
                lam_i = (double)__uint_as_float((pre << 10) | (uint32_t)b3);
            }
        }
        if (tid == 0) {
            if (bad) atomicOr(err, CSE_ERR_BAD_K);
            int64_t Rt = 0, X[4] = {0, 0, 0, 0};
            for (int w2 = 0; w2 < NW; ++w2) {
                Rt += s_red[0][w2];
                for (int a = 0; a < 4; ++a) X[a] += s_red[1 + a][w2];
            }
            if (o.R) o.R[i] = Rt;
            if (o.cp_key)   // the tile's (K, R) in the Clopper-Pearson memo, as k_cp_mark would
                o.cp_slot[i] = cp_memo_insert(((unsigned long long)(uint32_t)K << 32) | (uint32_t)Rt, o.cp_key,
                                              o.cp_cap, o.cp_list, o.cp_nkeys);
            for (int a = 0; a < 4; ++a) {
                if (o.Xrej) o.Xrej[i * 4 + a] = X[a];
                if (o.score) {
                    const double sg = bad ? NAN : o.sig[T.axis_off[a] + v[a]];
                    o.score[i * 4 + a] = (double)X[a] - (double)L.n3 * sg * (double)Rt;
                }
            }
            if (SELECT && o.lam_tile) o.lam_tile[i] = lam_i;
            if (SELECT) s_min = min(s_min, order_key(lam_i));
        }
        __syncthreads();
    }
    queue_reset_min(counter, o.min_key, s_min, SELECT ? o.min_out : nullptr, (int)gridDim.x);
}

template <bool TABLES>
__global__ void k_emit_bayes4(TileArgs T, Looks L, float drop, const uint8_t* __restrict__ cnt, int32_t NA,
                              int32_t k_stride, int32_t K_tiles, const uint8_t* __restrict__ D1,
                              const uint8_t* __restrict__ D2, const float4* __restrict__ F4,
                              const int64_t* __restrict__ off, float* __restrict__ S_out, int32_t* __restrict__ err,
                              bool nib, const uint8_t* __restrict__ score)
{
    __shared__ uint8_t inv[128];
    if (nib)
        for (int x = threadIdx.x; x <= L.n3; x += blockDim.x) inv[score[x]] = (uint8_t)x;
    __syncthreads();
    NodeConst C;
    if (!TABLES) C = node_const();
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
            int xl[3][4];
            for (int a = 0; a < 4; ++a) {
                const uint8_t* p = cnt + (int64_t)(T.axis_off[a] + v[a]) * k_stride + k;
                const int64_t plane = (int64_t)NA * k_stride;
                if (nib) {   // the packed form's two planes
                    xl[0][a] = p[0] >> 4;
                    xl[1][a] = xl[0][a] + (p[0] & 15);
                    xl[2][a] = inv[p[plane]];
                } else {
                    for (int l = 0; l < 3; ++l) xl[l][a] = p[l * plane];
                }
            }
            S_out[off[i] + k] = design_stat<TABLES>(L, D1, D2, F4, C, drop, xl, mask);
        }
    }
}

Looks make_looks(const DesignArgs& D)
{
    Looks L;
    L.n1 = D.look_n[0];
    L.n2 = D.look_n[1];
    L.n3 = D.look_n[2];
    L.S2 = (L.n1 + 1) + (L.n2 + 1);
    L.S3 = L.S2 + (L.n3 + 1);
    L.NP = L.S3 * (L.S3 + 1) / 2;
    L.NT = L.S3 * (L.S3 + 1) * (L.S3 + 2) / 6;
    return L;
}

int64_t b4_round16(int64_t n)
{
    return (n + 15) / 16 * 16;
}

int32_t b4_nt2(const Looks& L)
{
    return L.S2 * (L.S2 + 1) * (L.S2 + 2) / 6;
}

// bytes of the sorted second-analysis table (ten entries a word), padded to 16
int64_t b4_d2s_bytes(const Looks& L)
{
    return b4_round16(4 * (((int64_t)(L.n2 + 1) * b4_nt2(L) + 9) / 10));
}

// bytes of the first-analysis table in the packed form's shared memory (two
// entries a byte), padded to 16
int64_t b4_d1_bytes(const Looks& L)
{
    const int64_t n = (int64_t)(L.n1 + 1) * (L.n1 + 1) * (L.n1 + 1) * (L.n1 + 1);
    return b4_round16((n + 1) / 2);
}

constexpr int kSmemLimit = 96 * 1024;

template <typename Kern>
int b4_grid(cse_ctx* c, Kern kern, int nt, size_t smem, int64_t blocks, int64_t* grid)
{
    // one limit for every design (the tables take at most 70 KB): it belongs to the kernel, and
    // another thread may be launching a design with larger tables
    if (smem > 0 &&
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit) != cudaSuccess) {
        cudaGetLastError();
        return CSE_UNSUPPORTED_DESIGN;
    }
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, nt, smem) != cudaSuccess || per_sm < 1) {
        cudaGetLastError();
        return CSE_CUDA_ERROR;
    }
    *grid = (int64_t)per_sm * c->num_sms;
    if (*grid > blocks) *grid = blocks;
    return CSE_OK;
}

// The range of differences d the byte test holds for scores 0 .. top without a
// carry across bytes: 0 <= 128 - d - top and 128 - d + top <= 255 (d = dlo stands
// for every trial).
void b4_diff_range(int32_t top, int32_t* dlo, int32_t* nd)
{
    const int lo = top - 127 > -top ? top - 127 : -top;
    const int hi = 128 - top < top + 1 ? 128 - top : top + 1;
    *dlo = lo;
    *nd = hi > lo ? hi - lo + 1 : 1;
}

template <bool SEL, bool PACKED, int G, typename Off>
int launch_b4(cse_ctx* c, const TileArgs& T, int32_t NA, int32_t k_stride, int32_t K_tiles, double lambda,
              const SimOut& o, cudaStream_t s)
{
    auto kern = k_sim_bayes4<SEL, PACKED, G, Off>;
    constexpr int NT = b4_threads<PACKED>();
    const Looks L = make_looks(c->D);
    PackedConst Q{};
    if (PACKED) {
        const uint32_t m = (uint32_t)(L.n1 + 1), s2 = (uint32_t)L.S2;
        Q.w1hi = m | (1u << 8);
        Q.w1lo = (m << 16) | (1u << 24);
        Q.m1sq = m * m;
        Q.off1 = m * 0x01010100u;
        Q.off2 = s2 * 0x01010100u;
        Q.nt2 = b4_nt2(L);
    }
    const int32_t d1_bytes = PACKED ? (int32_t)b4_d1_bytes(L) : 0;
    const int32_t d2s_bytes = PACKED ? (int32_t)b4_d2s_bytes(L) : 0;
    const size_t smem = (size_t)d1_bytes + (size_t)d2s_bytes + (size_t)G * 256 * 4 + (SEL ? (size_t)G * kList * 4 : 0) +
                        (size_t)(NT / 32) * kQueue * 2;
    int64_t grid = 0;
    int st = b4_grid(c, kern, NT, smem, (T.n_tiles + G - 1) / G, &grid);
    if (st != CSE_OK) return st;
    // a warp's keys: its share of the sample and its 512 trials of every step
    constexpr int TT = b4_group<PACKED, G>(), NW = TT / 32;
    const int32_t key_seg = kSample / NW + (K_tiles + TT * 16 - 1) / (TT * 16) * 512;
    if (SEL && (st = cse_reserve_keys(c, sizeof(uint32_t) * G * NW * (size_t)key_seg, &grid, s)) != CSE_OK) return st;
    int32_t dlo = 0, nd = 1;
    b4_diff_range(c->bt_top, &dlo, &nd);
    if (SEL && o.min_out) c->min_folded = true;
    if (o.cp_key) c->cp_marked = true;
    cse_prof_begin(c, KID_SIM_BAYES4, s);
    kern<<<(unsigned)grid, NT, smem, s>>>(T, L, c->cnt, NA, k_stride, K_tiles, c->bt_d1, c->bt_d2, c->bt_f4,
                                          c->bt_score, c->bt_dmin, c->bt_top, dlo, nd, lambda_float_up(lambda),
                                          o.R || o.Xrej || o.score || o.cp_key, o, c->keys, key_seg, c->counter, c->err,
                                          Q, c->bt_d2s, d1_bytes, d2s_bytes);
    cse_prof_end(c, s);
    c->launches += 1;
    return cudaGetLastError() == cudaSuccess ? CSE_OK : CSE_CUDA_ERROR;
}

template <bool SEL>
int launch_b4_direct(cse_ctx* c, const TileArgs& T, int32_t NA, int32_t k_stride, int32_t K_tiles, double lambda,
                     const SimOut& o, cudaStream_t s)
{
    auto kern = k_sim_bayes4_direct<SEL>;
    int64_t grid = 0;
    int st = b4_grid(c, kern, BT, 0, T.n_tiles, &grid);
    if (st != CSE_OK) return st;
    if (SEL && (st = cse_reserve_keys(c, sizeof(uint32_t) * (size_t)k_stride, &grid, s)) != CSE_OK) return st;
    if (SEL && o.min_out) c->min_folded = true;
    if (o.cp_key) c->cp_marked = true;
    cse_prof_begin(c, KID_SIM_BAYES4, s);
    kern<<<(unsigned)grid, BT, 0, s>>>(T, make_looks(c->D), (float)c->D.drop, c->cnt, NA, k_stride, K_tiles,
                                       lambda_float_up(lambda), o, c->keys, c->counter, c->err);
    cse_prof_end(c, s);
    c->launches += 1;
    return cudaGetLastError() == cudaSuccess ? CSE_OK : CSE_CUDA_ERROR;
}

// Groups of a block: four tiles a block (two in the byte form) once every group
// of the resident blocks has a tile, one tile a block below that.
template <bool SEL, bool PACKED>
int launch_b4_tables(cse_ctx* c, const TileArgs& T, int32_t NA, int32_t k_stride, int32_t K_tiles, double lambda,
                     const SimOut& o, cudaStream_t s)
{
    constexpr int G = PACKED ? 4 : 2;
    // 32-bit offsets into the count table while it is smaller than 4 GB
    if ((uint64_t)(PACKED ? 2 : 3) * (uint64_t)NA * (uint64_t)k_stride > 0xFFFFFFFFull)
        return launch_b4<SEL, PACKED, 1, uint64_t>(c, T, NA, k_stride, K_tiles, lambda, o, s);
    // (a group's keys are K words: one tile a block for the largest K keeps the keys of a
    // launch at 1.3 GB, in the byte form 2.6 GB)
    if (T.n_tiles >= (int64_t)c->num_sms * 2 * G && K_tiles <= (1 << 17))
        return launch_b4<SEL, PACKED, G, uint32_t>(c, T, NA, k_stride, K_tiles, lambda, o, s);
    return launch_b4<SEL, PACKED, 1, uint32_t>(c, T, NA, k_stride, K_tiles, lambda, o, s);
}

}  // namespace

int cse_bayes4_setup(cse_ctx* c, cudaStream_t s)
{
    const Looks L = make_looks(c->D);
    const int64_t n1 = (int64_t)(L.n1 + 1) * (L.n1 + 1) * (L.n1 + 1) * (L.n1 + 1);
    const int64_t n2 = (int64_t)(L.n2 + 1) * L.S2 * L.S2 * L.S2;
    const int64_t n3 = (int64_t)(L.n3 + 1) * L.NT;   // float4 entries
    c->bt_tables = (n1 + n2 + 4 * n3) <= CSE_BAYES_TABLE_MAX;
    if (!c->bt_tables) return CSE_OK;   // direct evaluation per simulation
    if (cudaMalloc(&c->bt_d1, (size_t)n1) != cudaSuccess || cudaMalloc(&c->bt_d2, (size_t)n2) != cudaSuccess ||
        cudaMalloc(&c->bt_f4, (size_t)n3 * sizeof(float4)) != cudaSuccess) {
        cudaGetLastError();
        return CSE_OOM;
    }
    const float drop = (float)c->D.drop;
    cse_prof_begin(c, KID_BAYES_TABLE, s);
    k_table_d1<<<(unsigned)((n1 + 255) / 256), 256, 0, s>>>(c->bt_d1, L, drop);
    k_table_d2<<<(unsigned)((n2 + 255) / 256), 256, 0, s>>>(c->bt_d2, L, drop);
    // the packed per-trial form: every final-look code in seven bits, second-look
    // codes in six, both interim segments' counts in a nibble, and both
    // shared-memory tables within 70 KB (2 CTAs per SM)
    const int64_t d2s = b4_d2s_bytes(L);
    c->bt_packed = L.S3 <= 128 && L.S2 <= 64 && L.n1 <= 15 && L.n2 - L.n1 <= 15 && b4_d1_bytes(L) + d2s <= 70 * 1024;
    if (c->bt_packed) {
        if (cudaMalloc(&c->bt_d2s, (size_t)d2s) != cudaSuccess) {
            cudaGetLastError();
            return CSE_OOM;
        }
        const int64_t nw = ((int64_t)(L.n2 + 1) * b4_nt2(L) + 9) / 10;
        if (cudaMemsetAsync(c->bt_d2s, 0, (size_t)d2s, s) != cudaSuccess) {
            cudaGetLastError();
            return CSE_CUDA_ERROR;
        }
        k_table_d2s<<<(unsigned)((nw + 255) / 256), 256, 0, s>>>(c->bt_d2s, c->bt_d2, L, b4_nt2(L));
        c->launches += 1;
    }
    k_table_f4<<<(unsigned)((n3 + 255) / 256), 256, 0, s>>>(c->bt_f4, L);
    // scores of the final counts: in the packed form the angular transform (near
    // constant variance, so one difference cuts at about the same S for every
    // control count) scaled to 0 .. kScoreTop where that keeps them distinct; the
    // counts themselves otherwise
    uint8_t score[CSE_MAX_NMAX + 1];
    const double lo = asin(sqrt(1.0 / (L.n3 + 2.0))), hi = asin(sqrt((L.n3 + 1.0) / (L.n3 + 2.0)));
    bool distinct = c->bt_packed;
    for (int x = 0; x <= L.n3; ++x) {
        score[x] = (uint8_t)lround(kScoreTop * (asin(sqrt((x + 1.0) / (L.n3 + 2.0))) - lo) / (hi - lo));
        distinct &= x == 0 || score[x] > score[x - 1];
    }
    if (!distinct)
        for (int x = 0; x <= L.n3; ++x) score[x] = (uint8_t)x;
    c->bt_top = score[L.n3];
    uint32_t none[2 * CSE_MAX_NMAX + 1];
    for (uint32_t& x : none) x = 0x7F800000u;
    if (cudaMalloc(&c->bt_dmin, sizeof(none)) != cudaSuccess ||
        cudaMalloc(&c->bt_score, sizeof(score)) != cudaSuccess) {
        cudaGetLastError();
        return CSE_OOM;
    }
    if (cudaMemcpyAsync(c->bt_dmin, none, sizeof(none), cudaMemcpyHostToDevice, s) != cudaSuccess ||
        cudaMemcpyAsync(c->bt_score, score, (size_t)L.n3 + 1, cudaMemcpyHostToDevice, s) != cudaSuccess) {
        cudaGetLastError();
        return CSE_CUDA_ERROR;
    }
    k_table_dmin<<<(unsigned)(4 * c->num_sms), 256, 0, s>>>(c->bt_f4, L, c->bt_score, c->bt_dmin);
    cse_prof_end(c, s);
    c->launches += 4;
    return cudaGetLastError() == cudaSuccess ? CSE_OK : CSE_CUDA_ERROR;
}

int cse_launch_emit_bayes4(cse_ctx* c, const TileArgs& T, int32_t NA, int32_t k_stride, int32_t K_tiles,
                           const int64_t* off, float* S_out, cudaStream_t s)
{
    const int64_t grid = T.n_tiles < 4096 ? T.n_tiles : 4096;
    const Looks L = make_looks(c->D);
    if (c->bt_tables && !c->bt_direct)
        k_emit_bayes4<true><<<(unsigned)grid, 256, 0, s>>>(T, L, (float)c->D.drop, c->cnt, NA, k_stride, K_tiles,
                                                           c->bt_d1, c->bt_d2, c->bt_f4, off, S_out, c->err,
                                                           cse_count_nibbles(c), c->bt_score);
    else
        k_emit_bayes4<false><<<(unsigned)grid, 256, 0, s>>>(T, L, (float)c->D.drop, c->cnt, NA, k_stride, K_tiles,
                                                            c->bt_d1, c->bt_d2, c->bt_f4, off, S_out, c->err,
                                                           cse_count_nibbles(c), c->bt_score);
    c->launches += 1;
    return cudaGetLastError() == cudaSuccess ? CSE_OK : CSE_CUDA_ERROR;
}

int cse_launch_sim_bayes4(cse_ctx* c, const TileArgs& T, int32_t NA, int32_t k_stride, int32_t K_tiles,
                          double lambda, const SimOut& o, cudaStream_t s)
{
    const bool sel = (o.lam_tile != nullptr && o.ksel != nullptr);
    if (c->bt_tables && !c->bt_direct) {
        if (c->bt_packed)
            return sel ? launch_b4_tables<true, true>(c, T, NA, k_stride, K_tiles, lambda, o, s)
                       : launch_b4_tables<false, true>(c, T, NA, k_stride, K_tiles, lambda, o, s);
        return sel ? launch_b4_tables<true, false>(c, T, NA, k_stride, K_tiles, lambda, o, s)
                   : launch_b4_tables<false, false>(c, T, NA, k_stride, K_tiles, lambda, o, s);
    }
    return sel ? launch_b4_direct<true>(c, T, NA, k_stride, K_tiles, lambda, o, s)
               : launch_b4_direct<false>(c, T, NA, k_stride, K_tiles, lambda, o, s);
}
