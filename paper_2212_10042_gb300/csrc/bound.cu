// bound.cu -- per-tile FP64 bound pass: Clopper-Pearson upper bound, the
// q-optimised tilewise Tilt-Bound, and the calibration target alpha'.
//
// Exponential-family Tilt-Bound (Eq. tilt-bound:exp-fam) for independent
// binomial arms on the logit scale, A(theta) = sum_a n log(1 + e^theta_a):
//   log U(theta0, v, q, a) = (1 - 1/q) log a + sum_a phi_a(q, v_a),
//   phi_a(q, v_a) = psi_a(q v_a)/q - psi_a(v_a),  psi_a(x) = n (sp(theta0_a + x) - sp(theta0_a)).
// A is a sum over arms, so the maximum of log U over the 2^d vertices of the
// box (Thm. 3) is the sum over arms of the larger of the two per-arm terms
// (v_a = +h_a or -h_a): the vertex search costs 2d softplus per q, not d 2^d.
// The optimum over q (Thm. 2: quasi-convex in q) is found by bisection in
// s = log q on the sign of the hand-written derivative
//   d/dq log U = log a / q^2 + sum_a [q v_a psi_a'(q v_a) - psi_a(q v_a)] / q^2.
// The inverted bound (Eq. tilt-bound-inv) uses the same per-arm terms:
//   log U^-1 = q/(q-1) [log alpha - sum_a max_v phi_a],
// maximised over q by bisection on the sign of its derivative.
#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>

#include "cse_internal.cuh"

namespace {

#define CSE_HD __host__ __device__

constexpr double SMAX = 40.0;   // search range s = log q in [0, 40]
constexpr int BISECT_F32 = 4;        // FP32 bisection steps on [0, SMAX] before the secant
constexpr int SECANT_F32 = 16;       // cap on FP32 secant (Illinois) steps
constexpr float SECANT_TOL = 1e-5f;  // FP32 stage ends when the bracket is this narrow ...
constexpr float SECANT_STEP = 5e-6f; // ... or when a secant step is this short
constexpr int kSplitWarps = 3;      // warps a sub-partition up to which the signs are split (split_signs)
constexpr int POLISH_IT = 80;   // cap on FP64 safeguarded-Newton steps

struct ArmGeom {
    double th, h, n, sp0, d1p, d1m;   // d1p/d1m = sp(th +/- h) - sp(th)
};

CSE_HD __forceinline__ double softplus(double x) { return fmax(x, 0.0) + log1p(exp(-fabs(x))); }

CSE_HD __forceinline__ void arm_init(ArmGeom& g, double th, double h, double n)
{
    g.th = th;
    g.h = h;
    g.n = n;
    g.sp0 = softplus(th);
    g.d1p = softplus(th + h) - g.sp0;
    g.d1m = softplus(th - h) - g.sp0;
}

// ---------------------------------------------------------------------------
// Per-arm terms.  phi_a(q, v) = n [sp(th + q v) - sp(th)] / q - n [sp(th + v) - sp(th)];
// Phi(q) = sum_a max over v = +-h_a of phi_a; derivatives follow the maximising
// branch (on a tie, the one with the larger first derivative: right derivatives).
// ---------------------------------------------------------------------------

// FP64 value and first two q-derivatives along the maximising branches.
template <int D>
CSE_HD void tilt_phi(const ArmGeom* G, double q, double* Phi, double* dPhi, double* d2Phi, double* kdist = nullptr)
{
    constexpr int d = D;
    double P = 0.0, dP = 0.0, d2P = 0.0, kd = INFINITY;
    const double iq = 1.0 / q;
#pragma unroll
    for (int a = 0; a < d; ++a) {
        double best = -INFINITY, bestd = 0.0, bestd2 = 0.0;
        double ph[2], dph[2];
#pragma unroll
        for (int sg = 0; sg < 2; ++sg) {
            const double v = sg ? -G[a].h : G[a].h;
            const double qv = q * v;
            const double x = G[a].th + qv;
            const double e = exp(-fabs(x));
            const double l1e = log1p(e);
            const double sp = fmax(x, 0.0) + l1e - G[a].sp0;
            const double r = e / (1.0 + e);           // sigmoid(-|x|)
            const double sig = (x >= 0.0) ? 1.0 - r : r;
            const double phi = G[a].n * (sp * iq - (sg ? G[a].d1m : G[a].d1p));
            // q psi'(q v)/n - psi(q v)/n = qv sigmoid(x) - sp(x) + sp(th), written
            // without the cancellation of the two O(qv) terms at large q
            const double hq = (x >= 0.0) ? (G[a].sp0 - G[a].th) - qv * r - l1e : qv * r - l1e + G[a].sp0;
            const double dphi = G[a].n * hq * iq * iq;
            ph[sg] = phi;
            dph[sg] = dphi;
            if (phi > best || (phi == best && dphi > bestd)) {
                best = phi;
                bestd = dphi;
                bestd2 = G[a].n * (v * v * sig * (1.0 - sig) * iq - 2.0 * hq * iq * iq * iq);
            }
        }
        P += best;
        dP += bestd;
        d2P += bestd2;
        // first-order distance in q to the crossing of this arm's two branches
        kd = fmin(kd, fabs(ph[0] - ph[1]) / (fabs(dph[0] - dph[1]) + 1e-300));
    }
    *Phi = P;
    *dPhi = dP;
    if (d2Phi) *d2Phi = d2P;
    if (kdist) *kdist = kd;
}

// lim_{q->inf} Phi(q) = sum_a max(n h_a - n d1p, -n d1m)
template <int D>
CSE_HD double tilt_phi_inf(const ArmGeom* G)
{
    constexpr int d = D;
    double P = 0.0;
    for (int a = 0; a < d; ++a) P += G[a].n * fmax(G[a].h - G[a].d1p, -G[a].d1m);
    return P;
}

// Objective of the q search in s = log q.  kind 0: Tilt-Bound, G(s) = g(e^s),
// g(q) = (1 - 1/q) log a + Phi(q), minimised.  kind 1: inverted bound, negated so
// that it is also minimised: G(s) = -M(e^s), M(q) = q/(q-1) (log alpha - Phi(q)).
// Returns dG/ds (and d2G/ds2, value when asked).
template <int D>
CSE_HD double obj_ds(const ArmGeom* G, int kind, double lc, double s, double* d2, double* val,
                     double* kdist_s = nullptr)
{
    const double q = exp(s);
    double P, dP, d2P, kd;
    tilt_phi<D>(G, q, &P, &dP, &d2P, &kd);
    if (kdist_s) *kdist_s = kd / q;
    double g1, g2, v;
    if (kind == 0) {
        v = (1.0 - 1.0 / q) * lc + P;
        g1 = lc / (q * q) + dP;
        g2 = -2.0 * lc / (q * q * q) + d2P;
    } else {
        const double qm = q - 1.0, B = lc - P;
        v = -(q / qm * B);
        g1 = -(-B / (qm * qm) - q / qm * dP);
        g2 = -(2.0 * B / (qm * qm * qm) + 2.0 * dP / (qm * qm) - q / qm * d2P);
    }
    if (val) *val = v;
    if (d2) *d2 = q * g1 + q * q * g2;
    return q * g1;
}

// Coordinates in which the FP32 secant interpolates G'(s) linearly.  With Phi
// linear in q (its first-order form for small q h), kind 0 has dG/dq = G'(s)/q
// affine in 1/q^2, and kind 1 has the sign function of LaneTilt::ds32 affine in
// (q - 1)^2: so y = G'(s) e^{-s} against t = e^{-2s} for kind 0, and y = that
// function against t = (e^s - 1)^2 for kind 1.  The secant then converges in a
// few steps.
CSE_HD __forceinline__ void secant_point(int kind, float s, float g, float* t, float* y)
{
    if (kind == 0) {
        const float e = expf(-s);
        *t = e * e;
        *y = g * e;
    } else {
        const float e = expm1f(s);
        *t = e * e;
        *y = g;
    }
}

CSE_HD __forceinline__ float secant_s(int kind, float t)
{
    return kind == 0 ? -0.5f * logf(t) : log1pf(sqrtf(t));
}

// Quotient for the FP32 search stages, which need ~1e-6: the device uses the
// two-instruction approximate division (2 ulp).
CSE_HD __forceinline__ float fdiv_fast(float x, float y)
{
#ifdef __CUDA_ARCH__
    return __fdividef(x, y);
#else
    return x / y;
#endif
}

// ---------------------------------------------------------------------------
// A tile's objective by a group of lanes.  An FP64 warp instruction takes the
// same pipe time (64 cycles) with any number of active lanes, and one thread a
// tile left the pipe half idle on the 256^2 grid (1.7 warps a sub-partition) and
// a 64-tile call waiting for one warp's chain of ~1,000 of them.  The arms' terms
// are independent, so each lane takes one arm (D lanes a tile) or, SPLIT, one arm
// and one sign of v (2 D lanes); shuffles form the maximum over the signs and the
// sum over the arms, and every lane of the group follows the same search.
// ---------------------------------------------------------------------------
template <int D, bool SPLIT>
struct LaneTilt {
    static constexpr int NL = SPLIT ? 2 * D : D;   // lanes a tile
    static constexpr int NS = SPLIT ? 1 : 2;       // signs a lane
    double th, h, n, sp0;
    double d1[NS];     // sp(th + v) - sp(th) of the lane's signs (v = +h, then -h)
    float thf, hf, nf, sig0, sp0f, d1f[NS];
    int sg;            // first sign of the lane
    unsigned mask;     // the group's lanes

    __device__ __forceinline__ double v(int k) const { return (sg + k) ? -h : h; }

    __device__ __forceinline__ void init_f32()
    {
        thf = (float)th;
        hf = (float)h;
        nf = (float)n;
        sig0 = fdiv_fast(1.0f, 1.0f + expf(-thf));
        sp0f = (float)sp0;
#pragma unroll
        for (int k = 0; k < NS; ++k) d1f[k] = (float)d1[k];
    }

    __device__ __forceinline__ void init(double theta, double half, double n_max)
    {
        th = theta;
        h = half;
        n = n_max;
        sp0 = softplus(th);
#pragma unroll
        for (int k = 0; k < NS; ++k) d1[k] = softplus(th + v(k)) - sp0;
        init_f32();
    }

    // the other sign's value when the signs are split
    template <typename T>
    __device__ __forceinline__ T other(T x) const
    {
        return __shfl_xor_sync(mask, x, 1, NL);
    }

    template <typename T>
    __device__ __forceinline__ T arms_sum(T x) const
    {
#pragma unroll
        for (int o = NL / 2; o >= (SPLIT ? 2 : 1); o >>= 1) x += __shfl_xor_sync(mask, x, o, NL);
        return x;
    }

    // FP32 Phi and its q-derivative.  The difference sp(th + x) - sp(th) =
    // log1p(sigmoid(th) expm1(x)) for small |x| (no cancellation), directly otherwise.
    __device__ __forceinline__ void phi32(float q, float* Phi, float* dPhi) const
    {
        const float iq = fdiv_fast(1.0f, q);
        float p[2], dp[2];
#pragma unroll
        for (int k = 0; k < NS; ++k) {
            const float x = q * ((sg + k) ? -hf : hf);
            const float y = thf + x;
            const float e = expf(-fabsf(y));
            const float l1e = log1pf(e);
            const float r = fdiv_fast(e, 1.0f + e);
            float Dd, hq;   // hq = x sigmoid(y) - Dd without cancellation at large |x|
            if (fabsf(x) < 0.5f) {
                Dd = log1pf(sig0 * expm1f(x));
                hq = x * ((y >= 0.f) ? 1.0f - r : r) - Dd;
            } else {
                Dd = fmaxf(y, 0.0f) + l1e - sp0f;
                hq = (y >= 0.f) ? (sp0f - thf) - x * r - l1e : x * r - l1e + sp0f;
            }
            p[k] = nf * (Dd * iq - d1f[k]);
            dp[k] = nf * hq * iq * iq;
        }
        if (SPLIT) {   // in the order +h, -h on both lanes
            const float po = other(p[0]), dpo = other(dp[0]);
            p[1] = sg ? p[0] : po;
            dp[1] = sg ? dp[0] : dpo;
            p[0] = sg ? po : p[0];
            dp[0] = sg ? dpo : dp[0];
        }
        const bool second = p[1] > p[0] || (p[1] == p[0] && dp[1] > dp[0]);
        *Phi = arms_sum(second ? p[1] : p[0]);
        *dPhi = arms_sum(second ? dp[1] : dp[0]);
    }

    // sign function of the search in FP32: q dg/dq (kind 0), or minus dM/dq without
    // its division by (q - 1)^2 (kind 1)
    __device__ __forceinline__ float ds32(int kind, float lc, float s) const
    {
        const float q = expf(s);
        float P, dP;
        phi32(q, &P, &dP);
        return kind == 0 ? fdiv_fast(lc, q) + q * dP : (lc - P) + q * (q - 1.0f) * dP;
    }

    // FP64 dG/ds, d2G/ds2, value and the first-order distance in s to the nearest
    // crossing of an arm's two branches (see tilt_phi and obj_ds)
    __device__ double ds64(int kind, double lc, double s, double* d2, double* val, double* kdist) const
    {
        const double q = exp(s), iq = 1.0 / q;
        double p[2], dp[2], d2p[2];
#pragma unroll
        for (int k = 0; k < NS; ++k) {
            const double vk = v(k), qv = q * vk, x = th + qv;
            const double e = exp(-fabs(x));
            const double l1e = log1p(e);
            const double sp = fmax(x, 0.0) + l1e - sp0;
            const double r = e / (1.0 + e);   // sigmoid(-|x|)
            const double hq = (x >= 0.0) ? (sp0 - th) - qv * r - l1e : qv * r - l1e + sp0;
            p[k] = n * (sp * iq - d1[k]);
            dp[k] = n * hq * iq * iq;
            d2p[k] = n * iq * (vk * vk * r * (1.0 - r) - 2.0 * hq * iq * iq);
        }
        if (SPLIT) {
            const double po = other(p[0]), dpo = other(dp[0]), d2po = other(d2p[0]);
            p[1] = sg ? p[0] : po;
            dp[1] = sg ? dp[0] : dpo;
            d2p[1] = sg ? d2p[0] : d2po;
            p[0] = sg ? po : p[0];
            dp[0] = sg ? dpo : dp[0];
            d2p[0] = sg ? d2po : d2p[0];
        }
        const bool second = p[1] > p[0] || (p[1] == p[0] && dp[1] > dp[0]);
        const double P = arms_sum(second ? p[1] : p[0]);
        const double dP = arms_sum(second ? dp[1] : dp[0]);
        const double d2P = arms_sum(second ? d2p[1] : d2p[0]);
        if (kdist) {   // FP32: it is compared with a step of 1e-5
            float kd = fdiv_fast((float)fabs(p[0] - p[1]), fmaxf((float)fabs(dp[0] - dp[1]), 1e-30f));
#pragma unroll
            for (int o = NL / 2; o >= (SPLIT ? 2 : 1); o >>= 1) kd = fminf(kd, __shfl_xor_sync(mask, kd, o, NL));
            *kdist = (double)(kd * (float)iq);
        }
        double g1, g2, w;
        if (kind == 0) {
            w = (1.0 - iq) * lc + P;
            g1 = lc * iq * iq + dP;
            g2 = -2.0 * lc * iq * iq * iq + d2P;
        } else {
            const double iqm = 1.0 / (q - 1.0), t = q * iqm, B = lc - P;
            w = -(t * B);
            g1 = B * iqm * iqm + t * dP;
            g2 = -(2.0 * iqm * iqm * (B * iqm + dP) - t * d2P);
        }
        if (val) *val = w;
        if (d2) *d2 = q * g1 + q * q * g2;
        return q * g1;
    }

    // lim_{q->inf} Phi(q) = sum_a max(n h_a - n d1p, -n d1m)
    __device__ double phi_inf() const
    {
        double m = (sg == 0) ? h - d1[0] : -d1[0];
        if (SPLIT) m = fmax(m, other(m));
        else m = fmax(m, -d1[NS - 1]);
        return arms_sum(n * m);
    }
};

// Minimiser of the quasi-convex G over s in [0, SMAX].  FP32 stage: the sign of
// G' at s = 0, a few bisection steps, then a bracketing secant (Illinois: the
// stale end's value is halved when the same end moves twice running) in the
// coordinates of secant_point, down to ~1e-5 in s.  FP64 stage: safeguarded
// Newton from the secant's last point refines it (bisection fallback).
// Returns s*, *val = G(s*).
template <int D, bool SPLIT>
__device__ double q_search(const LaneTilt<D, SPLIT>& G, int kind, double lc, double* val)
{
    float flo = 0.0f, fhi = (float)SMAX, sx = NAN;
    const float lcf = (float)lc;
    const float f0 = G.ds32(kind, lcf, 0.0f);
    const bool at_one = !(f0 < 0.0f);
    if (at_one) {
        // G' not negative at q = 1: the boundary case below decides (FP64)
        fhi = (float)SMAX * 0x1p-22f;
    } else {
        float fa = f0, fb = NAN;
        for (int it = 0; it < BISECT_F32; ++it) {
            const float mid = 0.5f * (flo + fhi);
            const float fm = G.ds32(kind, lcf, mid);
            if (fm < 0.0f) { flo = mid; fa = fm; } else { fhi = mid; fb = fm; }
        }
        float ta, ya, tb, yb;
        secant_point(kind, flo, fa, &ta, &ya);
        secant_point(kind, fhi, fb, &tb, &yb);
        int side = 0;
        for (int it = 0; it < SECANT_F32; ++it) {
            float xn = 0.5f * (flo + fhi);   // bisection while G'(fhi) is unknown
            if (yb == yb) {
                const float xs = secant_s(kind, ta - ya * ((tb - ta) / (yb - ya)));
                if (xs == xs) {
                    if (!(xs > flo && xs < fhi)) {   // the root is within rounding of an end
                        sx = (xs < xn) ? flo : fhi;
                        break;
                    }
                    if (sx == sx && fabsf(xs - sx) <= SECANT_STEP) {
                        sx = xs;
                        break;
                    }
                    xn = xs;
                }
            }
            const float fx = G.ds32(kind, lcf, xn);
            float tx, yx;
            secant_point(kind, xn, fx, &tx, &yx);
            sx = xn;
            if (fx < 0.0f) {
                flo = xn; ta = tx; ya = yx;
                if (side < 0) yb *= 0.5f;
                side = -1;
            } else {
                fhi = xn; tb = tx; yb = yx;
                if (side > 0) ya *= 0.5f;
                side = 1;
            }
            if (fhi - flo <= SECANT_TOL) break;
        }
    }
    if (!(sx == sx)) sx = 0.5f * (flo + fhi);
    // minimum at the boundary q = 1 (the objective is quasi-convex in q, Thm. 2):
    // G' was not negative at s = 0 in FP32 and is not in FP64 either.  For the
    // Tilt-Bound the value at q = 1 is 0 exactly (U = 1).
    if (kind == 0 && at_one) {
        double v0;
        if (!(G.ds64(kind, lc, 0.0, nullptr, &v0, nullptr) < 0.0)) {
            *val = v0;
            return 0.0;
        }
    }
    // fast path: Newton from the FP32 estimate; at a smooth optimum two FP64
    // evaluations reach ~1e-20 in s, and the value at the last evaluated point is
    // exact to second order
    double s = (double)sx;
    {
        // one FP64 evaluation: at a smooth optimum a Newton step from the FP32
        // estimate and the second-order Taylor value are exact to O(step^3)
        double d2, v, kd;
        const double g1 = G.ds64(kind, lc, s, &d2, &v, &kd);
        if (d2 > 0.0) {
            const double step = g1 / d2;
            if (fabs(step) <= 4e-5 && kd > 16.0 * fabs(step) + 1e-6 && s - step > 0.0 && s - step < SMAX) {
                *val = v - 0.5 * g1 * step;
                return s - step;
            }
        }
    }
    {
        // Newton steps may leave the FP32 bracket (its derivative's sign can be
        // wrong close to the root) by up to 1e-2 in s; kinks go to the robust path
        const double flo_m = fmax(0.0, (double)flo - 1e-2), fhi_m = fmin(SMAX, (double)fhi + 1e-2);
        for (int it = 0; it < 6; ++it) {
            double d2, v;
            const double g1 = G.ds64(kind, lc, s, &d2, &v, nullptr);
            if (g1 == 0.0) {
                *val = v;
                return s;
            }
            if (!(d2 > 0.0)) break;
            const double step = g1 / d2;
            if (fabs(step) <= 1e-8) {
                *val = v;
                return s - step;
            }
            const double sn = s - step;
            if (!(sn > flo_m && sn < fhi_m)) break;
            s = sn;
        }
    }
    // robust path (kinks of the piecewise-smooth objective, or an FP32 bracket
    // spoilt by rounding): verified bracket, safeguarded Newton with bisection
    double lo = fmax(0.0, (double)flo - 1e-3), hi = fmin(SMAX, (double)fhi + 1e-3);
    if (lo > 0.0 && !(G.ds64(kind, lc, lo, nullptr, nullptr, nullptr) < 0.0)) lo = 0.0;
    if (kind == 0 && lo == 0.0 && !at_one) {   // the boundary test above, for a spoilt bracket
        double v0;
        if (!(G.ds64(kind, lc, 0.0, nullptr, &v0, nullptr) < 0.0)) {
            *val = v0;
            return 0.0;
        }
    }
    if (hi < SMAX && G.ds64(kind, lc, hi, nullptr, nullptr, nullptr) < 0.0) hi = SMAX;
    s = fmin(fmax((double)sx, lo), hi);
    for (int it = 0; it < POLISH_IT; ++it) {
        double d2;
        const double g1 = G.ds64(kind, lc, s, &d2, nullptr, nullptr);
        if (g1 == 0.0) break;
        // a Newton step below 1e-11 at a smooth point: the value is then exact to
        // ~d2 1e-22, well past FP64 (at a kink g1 does not shrink and bisection runs on)
        if (d2 > 0.0 && fabs(g1 / d2) <= 1e-11 * fmax(1.0, fabs(s))) {
            s -= g1 / d2;
            break;
        }
        if (g1 < 0.0) lo = s; else hi = s;
        if (hi - lo <= 1e-15 * fmax(1.0, hi)) break;
        double sn = s - g1 / d2;
        if (!(d2 > 0.0) || !(sn > lo && sn < hi)) sn = 0.5 * (lo + hi);
        if (fabs(sn - s) <= 4e-16 * fmax(1.0, fabs(s))) {
            s = sn;
            break;
        }
        s = sn;
    }
    G.ds64(kind, lc, s, nullptr, val, nullptr);
    return s;
}

// Plain form of the q search: FP64 bisection on the sign of G' over [0, SMAX]
// (64 halvings), no FP32 stage.  Same optimum, more FP64 work.
template <int D>
CSE_HD double q_search_plain(const ArmGeom* G, int kind, double lc, double* val)
{
    double lo = 0.0, hi = SMAX;
    for (int it = 0; it < 64; ++it) {
        const double mid = 0.5 * (lo + hi);
        if (mid <= lo || mid >= hi) break;
        if (obj_ds<D>(G, kind, lc, mid, nullptr, nullptr) < 0.0) lo = mid; else hi = mid;
    }
    const double s = 0.5 * (lo + hi);
    obj_ds<D>(G, kind, lc, s, nullptr, val);
    return s;
}

// log inf_q max_v U(theta0, v, q, a) from log a (a = 1 - l keeps its digits as
// log1p(-l)); *qstar the minimiser.  q = 1 gives U = 1 exactly, so the result
// is at most 0.
// Template parameters: the objective (an arm array, plain form, or a LaneTilt).
template <int D>
CSE_HD double search_any(const ArmGeom* G, int kind, double lc, double* val)
{
    return q_search_plain<D>(G, kind, lc, val);
}

template <int D, bool SPLIT>
__device__ double search_any(const LaneTilt<D, SPLIT>& G, int kind, double lc, double* val)
{
    return q_search(G, kind, lc, val);
}

template <int D>
CSE_HD double phi_inf_any(const ArmGeom* G)
{
    return tilt_phi_inf<D>(G);
}

template <int D, bool SPLIT>
__device__ double phi_inf_any(const LaneTilt<D, SPLIT>& G)
{
    return G.phi_inf();
}

template <int D, typename Obj>
__device__ double tilt_bound_log_la(const Obj& G, double la, double* qstar)
{
    if (la >= 0.0) {
        *qstar = 1.0;
        return 0.0;
    }
    if (la == -INFINITY) {
        *qstar = INFINITY;
        return -INFINITY;
    }
    double val;
    const double s = search_any<D>(G, 0, la, &val);
    if (s > SMAX - 1e-6) {
        const double vinf = la + phi_inf_any<D>(G);
        if (vinf <= val) {
            *qstar = INFINITY;
            return vinf;
        }
    }
    if (val > 0.0) {
        *qstar = 1.0;
        return 0.0;
    }
    *qstar = exp(s);
    return val;
}

// inf_q max_v U(theta0, v, q, a); returns log bound, *qstar.
template <int D, typename Obj>
__device__ double tilt_bound_log(const Obj& G, double a, double* qstar)
{
    if (a >= 1.0) {
        *qstar = 1.0;
        return 0.0;
    }
    if (!(a > 0.0)) {
        *qstar = INFINITY;
        return -INFINITY;
    }
    return tilt_bound_log_la<D>(G, log(a), qstar);
}

// sup_q min_v U^-1(theta0, v, q, alpha); returns log alpha', *qstar.
template <int D, typename Obj>
__device__ double alpha_prime_log(const Obj& G, double alpha, double* qstar)
{
    const double lal = log(alpha);
    double val;
    const double s = search_any<D>(G, 1, lal, &val);
    val = -val;
    if (s > SMAX - 1e-6) {
        const double vinf = lal - phi_inf_any<D>(G);
        if (vinf >= val) {
            *qstar = INFINITY;
            return vinf;
        }
    }
    *qstar = exp(s);
    return val;
}

// ---------------------------------------------------------------------------
// Clopper-Pearson (Eq. clopper-pearson:def): u with P(Binom(N, u) <= R) = delta,
// i.e. I_{1-u}(N - R, R + 1) = delta.  Newton in log space on the regularised
// incomplete beta function (continued fraction times its prefactor): an FP32
// solve to ~1e-6, then FP64 steps until the step is below 1e-9 relative
// (quadratic convergence leaves ~1e-18).
// ---------------------------------------------------------------------------

// Stirling-series remainder lgamma(z) - [(z - 1/2) log z - z + log(2 pi)/2], z >= 10.
CSE_HD __forceinline__ double stirling_rem(double z)
{
    const double r = 1.0 / z, r2 = r * r;
    return r * (1.0 / 12.0 - r2 * (1.0 / 360.0 - r2 * (1.0 / 1260.0 - r2 * (1.0 / 1680.0 - r2 / 1188.0))));
}

CSE_HD __forceinline__ float stirling_rem_f(float z)
{
    const float r = 1.0f / z, r2 = r * r;
    return r * (1.0f / 12.0f - r2 * (1.0f / 360.0f - r2 * (1.0f / 1260.0f)));
}

// lgamma of a positive integer below 19: log of the exactly representable factorial
CSE_HD __forceinline__ double lgamma_small_int(double z)
{
    double f = 1.0;
    for (int k = 2; k < (int)z; ++k) f *= (double)k;
    return log(f);
}

// log(x^a y^b / B(a, b)) for integer a, b >= 1, with lx = log x, ly = log y
// (y = 1 - x) and e = x (a + b) - a supplied accurately by the caller.
CSE_HD double log_bpre(double a, double b, double lx, double ly, double e)
{
    const double L2PI = 1.8378770664093454836;
    if (a >= 10.0 && b >= 10.0) {
        return a * log1p(e / a) + b * log1p(-e / b) + 0.5 * log(a * b / (a + b)) - 0.5 * L2PI
               - (stirling_rem(a) + stirling_rem(b) - stirling_rem(a + b));
    }
    if (b >= 10.0) {   // small a: lgamma(a+b) - lgamma(b) by the Stirling difference
        return a * lx + b * ly - lgamma_small_int(a) + a * log(a + b) + (b - 0.5) * log1p(a / b) - a
               + stirling_rem(a + b) - stirling_rem(b);
    }
    if (a >= 10.0) {
        return a * lx + b * ly - lgamma_small_int(b) + b * log(a + b) + (a - 0.5) * log1p(b / a) - b
               + stirling_rem(a + b) - stirling_rem(a);
    }
    return a * lx + b * ly - lgamma_small_int(a) - lgamma_small_int(b) + lgamma_small_int(a + b);
}

CSE_HD float log_bpre_f(float a, float b, float lx, float ly, float e)
{
    if (a >= 10.0f && b >= 10.0f) {
        return a * log1pf(e / a) + b * log1pf(-e / b) + 0.5f * logf(a * b / (a + b)) - 0.9189385332f
               - (stirling_rem_f(a) + stirling_rem_f(b) - stirling_rem_f(a + b));
    }
    return a * lx + b * ly - lgammaf(a) - lgammaf(b) + lgammaf(a + b);
}

// Continued fraction 1/(1 + d1/(1 + d2/(1 + ...))) of I_x(a, b), with
// d_{2m+1} = -(a+m)(a+b+m)x / ((a+2m)(a+2m+1)), d_{2m} = m(b-m)x / ((a+2m-1)(a+2m)).
// FP64, division-free: three-term recurrences of the equivalent fraction whose
// partial numerators / denominators are the polynomials p, q of d = p/q, rescaled
// by exact powers of two; one division per convergence check.
CSE_HD double beta_cf(double a, double b, double x)
{
    // d_{2m+1} = p_odd / q_odd, d_{2m} = p_even / q_even; the numerator and
    // denominator polynomials are advanced by their differences in m
    double po_f = a * (a + b);             // (a+m)(a+b+m) at m = 0
    double po_df = 2.0 * a + b + 1.0;      // its first difference at m = 0
    double qo = a * (a + 1.0);             // (a+2m)(a+2m+1) at m = 0
    double qo_d = 4.0 * a + 6.0;           // first difference (second difference 8)
    double pe_f = b - 1.0;                 // m (b-m) at m = 1
    double pe_df = b - 3.0;                // first difference at m = 1 (second difference -2)
    double qe = (a + 1.0) * (a + 2.0);     // (a+2m-1)(a+2m) at m = 1
    double qe_d = 4.0 * a + 10.0;          // first difference (second difference 8)
    double Am2 = 0.0, Am1 = 1.0, Bm2 = 1.0, Bm1 = 1.0;   // A_0, A_1, B_0, B_1
    double qprev = 1.0, f_old = 1.0;
    const double BIG = 0x1p600, SMALL = 0x1p-600;
    for (int k = 2; k < 4000; ++k) {
        double p, q;
        if (k & 1) {                       // level k uses d_{k-1}, k-1 even
            p = pe_f * x;
            q = qe;
            pe_f += pe_df;
            pe_df -= 2.0;
            qe += qe_d;
            qe_d += 8.0;
        } else {                           // k-1 odd
            p = -po_f * x;
            q = qo;
            po_f += po_df;
            po_df += 2.0;
            qo += qo_d;
            qo_d += 8.0;
        }
        const double an = qprev * p;
        const double A = q * Am1 + an * Am2;
        const double B = q * Bm1 + an * Bm2;
        Am2 = Am1;
        Am1 = A;
        Bm2 = Bm1;
        Bm1 = B;
        qprev = q;
        if (fabs(Bm1) > BIG) {             // exact rescaling by a power of two
            Am2 *= SMALL;
            Am1 *= SMALL;
            Bm2 *= SMALL;
            Bm1 *= SMALL;
        }
        if ((k & 7) == 0) {
            const double f = Am1 / Bm1;
            if (fabs(f - f_old) <= 1e-14 * fabs(f)) return f;
            f_old = f;
        }
    }
    return Am1 / Bm1;
}

// FP32 modified Lentz evaluation of the same fraction (start of the solve).
CSE_HD float beta_cf_f(float a, float b, float x)
{
    const float TINY = 1e-30f;
    const float qab = a + b, qap = a + 1.0f, qam = a - 1.0f;
    float c = 1.0f, dd = 1.0f - fdiv_fast(qab * x, qap);
    if (fabsf(dd) < TINY) dd = TINY;
    dd = fdiv_fast(1.0f, dd);
    float h = dd;
    for (int m = 1; m <= 300; ++m) {
        const float m2 = 2.0f * m;
        float aa = fdiv_fast(m * (b - m) * x, (qam + m2) * (a + m2));
        dd = 1.0f + aa * dd;
        if (fabsf(dd) < TINY) dd = TINY;
        c = 1.0f + fdiv_fast(aa, c);
        if (fabsf(c) < TINY) c = TINY;
        dd = fdiv_fast(1.0f, dd);
        h *= dd * c;
        aa = -fdiv_fast((a + m) * (qab + m) * x, (a + m2) * (qap + m2));
        dd = 1.0f + aa * dd;
        if (fabsf(dd) < TINY) dd = TINY;
        c = 1.0f + fdiv_fast(aa, c);
        if (fabsf(c) < TINY) c = TINY;
        dd = fdiv_fast(1.0f, dd);
        const float del = dd * c;
        h *= del;
        // the FP32 phase needs ~1e-6: a 1-ulp test may never be met under FMA rounding
        if (fabsf(del - 1.0f) <= 1e-6f) break;
    }
    return h;
}

// log P(Binom(N, u) <= R) = log I_{1-u}(b, a) and log pdf of Beta(a, b) at u,
// a = R + 1, b = N - R.  The prefactor is symmetric in (a, u) <-> (b, 1 - u).
CSE_HD double log_binom_cdf(double a, double b, double u, double* lpdf)
{
    const double lu = log(u), l1u = log1p(-u);
    const double e = fma(u, a + b, -a);   // u (a+b) - a
    const double lp = log_bpre(a, b, lu, l1u, e);
    *lpdf = lp - lu - l1u;
    if (u >= (a + 1.0) / (a + b + 2.0)) return lp + log(beta_cf(b, a, 1.0 - u)) - log(b);
    return log1p(-exp(lp) * beta_cf(a, b, u) / a);
}

CSE_HD float log_binom_cdf_f(float a, float b, float u, float* lpdf)
{
    const float lu = logf(u), l1u = log1pf(-u);
    const float e = fmaf(u, a + b, -a);
    const float lp = log_bpre_f(a, b, lu, l1u, e);
    *lpdf = lp - lu - l1u;
    if (u >= (a + 1.0f) / (a + b + 2.0f)) return lp + logf(beta_cf_f(b, a, 1.0f - u)) - logf(b);
    return log1pf(-expf(lp) * beta_cf_f(a, b, u) / a);
}

// Small R: log P(Binom(N, u) <= R) = N log(1-u) + log sum_{j<=R} C(N,j) w^j,
// w = u / (1-u), by the term recurrence t_{j+1} = t_j (N-j) w / (j+1); the
// Beta(R+1, N-R) log density at u is log((N-R) t_R) + (N-1) log(1-u) + ... .
constexpr int64_t CP_SMALL_R = 40;
CSE_HD double log_binom_cdf_small(int64_t R, int64_t N, double u, double* lpdf)
{
    const double l1u = log1p(-u);
    const double w = u / (1.0 - u);
    double t = 1.0, sum = 1.0;
    for (int64_t j = 0; j < R; ++j) {
        t *= (double)(N - j) * w / (double)(j + 1);
        sum += t;
    }
    const double base = (double)N * l1u;
    *lpdf = log((double)(N - R) * t) + base - l1u;
    return base + log(sum);
}

// Plain form: FP64 Newton from the normal-approximation start, no FP32 stage.
CSE_HD double cp_upper_plain(int64_t R, int64_t N, double delta)
{
    if (R >= N) return 1.0;
    if (R <= 0) return -expm1(log(delta) / (double)N);
    const double a = (double)R + 1.0, b = (double)(N - R);
    const double ld = log(delta);
    const double mean = a / (a + b);
    const double sd = sqrt(a * b / ((a + b) * (a + b) * (a + b + 1.0)));
    double u = fmin(mean + 2.5 * sd, 0.5 * (mean + 1.0));
    const bool small = R < CP_SMALL_R && N - R > CP_SMALL_R;
    double lo = 0.0, hi = 1.0;
    for (int it = 0; it < 100; ++it) {
        double lpdf;
        const double lF = small ? log_binom_cdf_small(R, N, u, &lpdf) : log_binom_cdf(a, b, u, &lpdf);
        const double f = lF - ld;
        const double nstep = f / (-exp(lpdf - lF));
        if (fabs(nstep) <= 4e-16 * u) break;
        if (f > 0.0) lo = u; else hi = u;
        double un = u - nstep;
        if (!(un > lo && un < hi)) un = 0.5 * (lo + hi);
        u = un;
    }
    return u;
}

// FP32 f(u) = log P(Binom(N,u) <= R) - log delta (the FP32 search stage)
CSE_HD float cp_f32(int64_t R, int64_t N, float u, float ldf, float* lpdf)
{
    const bool small = R < CP_SMALL_R && N - R > CP_SMALL_R;
    if (small) {
        const float l1u = log1pf(-u), w = u / (1.0f - u);
        float t = 1.0f, sum = 1.0f;
        for (int j = 0; j < (int)R; ++j) {
            t *= fdiv_fast((float)(N - j) * w, (float)(j + 1));
            sum += t;
        }
        const float base = (float)N * l1u;
        if (lpdf) *lpdf = logf((float)(N - R) * t) + base - l1u;
        return base + logf(sum) - ldf;
    }
    float lp;
    const float lF = log_binom_cdf_f((float)R + 1.0f, (float)(N - R), u, &lp);
    if (lpdf) *lpdf = lp;
    return lF - ldf;
}

// FP64 stage from an estimate u: Halley steps on phi(u) = log F(u) - log delta,
// phi' = -pdf/F, phi'' = -(pdf/F) ((a-1)/u - (b-1)/(1-u)) - (pdf/F)^2.  From an
// FP32-accurate estimate one step leaves an error of order step^3.
CSE_HD double cp_finish_fp64(int64_t R, int64_t N, double delta, double u)
{
    const double a = (double)R + 1.0, b = (double)(N - R);
    const double ld = log(delta);
    const bool small = R < CP_SMALL_R && N - R > CP_SMALL_R;
    double lo = 0.0, hi = 1.0;
    for (int it = 0; it < 60; ++it) {
        double lpdf;
        const double lF = small ? log_binom_cdf_small(R, N, u, &lpdf) : log_binom_cdf(a, b, u, &lpdf);
        const double f = lF - ld;
        if (f == 0.0) break;
        const double r = exp(lpdf - lF);
        const double p1 = -r;
        const double p2 = -r * ((a - 1.0) / u - (b - 1.0) / (1.0 - u)) - r * r;
        const double den = 2.0 * p1 * p1 - f * p2;
        const double du = (den != 0.0) ? -2.0 * f * p1 / den : -f / p1;
        if (fabs(du) <= 4e-16 * u) break;   // converged to rounding
        if (f > 0.0) lo = u; else hi = u;
        double un = u + du;
        if (!(un > lo && un < hi)) un = 0.5 * (lo + hi);
        const double step = fabs(un - u);
        u = un;
        if (step <= 3e-6 * fmin(u, 1.0 - u) || hi - lo <= 4e-16 * hi) break;
    }
    return u;
}

CSE_HD double cp_upper(int64_t R, int64_t N, double delta)
{
    if (R >= N) return 1.0;
    if (R <= 0) return -expm1(log(delta) / (double)N);
    const double a = (double)R + 1.0, b = (double)(N - R);
    const double mean = a / (a + b);
    const double sd = sqrt(a * b / ((a + b) * (a + b) * (a + b + 1.0)));
    double u = fmin(mean + 2.5 * sd, 0.5 * (mean + 1.0));
    // FP32 stage: safeguarded Newton
    {
        const float ldf = (float)log(delta);
        float uf = (float)u, lof = 0.0f, hif = 1.0f;
        for (int it = 0; it < 16; ++it) {
            float lpdf;
            const float f = cp_f32(R, N, uf, ldf, &lpdf);
            if (f > 0.0f) lof = uf; else hif = uf;
            const float dlF = -expf(lpdf - (f + ldf));
            float un = uf - f / dlF;
            if (!(un > lof && un < hif)) un = 0.5f * (lof + hif);
            const bool done = fabsf(un - uf) <= 1e-6f * uf;
            uf = un;
            if (done) break;
        }
        if (uf > 0.0f && uf < 1.0f) u = (double)uf;
    }
    return cp_finish_fp64(R, N, delta, u);
}

// ---------------------------------------------------------------------------
// Clopper-Pearson by groups of L lanes, one key a group.
//
// An FP64 warp instruction takes the same pipe time (64 cycles) however many of
// its lanes are active, so a key's FP64 work is spread over the lanes of a group
// and a warp solves 32 / L keys with one instruction stream:
//  * the continued fraction as a composition of linear fractional maps, i.e. a
//    product of 2x2 matrices (associative): each lane multiplies its consecutive
//    levels, a shuffle tree forms the ordered product, and the product of the
//    first half of the lanes gives, for free, the convergent at half the depth,
//    which is the convergence test;
//  * the two log1p of the prefactor, its three Stirling terms and the logarithm of
//    the fraction one a lane;
//  * the small-R binomial sum as an ordered product of (product, sum) pairs.
// The density over the tail, which the Halley step needs, follows from the
// fraction alone: pdf / tail = 1 / (h u (1 - u)).
// A key starts at the two-term Cornish-Fisher point of Beta(R + 1, N - R), takes
// FP32 Halley steps of the same evaluation to ~1e-5 standard deviations, then one
// FP64 Halley step (error of the order of the step cubed).  Levels needed for
// N <= 65536 at delta = 0.01, 0.005: at most 28 for 1e-6, 110 for 1e-15; a pass
// holds 32 in FP32 and 96 in FP64 (two to a step of the contracted fraction).
// ---------------------------------------------------------------------------
template <typename T>
struct Mat2 {
    T m00, m01, m10, m11;
};

template <typename T>
__device__ __forceinline__ Mat2<T> mat2_mul(const Mat2<T>& A, const Mat2<T>& B)
{
    return {fma(A.m00, B.m00, A.m01 * B.m10), fma(A.m00, B.m01, A.m01 * B.m11),
            fma(A.m10, B.m00, A.m11 * B.m10), fma(A.m10, B.m01, A.m11 * B.m11)};
}

// x 2^k (x normal or zero, the result too): an integer addition to the exponent
// field instead of an FP64 multiplication.
__device__ __forceinline__ double scale_exp(double x, int k)
{
    const int hi = __double2hiint(x);
    return (hi & 0x7FFFFFFF) ? __hiloint2double(hi + (k << 20), __double2loint(x)) : 0.0;
}

// Scales by the power of two that brings the largest entry into [1, 2): exact,
// and the convergents are ratios of entries, so they are unchanged.  Entries below
// 2^-900 of the largest become zero.  (FP32 entries stay in range without it.)
__device__ __forceinline__ void mat2_norm(Mat2<double>& A)
{
    auto ex = [](double x) { return (__double2hiint(x) >> 20) & 0x7ff; };
    const int e0 = ex(A.m00), e1 = ex(A.m01), e2 = ex(A.m10), e3 = ex(A.m11);
    const int e = max(max(e0, e1), max(e2, e3)), k = 1023 - e;
    A.m00 = e0 > e - 900 ? scale_exp(A.m00, k) : 0.0;
    A.m01 = e1 > e - 900 ? scale_exp(A.m01, k) : 0.0;
    A.m10 = e2 > e - 900 ? scale_exp(A.m10, k) : 0.0;
    A.m11 = e3 > e - 900 ? scale_exp(A.m11, k) : 0.0;
}

__device__ __forceinline__ void mat2_norm(Mat2<float>& A)
{
    const float m = fmaxf(fmaxf(A.m00, A.m01), fmaxf(A.m10, A.m11));   // entries are not negative
    const int e = min(max((__float_as_int(m) >> 23) & 0xff, 1), 253);
    const float sc = __int_as_float((254 - e) << 23);
    A.m00 *= sc;
    A.m01 *= sc;
    A.m10 *= sc;
    A.m11 *= sc;
}

// Right-multiplies C by the map t -> p / (q + k t), [[0, p], [k, q]].
template <typename T>
__device__ __forceinline__ void cf_step(Mat2<T>& C, T p, T q, T k)
{
    const T c00 = C.m00, c10 = C.m10;
    C.m00 = C.m01 * k;
    C.m01 = fma(c00, p, C.m01 * q);
    C.m10 = C.m11 * k;
    C.m11 = fma(c10, p, C.m11 * q);
}

template <typename T, int L>
__device__ __forceinline__ Mat2<T> mat2_down(const Mat2<T>& A, int s, unsigned mask)
{
    return {__shfl_down_sync(mask, A.m00, s, L), __shfl_down_sync(mask, A.m01, s, L),
            __shfl_down_sync(mask, A.m10, s, L), __shfl_down_sync(mask, A.m11, s, L)};
}

template <typename T, int L>
__device__ __forceinline__ Mat2<T> mat2_first(const Mat2<T>& A, unsigned mask)
{
    return {__shfl_sync(mask, A.m00, 0, L), __shfl_sync(mask, A.m01, 0, L), __shfl_sync(mask, A.m10, 0, L),
            __shfl_sync(mask, A.m11, 0, L)};
}

// h with I_x(a, b) = x^a (1-x)^b / B(a, b) h, from lam = a - (a + b) x >= 0: the even
// contraction of the fraction 1/(1 + d1/(1 + d2/(1 + ...))) of beta_cf, whose step
// n is the map t -> alpha_n / (beta_n + t) with
//   alpha_n = (a+n-1)(a+b+n-1) n (b-n) x^2 / (a+2n-1)^2      (alpha_0 = 1),
//   beta_n  = (a+2n)(1 + d_{2n} + d_{2n+1})
//           = n + n(b-n)x/(a+2n-1) + (a+n)(lam + 1 + n(2-x))/(a+2n+1):
// all terms positive for n < b, so nothing cancels (d_{2n+1} is near -1), and
// for integer b the fraction ends at n = b; the steps past it are left out.  h is
// the composition of the maps applied to t = 0: with Q the product of their
// matrices, Q01 / Q11.  In FP64 a step is multiplied through by (a+2n-1)^2
// (a+2n+1) instead of divided (a common factor does not change the map); in FP32
// it is scaled by a + 2n, which keeps the entries in range.  The even contraction of a
// continued fraction: Jones and Thron, Continued Fractions (1980), ch. 2.
// The convergents close in geometrically, so in the first pass a difference of 1e-9
// (FP32: 1e-3) between half and full depth leaves the full depth at rounding (5e-16
// at most, in extended precision, over N = 100 .. 2^20 and delta = 1e-6 .. 0.999); one pass
// does at the usual delta.  As u nears the mean more are needed, and from the second
// pass on the two depths compared are 24 steps apart in 72 and more, so the
// difference has to be at rounding itself (1e-14 there leaves 4e-16; 1e-9 left 7e-11 at
// N = 2^20, delta = 0.5).
template <typename T, int L>
__device__ T beta_cf_group(T a, T b, T x, T lam, int l, unsigned mask)
{
    constexpr bool F64 = sizeof(T) == 8;
    constexpr int STEPS = (F64 ? 48 : 16) / L;   // per lane and pass
    const T s = a + b;
    Mat2<T> P = {(T)1, (T)0, (T)0, (T)1};
    T f = (T)0;
    for (int pass = 0; pass < 40; ++pass) {
        Mat2<T> C = {(T)1, (T)0, (T)0, (T)1};
        const T g = (T)((pass * L + l) * STEPS);
#pragma unroll
        for (int i = 0; i < STEPS; ++i) {
            const T n = g + (T)i;
            if (n < b) {
                const T an = a + n, dm = an + (n - (T)1), dp = an + (n + (T)1);
                const T w = n * (b - n) * x, c = fma(n, (T)2 - x, lam + (T)1);
                const T num = n > (T)0 ? (an - (T)1) * (s + (n - (T)1)) * (w * x) : (T)1;
                if (F64) {
                    const T d2 = dm * dm;
                    // n = 0: alpha = 1, so the factor is dp alone
                    if (n > (T)0) cf_step(C, num * dp, fma(d2, fma(an, c, n * dp), w * dm * dp), d2 * dp);
                    else cf_step(C, dp, an * c, dp);
                } else {
                    const float im = fdiv_fast(1.0f, (float)dm), ip = fdiv_fast(1.0f, (float)dp);
                    const float k = fdiv_fast(1.0f, (float)(an + n));   // 1 / (a + 2n)
                    const float pv = n > (T)0 ? (float)num * im * im * k : k;
                    cf_step<T>(C, (T)pv, (T)(((float)n + (float)w * im + (float)(an * c) * ip) * k), (T)k);
                }
            }
            // a step grows FP64 entries by at most 2^85, shrinks FP32 ones by at most 2^-20
            if (F64 ? (i % 6) == 5 : (i % 4) == 3) mat2_norm(C);
        }
        mat2_norm(C);
        Mat2<T> half = C;
#pragma unroll
        for (int sh = 1; sh < L; sh <<= 1) {   // lane 0 ends with lanes 0..2sh-1
            half = C;
            C = mat2_mul(C, mat2_down<T, L>(C, sh, mask));
            mat2_norm(C);
        }
        // lane 0 forms both convergents; the group takes its decision
        const Mat2<T> Ph = mat2_mul(P, half);
        P = mat2_mul(P, C);
        mat2_norm(P);
        P = mat2_first<T, L>(P, mask);
        const T f_mid = __shfl_sync(mask, Ph.m01 / Ph.m11, 0, L);
        f = P.m01 / P.m11;
        if (!(fabs(f - f_mid) > (T)(F64 ? (pass == 0 ? 1e-9 : 1e-14) : 1e-3) * fabs(f))) break;
    }
    return f;
}

template <typename T, int L>
__device__ __forceinline__ T group_sum(T v, unsigned mask)
{
#pragma unroll
    for (int sh = L / 2; sh > 0; sh >>= 1) v += __shfl_xor_sync(mask, v, sh, L);
    return v;
}

__device__ __forceinline__ double g_log(double x) { return log(x); }
__device__ __forceinline__ float g_log(float x) { return logf(x); }
__device__ __forceinline__ double g_log1p(double x) { return log1p(x); }
__device__ __forceinline__ float g_log1p(float x) { return log1pf(x); }
__device__ __forceinline__ double g_stirling(double z) { return stirling_rem(z); }
__device__ __forceinline__ float g_stirling(float z) { return stirling_rem_f(z); }

// Log of the tail the solve works on and *r = density at u over that tail, for a, b >= 10
// (a = R + 1, b = N - R): upper (u above the mean) P(Binom <= R) = I_{1-u}(b, a), else its
// complement I_u(a, b).
template <typename T, int L>
__device__ T log_tail_cf(T a, T b, T u, bool upper, T* r, int l, unsigned mask)
{
    const T s = a + b, e = fma(u, s, -a);   // u (a + b) - a
    const T cf = upper ? beta_cf_group<T, L>(b, a, (T)1 - u, e, l, mask) : beta_cf_group<T, L>(a, b, u, -e, l, mask);
    *r = (T)1 / (cf * u * ((T)1 - u));
    T v = (T)0;
#pragma unroll
    for (int t = 0; t < 6; t += L) {   // term t + l on lane l
        const int k = t + l;
        if (k < 2) {
            const T z = k ? b : a;
            v += z * g_log1p((k ? -e : e) / z);
        } else if (k < 5) {
            const T st = g_stirling(k == 2 ? a : k == 3 ? b : s);
            v += k == 4 ? st : -st;
        } else if (k == 5) {   // log(sqrt(a b / (a + b)) cf)
            v += (T)0.5 * g_log(cf * cf * (a * b / s));
        }
    }
    return group_sum<T, L>(v, mask) - (T)0.91893853320467274178;   // log(2 pi) / 2
}

// The same for R < CP_SMALL_R, each lane taking a stretch of the terms: upper
//   log P(Binom(N, u) <= R) = N log(1-u) + log sum_{j<=R} C(N,j) w^j, w = u / (1-u),
// else (delta > 0.9, u well below the mean)
//   log P(Binom(N, u) > R) = log t_{R+1} + log(1 + sum of the next terms over t_{R+1}),
// whose terms fall fast: kTailTerms of them reach below rounding.
constexpr int kTailTerms = 96;

template <typename T, int L>
__device__ T log_tail_sum(int R, T N, T u, bool upper, T* r, int l, unsigned mask)
{
    const T w = u / ((T)1 - u);
    const int R1 = upper ? R : R + 1;
    const int per = (R1 + L - 1) / L, j0 = l * per + 1, j1 = min(R1, (l + 1) * per);
    T p = (T)1, sum = (T)0;   // product and sum of the partial products of the stretch
    for (int j = j0; j <= j1; ++j) {
        p *= (N - (T)(j - 1)) * w / (T)j;
        sum += p;
    }
    auto chain = [&](T& p0, T& s0) {   // the ordered composition over the lanes, in every lane
#pragma unroll
        for (int sh = 1; sh < L; sh <<= 1) {
            const T p2 = __shfl_down_sync(mask, p0, sh, L), s2 = __shfl_down_sync(mask, s0, sh, L);
            s0 = fma(p0, s2, s0);
            p0 *= p2;
        }
        p0 = __shfl_sync(mask, p0, 0, L);
        s0 = __shfl_sync(mask, s0, 0, L) + (T)1;
    };
    chain(p, sum);
    if (upper) {
        *r = (N - (T)R) * p / (sum * ((T)1 - u));
        return fma(N, g_log1p(-u), g_log(sum));
    }
    T q = (T)1, tail = (T)0;
    for (int i = 0; i < kTailTerms / L; ++i) {
        const T j = (T)(R + 2 + l * (kTailTerms / L) + i);
        q *= (N - (j - (T)1)) * w / j;   // zero from j = N + 1 on
        tail += q;
    }
    chain(q, tail);
    *r = (T)(R + 1) / (u * tail);
    return fma(N, g_log1p(-u), g_log(p * tail));
}

// One Halley step on phi(u) = log tail - target from f = phi(u): phi' = -r (upper)
// or r, phi'' = phi' ((a-1)/u - (b-1)/(1-u)) - r^2; kept inside the bracket (lo,
// hi), which the sign of f narrows.
template <typename T>
__device__ __forceinline__ T cp_halley(T u, T f, T r, T a, T b, bool upper, T* lo, T* hi)
{
    const T p1 = upper ? -r : r;
    // (numerator and denominator times u (1 - u): one division)
    const T v = u * ((T)1 - u), p2v = p1 * ((a - (T)1) - (a + b - (T)2) * u) - p1 * p1 * v;
    const T den = (T)2 * p1 * p1 * v - f * p2v;
    if ((f > (T)0) == upper) *lo = u;
    else *hi = u;
    const T un = u - (T)2 * f * p1 * v / den;
    return (un >= *lo && un <= *hi) ? un : (T)0.5 * (*lo + *hi);
}

// The serial solve, called (rarely) rather than inlined: its registers would halve
// the warps of the group solve.
__device__ __noinline__ double cp_upper_serial(int64_t R, int64_t N, double delta)
{
    return cp_upper(R, N, delta);
}

// u with P(Binom(N, u) <= R) = delta, 0 < R < N, all lanes of a group together; comp =
// 1 - delta from the caller, who may know it to more digits; z is the normal
// quantile of comp.
template <int L>
__device__ double cp_upper_group(int64_t R, int64_t N, double delta, double comp, float z, int l, unsigned mask)
{
    const double a = (double)R + 1.0, b = (double)(N - R);
    const bool small = R < CP_SMALL_R && (N - R > CP_SMALL_R || delta > 0.9);
    if (!small && (a < 10.0 || b < 10.0)) return cp_upper_serial(R, N, delta);   // few trials: every lane alike
    const bool upper = delta <= (small ? 0.9 : 0.5);
    const double target = log(upper ? delta : comp);
    const float af = (float)a, bf = (float)b, sf = af + bf;
    const float mean = af / sf, sd = sqrtf(af * bf / (sf * sf * (sf + 1.0f)));
    const float skew = 2.0f * (bf - af) * sqrtf(sf + 1.0f) / ((sf + 2.0f) * sqrtf(af * bf));
    float u = mean + sd * (z + skew * (z * z - 1.0f) * (1.0f / 6.0f));
    u = fminf(fmaxf(u, 0.02f * mean), 0.5f * (mean + 1.0f));
    float lof = 0.0f, hif = 1.0f;
    for (int it = 0; it < 12; ++it) {
        float r;
        const float lt = small ? log_tail_sum<float, L>((int)R, (float)N, u, upper, &r, l, mask)
                               : log_tail_cf<float, L>(af, bf, u, upper, &r, l, mask);
        const float un = cp_halley<float>(u, lt - (float)target, r, af, bf, upper, &lof, &hif);
        const float step = __shfl_sync(mask, fabsf(un - u), 0, L);   // one decision for the group
        u = __shfl_sync(mask, un, 0, L);
        if (!(__shfl_sync(mask, r, 0, L) > 0.0f)) break;
        if (!(step > 1e-3f * fminf(sd, fminf(u, 1.0f - u)))) break;   // the next one would be ~1e-9 of it
    }
    double ud = (u > 0.0f && u < 1.0f) ? (double)u : (double)mean;   // a poor start costs FP64 steps
    double lo = 0.0, hi = 1.0;
    for (int it = 0; it < 60; ++it) {
        double r;
        const double lt = small ? log_tail_sum<double, L>((int)R, (double)N, ud, upper, &r, l, mask)
                                : log_tail_cf<double, L>(a, b, ud, upper, &r, l, mask);
        const double un = cp_halley<double>(ud, lt - target, r, a, b, upper, &lo, &hi);
        const double step = __shfl_sync(mask, fabs(un - ud), 0, L);
        ud = __shfl_sync(mask, un, 0, L);
        // far on the wrong side of the mean the fraction loses its sign: the serial solve
        if (!(__shfl_sync(mask, r, 0, L) > 0.0)) return cp_upper_serial(R, N, delta);
        // Halley's error is at most 0.12 step^3 / sd^2 (largest at delta = 1/2): below 1e-16 of u
        if (!(step > fmin(2e-5 * (double)sd, 3e-6 * fmin(ud, 1.0 - ud))) || hi - lo <= 4e-16 * hi) break;
    }
    return ud;
}

// Device-side argument checks of tile i: a tile must meet some null hypothesis
// (null_mask != 0) and have half-widths h >= 0 (h = 0: a point); false and the
// error flag (reported by cse_sync as DEVICE_CHECK) otherwise.
template <int D>
__device__ bool tile_args_ok(const TileArgs& T, int64_t i, int32_t* err)
{
    bool ok = T.null_mask[i] != 0u;
#pragma unroll
    for (int a = 0; a < D; ++a) ok &= T.halfwidth[i * D + a] >= 0.0;   // false for NaN too
    if (!ok) atomicOr(err, CSE_ERR_BAD_K);
    return ok;
}

// Loads tile i's centre and half-widths; false (and the error flag) when an
// axis index is out of range or tile_args_ok fails.
template <int D>
__device__ bool load_tile(const TileArgs& T, int64_t i, double n_max, ArmGeom* G, int32_t* err)
{
    if (!tile_args_ok<D>(T, i, err)) return false;
#pragma unroll
    for (int a = 0; a < D; ++a) {
        const int v = T.center_idx[i * D + a];
        if (v < 0 || v >= T.n_axis[a]) {
            atomicOr(err, CSE_ERR_BAD_K);
            return false;
        }
        arm_init(G[a], T.axis[a][v], T.halfwidth[i * D + a], n_max);
    }
    return true;
}

// The same by the group of lanes l = 0 .. NL-1, each its own arm (and sign); the
// checks hold for the whole tile.  geom: each tile's softplus terms (sp(th),
// sp(th + h) - sp(th), sp(th - h) - sp(th), 3 doubles an arm), written by
// k_alpha_prime (store) and read by k_bounds of the same step (load), which takes
// the same values instead of recomputing them.
template <int D, bool SPLIT>
__device__ bool load_lane(const TileArgs& T, int64_t i, int l, double n_max, LaneTilt<D, SPLIT>& G, int32_t* err,
                          const double* __restrict__ geom_in, double* __restrict__ geom_out)
{
    constexpr int NL = LaneTilt<D, SPLIT>::NL;
    const int a = SPLIT ? l >> 1 : l;
    G.sg = SPLIT ? l & 1 : 0;
    G.mask = (NL == 32 ? 0xffffffffu : ((1u << NL) - 1u) << ((threadIdx.x & 31) & ~(NL - 1)));
    const double h = T.halfwidth[i * D + a];
    const int v = T.center_idx[i * D + a];
    int na = T.n_axis[0];
    const double* axis = T.axis[0];
#pragma unroll
    for (int b = 1; b < D; ++b)   // by selection: no runtime index into the argument
        if (a == b) {
            na = T.n_axis[b];
            axis = T.axis[b];
        }
    const bool ok = T.null_mask[i] != 0u && h >= 0.0 && v >= 0 && v < na;   // false for a NaN half-width too
    if (!__all_sync(G.mask, ok)) {
        if (l == 0) atomicOr(err, CSE_ERR_BAD_K);
        return false;
    }
    const double th = axis[v];
    if (geom_in) {
        const double* g = geom_in + (i * D + a) * 3;
        G.th = th;
        G.h = h;
        G.n = n_max;
        G.sp0 = g[0];
        G.d1[0] = g[1 + G.sg];
        if (!SPLIT) G.d1[SPLIT ? 0 : 1] = g[2];
        G.init_f32();
    } else {
        G.init(th, h, n_max);
    }
    if (geom_out) {
        double* g = geom_out + (i * D + a) * 3;
        if (G.sg == 0) g[0] = G.sp0;
        g[1 + G.sg] = G.d1[0];
        if (!SPLIT) g[2] = G.d1[SPLIT ? 0 : 1];
    }
    return true;
}

// Clopper-Pearson depends on a tile only through (R, K): every distinct pair is
// solved once.  k_cp_mark inserts each tile's key (K << 32 | R) into an
// open-addressing hash table (linear probing, at most `cap` probes, no waiting)
// and records its slot; k_cp_solve solves each occupied slot; k_bounds reads it.
constexpr unsigned long long kEmptyKey = kCpEmptyKey;

__global__ void k_cp_mark(int64_t n_tiles, const int64_t* __restrict__ R, const int32_t* __restrict__ K,
                          unsigned long long* __restrict__ keys, uint32_t cap, int32_t* __restrict__ slot,
                          uint32_t* __restrict__ list, int32_t* __restrict__ n_keys, bool lower)
{
    pdl_entry();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_tiles) return;
    // Upper bound: the solve for R at delta.  Lower bound (see k_bounds): for
    // R > K/2 the upper solve for the K - R failures at delta, else the solve
    // for R - 1 at 1 - delta, tagged by the key's top bit; R = 0 needs none.
    int64_t Rk = R[i];
    unsigned long long tag = 0ull;
    if (lower) {
        if (2 * R[i] > (int64_t)K[i]) {
            Rk = (int64_t)K[i] - R[i];
        } else {
            Rk = R[i] - 1;
            tag = 1ull << 63;
        }
        if (Rk < 0) {
            slot[i] = -1;
            return;
        }
    }
    const unsigned long long key = tag | ((unsigned long long)(uint32_t)K[i] << 32) | (uint32_t)Rk;
    slot[i] = cp_memo_insert(key, keys, cap, list, n_keys);
}

// The distinct (K, R) keys, a group of 8 lanes each: key t goes to group t / W of
// warp t % W (W warps in the grid), so keys spread over the warps before they
// share one.  Beyond kCpManyKeys the FP64 pipe is full and the total work counts:
// 2 lanes a key do less of it (fewer tree steps, more of the serial levels).
// Bound by the latency of one warp's chain of FP64 instructions until every
// sub-partition has a few warps.  Against a warp for each of the first 1,216 keys
// (bracketing by FP32 rounds, 256 levels) and a thread for each further key: one
// arm, 64 keys 37 -> 28 us; 1,500 distinct keys 212 -> 29; 6,036 keys 353 -> 64;
// two-arm batch 350 -> 60; basket 16^4 274 -> 110.
constexpr int kCpThreads = 128;
constexpr int kCpBlocksPerSM = 3;
constexpr int kCpManyKeys = 40000;

template <int L>
__device__ __forceinline__ void cp_solve_keys(unsigned long long* __restrict__ keys, const uint32_t* __restrict__ list,
                                              int n, double delta0, double delta1, float z0,
                                              double* __restrict__ u0s)
{
    const int lane = threadIdx.x & 31, l = lane & (L - 1), g = lane / L;
    const unsigned mask = (L == 32 ? 0xffffffffu : ((1u << L) - 1u) << (g * L));
    const int W = gridDim.x * (kCpThreads / 32);
    for (int t = g * W + (threadIdx.x >> 5) * gridDim.x + blockIdx.x; t < n; t += W * (32 / L)) {
        const uint32_t h = list[t];
        const unsigned long long key = keys[h];
        const int64_t R = (int64_t)(uint32_t)key, N = (int64_t)((key >> 32) & 0x7FFFFFFFull);
        const bool tag = (key >> 63) != 0;   // the lower bound's solve at delta1 = 1 - delta0
        const double delta = tag ? delta1 : delta0, comp = tag ? delta0 : delta1;
        double u;
        if (R >= N) u = 1.0;
        else if (R <= 0) u = -expm1((tag ? log1p(-comp) : log(delta)) / (double)N);
        else u = cp_upper_group<L>(R, N, delta, comp, tag ? -z0 : z0, l, mask);
        __syncwarp(mask);
        if (l == 0) {
            u0s[h] = u;
            keys[h] = kEmptyKey;   // the table is empty again for the next call
        }
    }
}

__global__ void __launch_bounds__(kCpThreads, kCpBlocksPerSM) k_cp_solve(unsigned long long* __restrict__ keys,
                                                         const uint32_t* __restrict__ list,
                                                         const int32_t* __restrict__ n_keys, double delta0,
                                                         double delta1, float z0, double* __restrict__ u0s)
{
    pdl_entry();
    const int n = *n_keys;
    if (n <= kCpManyKeys) cp_solve_keys<8>(keys, list, n, delta0, delta1, z0, u0s);
    else cp_solve_keys<2>(keys, list, n, delta0, delta1, z0, u0s);
}

// Upper: u0 = Clopper-Pearson upper bound of R / K, bound = optimised tile
// Tilt-Bound.  LOWER (Rem. extension-lower): u0 = lower Clopper-Pearson bound
// l (P(Binom(K, l) >= R) = delta), bound = 1 - U_tile(1 - l) = -expm1(log U_tile).
// 1 - l enters as log(1 - l): for R <= K/2 l is the upper solve for R - 1 at
// 1 - delta and log(1 - l) = log1p(-l); for R > K/2 (l near 1) 1 - l is the
// upper solve for the K - R failures at delta (binomial symmetry), taken
// directly so that its digits are not lost to the subtraction.
template <int D, bool LOWER, typename Obj, typename Cp>
__device__ __forceinline__ void bound_of(const Obj& G, int64_t Ri, int64_t Ki, double delta, Cp cp, double* u_out,
                                         double* b_out, double* q_out)
{
    if (LOWER) {
        double l, la;
        if (2 * Ri > Ki) {
            const double ap = cp(Ki - Ri, delta);
            l = Ri == Ki ? exp(log(delta) / (double)Ki) : 1.0 - ap;   // l^K = delta when every trial rejects
            la = log(ap);
        } else if (Ri <= 0) {
            l = 0.0;
            la = 0.0;
        } else {
            l = cp(Ri - 1, 1.0 - delta);
            la = log1p(-l);
        }
        const double lb = tilt_bound_log_la<D>(G, la, q_out);
        *u_out = l;
        *b_out = (lb >= 0.0) ? 0.0 : -expm1(lb);
        return;
    }
    const double u = cp(Ri, delta);
    *u_out = u;
    *b_out = exp(tilt_bound_log<D>(G, u, q_out));
}

// Plain form: one thread a tile, FP64 throughout, its own Clopper-Pearson solve.
template <int D, bool LOWER>
__global__ void __launch_bounds__(128) k_bounds_plain(TileArgs T, int32_t n_max, const int64_t* __restrict__ R,
                                                      double delta, double* __restrict__ u0,
                                                      double* __restrict__ bound, double* __restrict__ qstar,
                                                      int32_t* __restrict__ err)
{
    pdl_entry();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= T.n_tiles) return;
    ArmGeom G[D];
    double u = NAN, b = NAN, q = NAN;
    if (load_tile<D>(T, i, (double)n_max, G, err)) {
        const int64_t Ki = T.K[i];
        bound_of<D, LOWER>((const ArmGeom*)G, R[i], Ki, delta,
                           [&](int64_t r, double dl) { return cp_upper_plain(r, Ki, dl); }, &u, &b, &q);
    }
    if (u0) u0[i] = u;
    if (bound) bound[i] = b;
    if (qstar) qstar[i] = q;
}

// A group of NL lanes a tile (see LaneTilt).  slot: each tile's entry of the
// Clopper-Pearson memo, whose values are u0s (every key it needs is there: the
// table holds at least two slots a tile).
template <int D, bool SPLIT, bool LOWER>
__global__ void __launch_bounds__(64) k_bounds(TileArgs T, int32_t n_max, const int64_t* __restrict__ R, double delta,
                                               double* __restrict__ u0, double* __restrict__ bound,
                                               double* __restrict__ qstar, int32_t* __restrict__ err,
                                               const int32_t* __restrict__ slot, const double* __restrict__ u0s,
                                               const double* __restrict__ geom, int32_t* __restrict__ nkeys_reset)
{
    pdl_entry();
    constexpr int NL = LaneTilt<D, SPLIT>::NL;
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, i = t / NL;
    const int l = (int)(t % NL);
    if (i >= T.n_tiles) return;
    // k_cp_solve has read the key count (it ran before this kernel): zero it for the next call
    if (t == 0 && nkeys_reset) *nkeys_reset = 0;
    LaneTilt<D, SPLIT> G;
    double u = NAN, b = NAN, q = NAN;
    if (load_lane(T, i, l, (double)n_max, G, err, geom, nullptr)) {
        const int64_t Ki = T.K[i];
        const int32_t sl = slot ? slot[i] : -1;
        bound_of<D, LOWER>(G, R[i], Ki, delta,
                           [&](int64_t, double) { return sl >= 0 ? u0s[sl] : NAN; }, &u, &b, &q);
    }
    if (l != 0) return;
    if (u0) u0[i] = u;
    if (bound) bound[i] = b;
    if (qstar) qstar[i] = q;
}

__device__ __forceinline__ void store_alpha(double ap, int32_t K, int64_t i, double* __restrict__ aprime,
                                            int32_t* __restrict__ ksel)
{
    if (aprime) aprime[i] = ap;
    double kf = floor(((double)K + 1.0) * ap);
    if (kf > (double)K) kf = (double)K;
    if (ksel) ksel[i] = ap == ap ? (int32_t)kf : 0;
}

template <int D>
__global__ void __launch_bounds__(128) k_alpha_prime_plain(TileArgs T, int32_t n_max, double alpha,
                                                           double* __restrict__ aprime, int32_t* __restrict__ ksel,
                                                           int32_t* __restrict__ err)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= T.n_tiles) return;
    ArmGeom G[D];
    double q, ap = NAN;
    if (load_tile<D>(T, i, (double)n_max, G, err)) ap = exp(alpha_prime_log<D>((const ArmGeom*)G, alpha, &q));
    store_alpha(ap, T.K[i], i, aprime, ksel);
}

template <int D, bool SPLIT>
__global__ void __launch_bounds__(64) k_alpha_prime(TileArgs T, int32_t n_max, double alpha,
                                                    double* __restrict__ aprime, int32_t* __restrict__ ksel,
                                                    int32_t* __restrict__ err, double* __restrict__ geom)
{
    constexpr int NL = LaneTilt<D, SPLIT>::NL;
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, i = t / NL;
    const int l = (int)(t % NL);
    if (i >= T.n_tiles) return;
    LaneTilt<D, SPLIT> G;
    double q, ap = NAN;
    if (load_lane(T, i, l, (double)n_max, G, err, (const double*)nullptr, geom))
        ap = exp(alpha_prime_log<D>(G, alpha, &q));
    if (l == 0) store_alpha(ap, T.K[i], i, aprime, ksel);
}

// min over v[0..n): each block folds its stretch on integer keys (ALU, not the
// FP64 pipe), one atomicMin per block into *key (set to all ones before the
// launch), and the last block to finish (a ticket counter, no waiting) writes
// the decoded minimum and resets the ticket.
__global__ void __launch_bounds__(256) k_min(const double* __restrict__ v, int64_t n, double* __restrict__ out,
                                             unsigned long long* __restrict__ key, unsigned int* __restrict__ ticket)
{
    pdl_entry();
    __shared__ unsigned long long red[8];
    __shared__ bool last;
    unsigned long long m = ~0ull;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        m = min(m, order_key(v[i]));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = min(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < (int)(blockDim.x >> 5); ++w) m = min(m, red[w]);
        atomicMin(key, m);
        __threadfence();
        last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (last && threadIdx.x == 0) {
        __threadfence();
        const unsigned long long k = atomicAdd(key, 0ull);
        *out = (k == ~0ull) ? INFINITY : order_unkey(k);
        *key = ~0ull;   // reset for the next launch
        *ticket = 0u;
    }
}

__global__ void k_backward(int64_t n, int32_t d, const double* __restrict__ g, const double* __restrict__ score,
                           const int32_t* __restrict__ K, double* __restrict__ out)
{
    pdl_entry();
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n * d) return;
    const int64_t i = j / d;
    out[j] = g[i] * score[j] / (double)K[i];
}

}  // namespace

// z with Phi(z) = p (0 < p < 1), to ~1e-7: the start of the Clopper-Pearson solves.
static double normal_quantile(double p)
{
    double lo = -40.0, hi = 40.0;
    for (int it = 0; it < 60; ++it) {
        const double mid = 0.5 * (lo + hi);
        if (0.5 * erfc(-mid * 0.70710678118654752440) < p) lo = mid;
        else hi = mid;
    }
    return 0.5 * (lo + hi);
}

// Lanes a tile: two per arm while the tiles give every sub-partition at most
// kSplitWarps warps (what counts is the latency of one tile's chain), one per arm
// beyond (the FP64 pipe is full and the signs' common work is done once).  alpha' /
// bound, against one thread a tile: one arm, 64 tiles 31 / 38 -> 21 / 17 us; two
// arms, 1,891 tiles, band 67 + 58 -> 26 + 21; four arms, 6,036 tiles 183 -> 58
// (bound); two arms, 32,896 tiles 75 / 62 -> 68 / 48 (92 / 72 with the signs split);
// 2^18 tiles 557 / 411 -> 538 / 341; four arms, 59,992 tiles 261 / 219 -> 257 / 171.
inline bool split_signs(const cse_ctx* c, const TileArgs& T)
{
    return T.n_tiles * 2 * T.d <= (int64_t)c->num_sms * 4 * 32 * kSplitWarps;
}

template <int D, bool SPLIT>
void launch_bounds_s(cse_ctx* c, const TileArgs& T, const int64_t* R, double delta, bool lower, double* u0,
                     double* bound, double* qstar, const int32_t* slot, const double* geom, cudaStream_t s)
{
    constexpr int NL = LaneTilt<D, SPLIT>::NL;
    const unsigned blocks = (unsigned)((T.n_tiles * NL + 63) / 64);
    int32_t* nk = slot ? c->cp_nkeys : nullptr;
    if (lower)
        cse_launch(c->pdl, k_bounds<D, SPLIT, true>, dim3(blocks), dim3(64), 0, s, T, c->D.n_max, R, delta, u0, bound,
                   qstar, c->err, slot, c->cp_val, geom, nk);
    else
        cse_launch(c->pdl, k_bounds<D, SPLIT, false>, dim3(blocks), dim3(64), 0, s, T, c->D.n_max, R, delta, u0, bound,
                   qstar, c->err, slot, c->cp_val, geom, nk);
}

template <int D>
void launch_bounds_d(cse_ctx* c, const TileArgs& T, const int64_t* R, double delta, bool lower, double* u0,
                     double* bound, double* qstar, const int32_t* slot, const double* geom, cudaStream_t s)
{
    if (c->plain) {
        const unsigned blocks = (unsigned)((T.n_tiles + 127) / 128);
        if (lower)
            cse_launch(c->pdl, k_bounds_plain<D, true>, dim3(blocks), dim3(128), 0, s, T, c->D.n_max, R, delta, u0,
                       bound, qstar, c->err);
        else
            cse_launch(c->pdl, k_bounds_plain<D, false>, dim3(blocks), dim3(128), 0, s, T, c->D.n_max, R, delta, u0,
                       bound, qstar, c->err);
    } else if (split_signs(c, T)) {
        launch_bounds_s<D, true>(c, T, R, delta, lower, u0, bound, qstar, slot, geom, s);
    } else {
        launch_bounds_s<D, false>(c, T, R, delta, lower, u0, bound, qstar, slot, geom, s);
    }
}

template <int D, bool SPLIT>
void launch_alpha_s(cse_ctx* c, const TileArgs& T, double alpha, double* ap, int32_t* ksel, double* geom,
                    cudaStream_t s)
{
    constexpr int NL = LaneTilt<D, SPLIT>::NL;
    k_alpha_prime<D, SPLIT><<<(unsigned)((T.n_tiles * NL + 63) / 64), 64, 0, s>>>(T, c->D.n_max, alpha, ap, ksel,
                                                                                c->err, geom);
}

template <int D>
void launch_alpha_d(cse_ctx* c, const TileArgs& T, double alpha, double* ap, int32_t* ksel, double* geom,
                    cudaStream_t s)
{
    if (c->plain)
        k_alpha_prime_plain<D><<<(unsigned)((T.n_tiles + 127) / 128), 128, 0, s>>>(T, c->D.n_max, alpha, ap, ksel,
                                                                                 c->err);
    else if (split_signs(c, T))
        launch_alpha_s<D, true>(c, T, alpha, ap, ksel, geom, s);
    else
        launch_alpha_s<D, false>(c, T, alpha, ap, ksel, geom, s);
}

int cse_launch_bounds(cse_ctx* c, const TileArgs& T, const int64_t* R, double delta, bool lower, double* u0,
                      double* bound, double* qstar, cudaStream_t s, const double* geom, bool marked)
{
    const unsigned blocks = (unsigned)((T.n_tiles + 127) / 128);
    const int32_t* slot = nullptr;
    if (!c->plain && c->cp_cap >= 2 * (uint64_t)T.n_tiles) {
        // one Clopper-Pearson solve per distinct (R, K)
        // the key table is empty and the key count zero on entry: k_cp_solve empties
        // the slots it solves and k_bounds zeroes the count (both set at allocation)
        cse_prof_begin(c, KID_CP, s);
        if (!(marked && !lower)) {
            cse_launch(c->pdl, k_cp_mark, dim3(blocks), dim3(128), 0, s, T.n_tiles, R, T.K, c->cp_key,
                       (uint32_t)c->cp_cap, c->cp_slot, c->cp_list, c->cp_nkeys, lower);
            c->launches += 1;
        }
        // a group of 8 lanes per key at most, spread over the SMs
        const int64_t full = (int64_t)c->num_sms * kCpBlocksPerSM;
        const int64_t blocks_cp = std::min<int64_t>(full, (T.n_tiles + kCpThreads / 32 - 1) / (kCpThreads / 32));
        cse_launch(c->pdl, k_cp_solve, dim3((unsigned)blocks_cp), dim3(kCpThreads), 0, s, c->cp_key, c->cp_list,
                   c->cp_nkeys, delta, 1.0 - delta, (float)normal_quantile(1.0 - delta), c->cp_val);
        cse_prof_end(c, s);
        c->launches += 1;
        slot = c->cp_slot;
    }
    cse_prof_begin(c, KID_BOUNDS, s);
    switch (T.d) {
    case 1: launch_bounds_d<1>(c, T, R, delta, lower, u0, bound, qstar, slot, geom, s); break;
    case 2: launch_bounds_d<2>(c, T, R, delta, lower, u0, bound, qstar, slot, geom, s); break;
    case 4: launch_bounds_d<4>(c, T, R, delta, lower, u0, bound, qstar, slot, geom, s); break;
    default: return CSE_UNSUPPORTED_DESIGN;
    }
    cse_prof_end(c, s);
    c->launches += 1;
    return cudaGetLastError() == cudaSuccess ? CSE_OK : CSE_CUDA_ERROR;
}

// k_alpha_prime runs beside the table kernels (second stream) and uses no
// shared memory.  Left to itself its SMs take a small shared-memory carveout,
// and a table kernel's blocks (16 KB of shared memory each) then wait on every
// SM until the alpha' blocks there have finished, as an SM changes its
// carveout only when idle.  Asking for the largest carveout lets both run.
int cse_bound_set_attrs()
{
    auto most = [](auto kern) {
        return cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    };
    cudaError_t e = most(k_alpha_prime<1, false>);
    if (e == cudaSuccess) e = most(k_alpha_prime<1, true>);
    if (e == cudaSuccess) e = most(k_alpha_prime<2, false>);
    if (e == cudaSuccess) e = most(k_alpha_prime<2, true>);
    if (e == cudaSuccess) e = most(k_alpha_prime<4, false>);
    if (e == cudaSuccess) e = most(k_alpha_prime<4, true>);
    if (e == cudaSuccess) e = most(k_alpha_prime_plain<1>);
    if (e == cudaSuccess) e = most(k_alpha_prime_plain<2>);
    if (e == cudaSuccess) e = most(k_alpha_prime_plain<4>);
    return e == cudaSuccess ? CSE_OK : CSE_CUDA_ERROR;
}

int cse_launch_alpha_prime(cse_ctx* c, const TileArgs& T, double alpha, double* aprime_out,
                           int32_t* ksel, cudaStream_t s, double* geom)
{
    cse_prof_begin(c, KID_ALPHA_PRIME, s);
    switch (T.d) {
    case 1: launch_alpha_d<1>(c, T, alpha, aprime_out, ksel, geom, s); break;
    case 2: launch_alpha_d<2>(c, T, alpha, aprime_out, ksel, geom, s); break;
    case 4: launch_alpha_d<4>(c, T, alpha, aprime_out, ksel, geom, s); break;
    default: return CSE_UNSUPPORTED_DESIGN;
    }
    cse_prof_end(c, s);
    c->launches += 1;
    return cudaGetLastError() == cudaSuccess ? CSE_OK : CSE_CUDA_ERROR;
}

int cse_launch_min(cse_ctx* c, const double* lam_tile, int64_t n, double* out, cudaStream_t s)
{
    int64_t blocks = (n + 255) / 256;
    if (blocks > 2 * (int64_t)c->num_sms) blocks = 2 * (int64_t)c->num_sms;
    if (blocks < 1) blocks = 1;
    // min_key is all ones and the ticket zero on entry (set at creation, restored by the last block)
    cse_prof_begin(c, KID_MIN, s);
    cse_launch(c->pdl, k_min, dim3((unsigned)blocks), dim3(256), 0, s, lam_tile, n, out, c->min_key, c->min_ticket);
    cse_prof_end(c, s);
    c->launches += 1;
    return cudaGetLastError() == cudaSuccess ? CSE_OK : CSE_CUDA_ERROR;
}

int cse_launch_backward(int64_t n, int32_t d, const double* g, const double* score, const int32_t* K,
                        double* out, cudaStream_t s)
{
    const int64_t tot = n * d;
    if (tot == 0) return CSE_OK;
    cse_launch(true, k_backward, dim3((unsigned)((tot + 255) / 256)), dim3(256), 0, s, n, d, g, score, K, out);
    return cudaGetLastError() == cudaSuccess ? CSE_OK : CSE_CUDA_ERROR;
}
