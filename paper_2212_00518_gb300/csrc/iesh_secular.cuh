// iesh_secular.cuh -- roots of the secular equation of an arrowhead matrix
// (internal to the library), templated on the arithmetic type.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "iesh_common.cuh"

namespace iesh {

template <class R>
struct Roundoff;
template <>
struct Roundoff<double> {
    static constexpr double u = 1.1102230246251565e-16;  // 2^-53
    static constexpr double tiny = 1e-300;
};
template <>
struct Roundoff<float> {
    static constexpr float u = 5.9604645e-08f;  // 2^-24
    static constexpr float tiny = 1e-37f;
};


// Reciprocal of a pole distance.  FP64: the PTX approximate reciprocal
// r0 = 1/d (1 + e'), e = 1 - d r0, refined by the first terms of the
// geometric series 1/d = r0 / (1 - e) = r0 (1 + e + e^2 + ...); with the
// estimate's relative error |e| far below 2^-18 the truncated e^3 term is
// below 2^-54, so the result is within about an ulp of 1/d.  Three FMAs
// replace a full division in the secular sums, which are the FP64-bound
// part of the eigen solve, in the couplings d_jk and in the iteration's
// safeguarded proposals.  Inputs are pole distances, eigenvalue gaps and
// proposal denominators; a zero or subnormal input (the estimate flushes
// subnormals to zero) gives a non-finite result, which the callers either
// cannot produce or reject.
template <class R>
__device__ __forceinline__ R pole_recip(R d)
{
    return R(1) / d;
}
template <>
__device__ __forceinline__ double pole_recip<double>(double d)
{
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(d));
    const double e = fma(-d, r, 1.0);
    return fma(r, fma(e, e, e), r);
}

// FP32: the approximate reciprocal (1 ulp) and one Newton step, in place of a
// correctly rounded division's eight or so instructions.
template <>
__device__ __forceinline__ float pole_recip<float>(float d)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(d));
    return fmaf(r, fmaf(-d, r, 1.0f), r);
}

// Double-float numbers (hi + lo, two FP32 values, about 48 significant bits)
// for the secular sums of the mixed-precision path: the FP32 pipe is 64x
// wider than the FP64 pipe on this part.  Error-free transformations:
// Knuth's TwoSum, Dekker's Fast2Sum (|a| >= |b|) and the FMA product error.
struct dfl {
    float hi, lo;
};
__device__ __forceinline__ dfl dfl_two_sum(float a, float b)
{
    const float s = a + b, bb = s - a;
    return {s, (a - (s - bb)) + (b - bb)};
}
__device__ __forceinline__ dfl dfl_fast_two_sum(float a, float b)
{
    const float s = a + b;
    return {s, b - (s - a)};
}
// a + b with an error of a few units of 2^-46 (|a| + |b|)
__device__ __forceinline__ dfl dfl_add(dfl a, dfl b)
{
    dfl s = dfl_two_sum(a.hi, b.hi);
    s.lo += a.lo + b.lo;
    return dfl_fast_two_sum(s.hi, s.lo);
}
__device__ __forceinline__ dfl dfl_mul(dfl a, dfl b)
{
    const float p = a.hi * b.hi;
    float e = fmaf(a.hi, b.hi, -p);
    e = fmaf(a.hi, b.lo, e);
    e = fmaf(a.lo, b.hi, e);
    return dfl_fast_two_sum(p, e);
}
// 1/a: the FP32 reciprocal estimate r0 (1 ulp) corrected by r0 (e + e^2), e =
// 1 - a r0
__device__ __forceinline__ dfl dfl_rcp(dfl a)
{
    float r0;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r0) : "f"(a.hi));
    float e = fmaf(-a.hi, r0, 1.0f);
    e = fmaf(-a.lo, r0, e);
    return dfl_fast_two_sum(r0, r0 * fmaf(e, e, e));
}
// a += b with the low parts summed on their own (renormalised once, by
// dfl_value or dfl_add, at the end of a sum)
__device__ __forceinline__ void dfl_acc(dfl &a, dfl b)
{
    const dfl s = dfl_two_sum(a.hi, b.hi);
    a.hi = s.hi;
    a.lo += s.lo + b.lo;
}
__device__ __forceinline__ dfl dfl_from(double x)
{
    const float h = (float)x;
    return {h, (float)(x - (double)h)};
}
__device__ __forceinline__ double dfl_value(dfl a) { return (double)a.hi + (double)a.lo; }

// Pole data of the secular sums.  diff (optional): FP64 table of the pole
// differences diff[k M + o] = eps_o - eps_k; ddf, z2df (double-float mode):
// the same differences and z_k^2 as double-float pairs.
// Two-orbital double-float mode (EV_TWO_DF): the M poles are nb bath poles
// with one extra pole h_- inserted at index hpos (hpos < 0: none); ddf is
// the bath table [nb][nb], hdf[k] = h_- - eps_k as double-float pairs, and
// z2df the weights of all M poles in sorted order.
// Nested double-float mode (EV_NESTED): the M poles are roots mu_k = eps_{ob[k]}
// + tau_k of an inner arrowhead over nb bath poles; ddf is the bath table
// [nb][nb], hdf[k] = tau_k as a double-float pair and ob[k] its bath pole,
// so mu_o - mu_k = (eps_{ob[o]} - eps_{ob[k]}) + (tau_o - tau_k) keeps its
// relative accuracy however close the two roots are.
// EV_POLE_DF and EV_POLE_F32 (starting stages): the poles themselves as
// double-float pairs in hdf; the differences are formed per term.
template <class R>
struct Poles {
    int M;
    const R *__restrict__ eps, *__restrict__ z2, *__restrict__ diff;
    const float2 *__restrict__ ddf, *__restrict__ z2df;
    int nb, hpos;
    R hm;
    const float2 *__restrict__ hdf;
    const int *__restrict__ ob;
};

// Evaluation modes of the secular sums: EV_PLAIN (eps_o - eps_k formed per
// term), EV_TABLE (FP64 table), EV_DFLOAT (double-float sums on the FP32
// pipe; the origin term and the assembly of g stay FP64), EV_TWO_DF,
// EV_NESTED and EV_POLE_DF (double-float, see Poles), EV_POLE_F32 (FP32 sums).
enum { EV_PLAIN = 0, EV_TABLE = 1, EV_DFLOAT = 2, EV_TWO_DF = 3, EV_NESTED = 4, EV_POLE_DF = 5, EV_POLE_F32 = 6 };
__host__ __device__ constexpr bool ev_is_df(int ev) { return ev == EV_DFLOAT || ev == EV_TWO_DF || ev == EV_NESTED || ev == EV_POLE_DF; }

// mu_o - mu_k + td for the nested poles (EV_NESTED), in double-float.
template <class R>
__device__ __forceinline__ dfl nested_gap(const Poles<R> &P, int o, int k, dfl td)
{
    const float2 e = P.ddf[(size_t)P.ob[k] * P.nb + P.ob[o]];  // eps_ob[o] - eps_ob[k]
    const float2 to = P.hdf[o], tk = P.hdf[k];
    const dfl dtau = dfl_add({to.x, to.y}, {-tk.x, -tk.y});
    return dfl_add(dfl_add({e.x, e.y}, dtau), td);
}

// ============================================================= eigenpairs
// The one-electron Hamiltonian of Sec. II B is an arrowhead matrix:
// diag(h, eps_1..eps_M) bordered by z_k = V_k(x).  Its eigenvalues are the
// roots of g(lam) = lam - h - sum_k z_k^2 / (lam - eps_k), one in each gap
// of the sorted poles, and the eigenvector of root lam has impurity
// component q0 = 1 / sqrt(g'(lam)) (chosen > 0) and bath components
// z_k q0 / (lam - eps_k).  Each root is found in the shifted variable
// tau = lam - eps_o relative to its nearer pole o, so lam - eps_k =
// (eps_o - eps_k) + tau keeps full relative accuracy.
// gp = gp_rest + the origin's share; rt = 1 / tau; s3 = sum over k != o of
// z_k^2 / (lam - eps_k)^3 (FP32, where the mode forms it), so g'' = -2 (s3 +
// (gp - gp_rest) rt): the origin's share, of order gap^3 / z^4, leaves FP32's
// range once z^2 is below about 10^-21 (a coupling that decays to 10^-8 of its
// value) and is formed in R.  sabs = the scale of g's rounding error.
template <class R>
struct Sec {
    R g, gp, gp_rest, qo, rt, sabs;
    float s3;
};

// With ABS the sum of |z_k^2 / (lam - eps_k)| over k != o is accumulated into
// e.sabs; without it e.sabs is left at zero for the caller to fill in (the
// FP32 and double-float modes form it in FP32 along the way).  EV selects how
// the sums over k != o are formed (see EV_*); the terms k != o have |lam -
// eps_k| >= half a pole gap, so their double-float range is safe.
template <class R, bool ABS, int EV>
__device__ __forceinline__ Sec<R> sec_eval(const Poles<R> &P, int o, R tau, R eomh)
{
    const int M = P.M;
    R s1 = 0, s2 = 0, sa = 0;
    float s3 = 0.f;
    if constexpr (ev_is_df(EV)) {
        // two accumulator sets (even and odd poles), added at the end: the
        // double-float additions are a serial chain, two chains run at once
        const dfl td = dfl_from((double)tau);
        dfl d1[2] = {{0.f, 0.f}, {0.f, 0.f}}, d2[2] = {{0.f, 0.f}, {0.f, 0.f}};
        float da = 0.f;
        const bool oh = EV == EV_TWO_DF && o == P.hpos;
        const int ob = EV != EV_TWO_DF ? 0 : (oh ? 0 : ((P.hpos >= 0 && o > P.hpos) ? o - 1 : o));
        const float2 po = EV == EV_POLE_DF ? P.hdf[o] : make_float2(0.f, 0.f);
        auto term = [&](int k, int h) {
            int q = k;  // index of the weight
            dfl x;      // lam - eps_k
            if constexpr (EV == EV_DFLOAT) {
                const float2 dk = P.ddf[(size_t)k * M + o];
                x = dfl_add({dk.x, dk.y}, td);
            } else if constexpr (EV == EV_TWO_DF) {
                q = (P.hpos >= 0 && k >= P.hpos) ? k + 1 : k;
                const float2 dk = oh ? P.hdf[k] : P.ddf[(size_t)k * P.nb + ob];
                x = dfl_add({dk.x, dk.y}, td);
            } else if constexpr (EV == EV_NESTED) {
                if (k == o) return;
                x = nested_gap(P, o, k, td);
            } else {
                const float2 pk = P.hdf[k];
                x = dfl_add(dfl_add({po.x, po.y}, {-pk.x, -pk.y}), td);
            }
            const float2 zk = P.z2df[q];
            const dfl r = dfl_rcp(x);
            const dfl v = dfl_mul({zk.x, zk.y}, r);
            if (q != o) {
                const dfl w = dfl_mul(v, r);
                dfl_acc(d1[h], v);
                dfl_acc(d2[h], w);
                da += fabsf(v.hi);
                s3 = fmaf(w.hi, r.hi, s3);
            }
        };
        const int nk = EV == EV_TWO_DF ? P.nb : M;
        int k = 0;
        for (; k + 1 < nk; k += 2) {
            term(k, 0);
            term(k + 1, 1);
        }
        if (k < nk) term(k, 0);
        s1 = (R)dfl_value(dfl_add(d1[0], d1[1]));
        s2 = (R)dfl_value(dfl_add(d2[0], d2[1]));
        sa = (R)da;
        if constexpr (EV == EV_TWO_DF)  // the h_- term in R
            if (P.hpos >= 0 && !oh) {
                const R r = pole_recip<R>((P.eps[o] - P.hm) + tau);
                const R qv = P.z2[P.hpos] * r, wv = qv * r;
                s1 += qv;
                s2 += wv;
                sa += fabs(qv);
                s3 = fmaf((float)wv, (float)r, s3);
            }
    } else if constexpr (EV == EV_POLE_F32) {
        const float tf = (float)tau, po = P.hdf[o].x;
        float f1 = 0.f, f2 = 0.f, fa = 0.f;
#pragma unroll 4
        for (int k = 0; k < M; ++k) {
            // (the origin's distance may be below FP32's range)
            const float r = k != o ? pole_recip<float>((po - P.hdf[k].x) + tf) : 0.f;
            const float v = P.z2df[k].x * r, w = v * r;
            f1 += v;
            f2 += w;
            fa += fabsf(v);
            s3 = fmaf(w, r, s3);
        }
        s1 = (R)f1, s2 = (R)f2, sa = (R)fa;
    } else {
        const R eo = P.eps[o];
#pragma unroll 4
        for (int k = 0; k < M; ++k) {
            const R dko = EV == EV_TABLE ? P.diff[(size_t)k * M + o] : (eo - P.eps[k]);
            const R r = pole_recip<R>(dko + tau);
            const R q = P.z2[k] * r;
            if (k != o) {
                s1 += q;
                if constexpr (sizeof(R) == 4) {
                    const R w = q * r;
                    s2 += w;
                    s3 = fmaf(w, r, s3);
                    sa += fabs(q);
                } else {
                    s2 = fma(q, r, s2);
                    if (ABS) sa += fabs(q);
                }
            }
        }
    }
    // origin term: one reciprocal of tau (never zero or subnormal: the
    // iteration keeps it strictly inside its bracket) serves both quotients
    const R rt = pole_recip<R>(tau);
    const R qo = P.z2[o] * rt, wo = qo * rt;
    Sec<R> e;
    e.g = (eomh + tau) - s1 - qo;
    e.gp_rest = R(1) + s2;
    e.gp = e.gp_rest + wo;
    e.qo = qo;
    e.rt = rt;
    e.sabs = sa;
    e.s3 = s3;
    return e;
}

// One step of the fixed-weight iteration as a correction delta to tau: the
// origin pole (weight s at distance -tau) is kept exactly and the rest of g
// is modelled by one more pole at distance -tp (tp = tau -+ D, the other end
// of the gap; kinds 0 and 1) or by a linear term for the two outermost roots
// (kind 2: below all poles, kind 3: above), matched in value and slope:
//   kinds 0, 1: A d^2 + B d + G = 0, A = g + s/tau + ee tp,
//               B = g (tau + tp) + s tp/tau + ee tp tau, G = g tau tp;
//   kinds 2, 3: A = ee, B = g + ee tau + s/tau, G = g tau,
// ee the slope of the rest.  The model root in the gap is the one where the
// quadratic decreases (kind 3: increases).  A correction needs no more than
// FP32: its relative error, 10^-6, only enters the next iterate's error
// (FP64 instructions on this iteration's serial path cost more than they
// save: a warp's takes 64 cycles of its scheduler's FP64 pipe).
template <class T>
__device__ __forceinline__ T sec_step(int kind, T g, T ee, T s, T tau, T tp)
{
    const T srt = s * pole_recip<T>(tau);
    T A, B, G;
    if (kind <= 1) {
        A = g + srt + ee * tp;
        B = g * (tau + tp) + tp * (srt + ee * tau);
        G = g * tau * tp;
    } else {
        A = ee;
        B = g + ee * tau + srt;
        G = g * tau;
    }
    const T rb = pole_recip<T>(B), a = A * rb, b = G * rb;
    const T sq = sqrt(fmax(T(1) - T(4) * a * b, T(0)));
    if ((B < T(0)) != (kind == 3)) return T(-2) * b * pole_recip<T>(T(1) + sq);
    return (T(1) + sq) * T(-0.5) * pole_recip<T>(a);
}

// The step at tau, in FP32 where its quantities are inside FP32's range.
template <class R>
__device__ __forceinline__ R sec_delta(int kind, const Sec<R> &e, R s, R tau, R D)
{
    if constexpr (sizeof(R) == 8) {
        const float tf = (float)tau, sf = (float)s, ef = (float)e.gp_rest, df = (float)D;
        if (fabsf(tf) > 1e-18f && sf > 1e-25f && ef < 1e18f)
            return (R)sec_step<float>(kind, (float)e.g, ef, sf, tf, kind == 0 ? tf - df : tf + df);
    }
    return sec_step<R>(kind, e.g, e.gp_rest, s, tau, kind == 0 ? tau - D : tau + D);
}

// A correction this small against the distance to the nearer end of the gap
// ends the iteration: tau takes it, and gp its first-order change g'' delta
// (what is left out is of second order, below the mode's rounding; the change
// is at most 2 limit gp, so a larger one is an overflow).  FP32: 2^-13;
// double-float sums: 2^-23; the last FP64 evaluation of a staged solve: 2^-31.
template <class R>
__device__ __forceinline__ bool sec_accept(int kind, R D, R limit, R delta, R &tau, Sec<R> &e)
{
    const R tp = kind == 0 ? tau - D : tau + D;
    const R dist = kind <= 1 ? fmin(fabs(tau), fabs(tp)) : fabs(tau);
    if (!(fabs(delta) <= limit * dist)) return false;
    const R change = R(-2) * ((e.gp - e.gp_rest) * (delta * e.rt) + (R)(e.s3 * (float)delta));
    if (!(fabs(change) <= R(1e-3) * e.gp)) return false;
    e.gp += change;
    tau += delta;
    return true;
}

// Safeguarded iteration for one root in the shifted variable tau about the
// origin pole o; [lo, hi] brackets the sign change.  On return e is evaluated
// at tau (or corrected to it).
template <class R, int EV>
__device__ bool sec_iterate(const Poles<R> &P, R h, int o, int kind, R D, R &lo, R &hi, R &tau,
                            Sec<R> &e, bool have, R ulps = R(8))
{
    // rounding unit of the sums: 2^-44 covers the double-float sums
    constexpr bool kF32 = sizeof(R) == 4 || EV == EV_POLE_F32;
    // (a stage before another one is run down to its corrections' limit)
    const R u = ev_is_df(EV) ? R(5.684341886080802e-14) : (kF32 ? R(Roundoff<float>::u) : R(Roundoff<R>::u));
    const R limit = kF32 ? R(1.2207031e-4) : (ev_is_df(EV) ? R(1.1920929e-7) : R(0));
    const R eomh = P.eps[o] - h;
    const R s = P.z2[o];
    // the non-origin part of the error scale varies slowly with tau (those
    // poles are at least half a gap away): take it from the first evaluation
    if (!have) e = sec_eval<R, true, EV>(P, o, tau, eomh);
    const R sa_rest = e.sabs;
    for (int it = 0; it < 80; ++it) {
        if (it) e = sec_eval<R, false, EV>(P, o, tau, eomh);
        e.sabs = sa_rest + fabs(e.qo) + fabs(eomh) + fabs(tau);
        if (fabs(e.g) <= ulps * u * e.sabs) return true;
        if (e.g < R(0)) lo = tau;
        else hi = tau;
        const R delta = sec_delta<R>(kind, e, s, tau, D);
        R tn = tau + delta;
        const bool in = tn > lo && tn < hi;
        if (limit > R(0) && in && sec_accept<R>(kind, D, limit, delta, tau, e)) return true;
        if (!in) tn = R(0.5) * (lo + hi);
        const bool tiny = fabs(tn - tau) <= R(2) * u * fabs(tn);
        tau = tn;
        if (tiny) {
            e = sec_eval<R, false, EV>(P, o, tau, eomh);
            return true;
        }
    }
    e = sec_eval<R, false, EV>(P, o, tau, eomh);
    return false;
}

// Root r (0..M) of the secular equation, lam and q0 = 1/sqrt(g'(lam)), and
// optionally its origin pole o and offset tau = lam - eps_o (unrounded).
// Cold start: the sign of g at the middle of the pole gap picks the nearer
// pole as origin and the half-gap as bracket.  Warm start (previous root
// `guess`, which lies in the same gap): origin = pole nearer the guess,
// bracket = the whole gap, started at the guess; if the root ends in the
// far half of the gap it is refined once more about the other pole.
// EV: how the final sums are formed (see sec_eval).  EVP, EV0 (R = double):
// cheaper sums for a staged solve -- the iteration runs with EV0 (cold
// starts only), then EVP, to their own accuracy, and EV evaluates once more
// and corrects: an FP64 term costs about 450 cycles of a scheduler (7
// instructions at 64 cycles a warp), a double-float one 55 and an FP32 one
// 12.  Where the correction is not small (a root so close to its pole or so
// sensitive that the stage before could not resolve it) EV iterates.
template <class R, int EV = EV_PLAIN, int EVP = EV, int EV0 = EVP>
__device__ void secular_root(int r, const Poles<R> &P, R h, R Z2, bool warm, R guess, R &lam, R &q0,
                             uint32_t &st, int *o_out = nullptr, R *tau_out = nullptr)
{
    const int M = P.M;
    const R *__restrict__ eps = P.eps;
    int o, kind;
    R lo, hi, D = 0, tau;
    Sec<R> e;
    bool have = false, conv, cold = true;
    if (r > 0 && r < M) {
        const int L = r - 1;
        D = eps[r] - eps[L];
        if (warm && guess > eps[L] && guess < eps[r]) {
            cold = false;
            if (guess - eps[L] <= eps[r] - guess) {
                o = L; kind = 0; lo = 0; hi = D; tau = guess - eps[L];
            } else {
                o = r; kind = 1; lo = -D; hi = 0; tau = guess - eps[r];
            }
        } else {
            e = sec_eval<R, true, EV0>(P, L, R(0.5) * D, eps[L] - h);
            have = true;
            if (e.g >= R(0)) {
                o = L; kind = 0; lo = 0; hi = R(0.5) * D; tau = R(0.5) * D;
            } else {
                // the same sums about the other pole: the two ends' terms
                // change places
                o = r; kind = 1; lo = -R(0.5) * D; hi = 0; tau = -R(0.5) * D;
                const R rd = pole_recip<R>(tau), qr = P.z2[r] * rd, qL = e.qo;
                e.gp_rest += (e.gp - e.gp_rest) - qr * rd;
                e.sabs += fabs(qL) - fabs(qr);
                e.qo = qr;
                e.rt = rd;
            }
            // coarser sums may misjudge a root near the middle: the later
            // stages get the whole gap
            if constexpr (EV0 != EV) {
                lo = kind == 0 ? R(0) : -D;
                hi = kind == 0 ? D : R(0);
            }
        }
    } else {
        if (r == 0) {
            o = 0; kind = 2;
            const R t = h - eps[0];
            const R lb = R(0.5) * ((h + eps[0]) - sqrt(t * t + R(4) * Z2));
            lo = (lb - eps[0]) * (R(1) + R(64) * Roundoff<R>::u) - Roundoff<R>::tiny;
            hi = 0;
            tau = R(0.5) * lo;
        } else {
            o = M - 1; kind = 3;
            const R t = h - eps[M - 1];
            const R ub = R(0.5) * ((h + eps[M - 1]) + sqrt(t * t + R(4) * Z2));
            lo = 0;
            hi = (ub - eps[M - 1]) * (R(1) + R(64) * Roundoff<R>::u) + Roundoff<R>::tiny;
            tau = R(0.5) * hi;
        }
        if (warm) {
            const R tg = guess - eps[o];
            if (tg > lo && tg < hi) {
                tau = tg;
                cold = false;
            }
        }
    }
    // the bracket of a stage with coarser sums is its own: a sign decided by
    // rounding must not shut the root out of the next stage's
    if constexpr (EV0 != EVP)
        if (cold) {
            R l0 = lo, h0 = hi;
            sec_iterate<R, EV0>(P, h, o, kind, D, l0, h0, tau, e, have);
            have = false;
        }
    R lp = lo, hp = hi;
    constexpr R ulps = EVP == EV ? R(8) : R(0.25);
    conv = sec_iterate<R, EVP>(P, h, o, kind, D, lp, hp, tau, e, have, ulps);
    if constexpr (EVP == EV) lo = lp, hi = hp;
    if (!cold && kind <= 1) {
        bool moved = false;
        if (kind == 0 && tau > R(0.5) * D) {
            o = r; kind = 1; lo = fmin(lo - D, -R(0.5) * D); hi = 0; tau = tau - D;
            moved = true;
        } else if (kind == 1 && tau < -R(0.5) * D) {
            o = r - 1; kind = 0; lo = 0; hi = fmax(hi + D, R(0.5) * D); tau = tau + D;
            moved = true;
        }
        if (moved) {
            lp = lo, hp = hi;
            conv = sec_iterate<R, EVP>(P, h, o, kind, D, lp, hp, tau, e, false, ulps);
        }
    }
    if constexpr (EVP != EV) {
        const float s3 = e.s3;
        e = sec_eval<R, false, EV>(P, o, tau, eps[o] - h);
        e.s3 = s3;
        const R delta = sec_delta<R>(kind, e, P.z2[o], tau, D);
        if (!(conv && tau + delta > lo && tau + delta < hi && sec_accept<R>(kind, D, R(4.656612873077393e-10), delta, tau, e)))
            conv = sec_iterate<R, EV>(P, h, o, kind, D, lo, hi, tau, e, false);
    }
    if (!conv) st |= ST_SECULAR;
    lam = eps[o] + tau;
    if constexpr (sizeof(R) == 4) q0 = R(1) / sqrt(e.gp);
    else q0 = rsqrt(e.gp);
    if (o_out) *o_out = o;  // lam = eps[o] + tau with tau exact
    if (tau_out) *tau_out = tau;
}


}  // namespace iesh
