// iesh_hop_fx.cuh -- the determinant ratios C_m S^{-1} of the FP64 hop kernel
// (k_hop in iesh_step.cu) in 64-bit fixed point.
//
// The FP64 pipe takes 64 cycles of a scheduler per warp instruction on this
// chip, so the two substitutions of all unoccupied rows (4 (N - Ne) Ne^2 FP64
// FMAs and the quads' reductions) were 77% of the kernel.  A complex product
// of 57-bit integers is twelve 32 x 32 -> 64 multiply-adds on the integer pipe.
//
// With P S = L U, column j of S and of the rows c scaled by 2^p_j, p_j the
// exponent of 1 / U_jj (the ratios do not change), U' = U diag(2^p) and D' =
// diag U', 1 / D' with entries in [1, 2.9): x = c diag(2^p) U1^{-1} D'^{-1}
// L^{-1}, U1 = D'^{-1} U'.  So no pivot multiplies the rounding of a row, and a
// scaled electron gives the same bits.
// U1 and L are held as a = a1 2^26 + a0, |a0| <= 2^25, in the unit 2^-56 (their
// entries must be below 1.75), a row as y = y1 2^30 + y0, |y0| <= 2^29.  A sum of
// products in y's unit is
//   sum y a / 2^56 = sum y1 a1 + (sum y1 a0 + (sum y0 a1 >> 4)) >> 26;
// y0 a0, at most 1/4 of the unit per product with zero mean, is left out.  With
// column sums of |re| + |im| of U1 and L below 2^b (b <= 4, and below 15) every
// y and x must stay below 2^l, l = min(60, 62 - b): then no total exceeds 2^62
// (the first sum may wrap, only the total is used) and the others stay below
// 2^63.  A row's unit puts its largest scaled entry into [2^(l-4), 2^(l-3)); a row
// that grows past 2^l is formed again in a unit 2^3 larger, up to three times.
// The error is about 2^-56.5 of a row's largest entry, on the way or in the
// result, for b <= 2: a slot whose ratios are far below the row's others keeps
// that absolute error (10^-6 of them: 10^-10 of the slot's own, where FP64 had
// 10^-15).  What does not fit -- larger entries or sums, rows that grow further,
// numbers that are not finite -- goes to the FP64 substitution, from the saved
// factors; entries and sums are known before the first row.  Of strongly mixed
// columns (random ones, N = 101) two trajectories in three leave by their sums:
// 2.98 ms per 2048 trajectories, 1.86 ms where none does.
//
// What bounds it: half of the kernel is now the FP64 factorisation; a product
// is twelve multiply-adds and some twenty other integer instructions.  Four
// lanes per row, as in the FP64 substitution: the rows of a warp read the same
// factor entries, and 64 rows a pass fill the block.
// Measured, hop kernel per step: N = 101, Ne = 50, 4096 trajectories 7.70 ->
// 3.42 ms; N = 201, Ne = 100, 1024 trajectories 13.4 -> 7.6 ms; N = 41, Ne = 20,
// 1000 trajectories 0.36 -> 0.24 ms; two orbitals, N = 102, 1024 trajectories
// 2.14 -> 1.06 ms.  With the low products too (sixteen multiply-adds): 3.59 and
// 8.2 ms for the same errors.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "iesh_hop.cuh"

namespace iesh {

constexpr int kHopFxMaxNe = 112;  // 28 products per lane: sum y1 a0 below 2^61

// n = n1 2^B + n0, |n0| <= 2^(B-1)
template <int B>
__device__ __forceinline__ int4 fx_pack(long long re, long long im)
{
    int4 v;
    v.x = (int)((re + (1ll << (B - 1))) >> B);
    v.y = (int)(re - ((long long)v.x << B));
    v.z = (int)((im + (1ll << (B - 1))) >> B);
    v.w = (int)(im - ((long long)v.z << B));
    return v;
}
__device__ __forceinline__ long long fx_join(int n1, int n0) { return ((long long)n1 << 30) + n0; }  // of y
__device__ __forceinline__ long long wide(int a, int b) { return (long long)a * (long long)b; }

// The sums of y a: y1 a1, y1 a0, y0 a1, of the real and the imaginary part.
struct FxSum {
    long long hr, hi, mr, mi, nr, ni;
};
__device__ __forceinline__ void fx_mad(FxSum &s, int4 y, int4 a)
{
    const int nz = -y.z, nw = -y.w;  // -im
    s.hr += wide(y.x, a.x);
    s.hi += wide(y.x, a.z);
    s.hr += wide(nz, a.z);
    s.hi += wide(y.z, a.x);
    s.mr += wide(y.x, a.y);
    s.mi += wide(y.x, a.w);
    s.mr += wide(nz, a.w);
    s.mi += wide(y.z, a.y);
    s.nr += wide(y.y, a.x);
    s.ni += wide(y.y, a.z);
    s.nr += wide(nw, a.z);
    s.ni += wide(y.w, a.x);
}
// the sum in y's unit, over the quad
__device__ __forceinline__ void fx_total(const FxSum &s, unsigned quad, long long &re, long long &im)
{
    const long long half = 1ll << 25;
    re = (long long)((unsigned long long)s.hr + (unsigned long long)((s.mr + (s.nr >> 4) + half) >> 26));
    im = (long long)((unsigned long long)s.hi + (unsigned long long)((s.mi + (s.ni >> 4) + half) >> 26));
    re += __shfl_xor_sync(quad, re, 1);
    im += __shfl_xor_sync(quad, im, 1);
    re += __shfl_xor_sync(quad, re, 2);
    im += __shfl_xor_sync(quad, im, 2);
}
// nonzero unless -2^l <= n < 2^l
__device__ __forceinline__ int fx_out(long long n, int l) { return ((int)(n >> l) + 1) & ~1; }

// Substitutes all unoccupied rows; emit(m, a, Re (C_m S^{-1})_a) for each
// entry.  A, dinv, perm: the factors as k_hop leaves them; off, sum_u and
// sum_l [Ne]: shared, free; scr: 2 Ne N doubles.  All threads of the CTA
// call it after a barrier.  False: A and dinv are unchanged and the entries
// that were emitted are to be formed again.
template <class Emit>
__device__ __forceinline__ bool hop_fixed(double2 *A, double2 *dinv, const int *perm, int *off, int *sum_u, int *sum_l,
                                          const int *unocc, const double2 *Ct, int N, int Ne, double *scr, Emit emit)
{
    const int nu = N - Ne, tid = threadIdx.x, lane = tid & 31;
    double2 *saved = reinterpret_cast<double2 *>(scr);                       // [Ne][Ne]
    int4 *Y = reinterpret_cast<int4 *>(saved + (int64_t)Ne * Ne);            // [Ne][nu]
    int4 *F = reinterpret_cast<int4 *>(A);
    static_assert(kMaxHopElectrons <= kHopFxMaxNe, "28 products per lane at most");
    __shared__ int s_big;  // largest column sum (2^30: outside the range)
    if (tid == 0) s_big = 0;
    auto exponent = [&](int j) { return (pivot_key(dinv[j]) >> 20) - 1023; };  // p_j
    int bad = 0;
    for (int i = tid; i < Ne; i += blockDim.x) {
        off[i] = perm[i] * Ne;
        sum_u[i] = sum_l[i] = 0;
    }
    __syncthreads();
    // U1 and L in fixed point, in place
    for (int idx = tid; idx < Ne * Ne; idx += blockDim.x) {
        const int k = idx / Ne, j = idx - k * Ne, at = off[k] + j;
        double2 v = A[at];
        saved[at] = v;
        if (j == k) continue;
        int d = 0;  // U1 = U_kj / U_kk 2^(p_j - p_k)
        if (j > k) {
            v = cmul(v, dinv[k]);
            d = max(-800, min(800, exponent(j) - exponent(k)));
        }
        if (pivot_key(v) >= 0x3ffc0000 - d * (1 << 20)) {  // 1.75 or more, or not finite
            bad = 1;
            continue;
        }
        const double sc = __hiloint2double((1023 + 56 + d) << 20, 0);
        const int4 f = fx_pack<26>(__double2ll_rn(v.x * sc), __double2ll_rn(v.y * sc));
        F[at] = f;
        atomicAdd(&(j > k ? sum_u : sum_l)[j], (abs(f.x) >> 10) + (abs(f.z) >> 10) + 2);  // in units of 2^-20
    }
    __syncthreads();
    int big = bad << 30;
    for (int i = tid; i < Ne; i += blockDim.x) {
        big = max(big, max(sum_u[i], sum_l[i]));
        int p = exponent(i);
        if (p > 400 || p < -400) {
            big = 1 << 30;
            p = 0;
        }
        sum_u[i] = p;
        const double sc = __hiloint2double((1023 - p) << 20, 0);
        dinv[i] = make_double2(dinv[i].x * sc, dinv[i].y * sc);  // 1 / U'_ii
    }
    if (big) atomicMax(&s_big, big);
    __syncthreads();
    big = s_big;
    bad = big >= 15 << 20;
    const int *unit = sum_u;  // p_j
    const int l = min(60, 62 - (32 - __clz(big >> 20)));
    const int sub = tid & 3, grp = tid >> 2, ngrp = blockDim.x >> 2;
    const unsigned quad = 0xFu << (lane & ~3);
    if (!bad)
        for (int u0 = 0; u0 < nu; u0 += ngrp) {
            const int u = u0 + grp;
            const bool live = u < nu;
            const int m = live ? unocc[u] : 0;
            int4 *y = Y + (live ? u : 0);
            // the exponent of the row's largest scaled entry
            int e = -4096;
            if (live)
                for (int i = sub; i < Ne; i += 4) {
                    const int key = pivot_key(Ct[(int64_t)i * N + m]);
                    if (key) e = max(e, key >= 0x7ff00000 ? 4096 : (key >> 20) - 1023 + unit[i]);
                }
            e = max(e, __shfl_xor_sync(quad, e, 1));
            e = max(e, __shfl_xor_sync(quad, e, 2));
            if (e == -4096) e = 0;
            int room = 4, out = 0;  // of this row
            if (e > 500 || e < -500) {
                bad = 1;
                e = 0;
            }
          again:
            if (live && !bad)
                for (int i = sub; i < Ne; i += 4) {
                    const double2 c = Ct[(int64_t)i * N + m];
                    const double up = __hiloint2double((1023 + l - room - e + unit[i]) << 20, 0);
                    *reinterpret_cast<longlong2 *>(y + i * nu) = make_longlong2(__double2ll_rn(c.x * up), __double2ll_rn(c.y * up));
                }
            __syncwarp(quad);
            // y U1 = c
            for (int jc = 0; jc < Ne; ++jc) {
                FxSum s = {0, 0, 0, 0};
                if (live)
#pragma unroll 2
                    for (int i = sub; i < jc; i += 4) fx_mad(s, y[i * nu], F[off[i] + jc]);
                long long re, im;
                fx_total(s, quad, re, im);
                if (live && sub == (jc & 3)) {
                    const longlong2 c = *reinterpret_cast<const longlong2 *>(y + jc * nu);
                    re = c.x - re;
                    im = c.y - im;
                    out |= fx_out(re, l) | fx_out(im, l);
                    y[jc * nu] = fx_pack<30>(re, im);
                }
                __syncwarp(quad);
            }
            // y D'^{-1}
            if (live)
                for (int i = sub; i < Ne; i += 4) {
                    const int4 v = y[i * nu];
                    const double2 r = cmul(make_double2((double)fx_join(v.x, v.y), (double)fx_join(v.z, v.w)), dinv[i]);
                    if (pivot_key(r) >= (1023 + l) << 20) {
                        out = 1;
                        y[i * nu] = make_int4(0, 0, 0, 0);
                    } else {
                        y[i * nu] = fx_pack<30>(__double2ll_rn(r.x), __double2ll_rn(r.y));
                    }
                }
            __syncwarp(quad);
            // x L = y
            for (int jc = Ne - 2; jc >= 0; --jc) {
                FxSum s = {0, 0, 0, 0};
                if (live)
#pragma unroll 2
                    for (int i = jc + 1 + ((sub - (jc + 1)) & 3); i < Ne; i += 4) fx_mad(s, y[i * nu], F[off[i] + jc]);
                long long re, im;
                fx_total(s, quad, re, im);
                if (live && sub == (jc & 3)) {
                    const int4 v = y[jc * nu];
                    re = fx_join(v.x, v.y) - re;
                    im = fx_join(v.z, v.w) - im;
                    out |= fx_out(re, l) | fx_out(im, l);
                    y[jc * nu] = fx_pack<30>(re, im);
                }
                __syncwarp(quad);
            }
            // (a row that has been given up is of no further use)
            if (__any_sync(quad, out) && !bad) {
                if (room < 13) {
                    room += 3;
                    out = 0;
                    goto again;
                }
                bad = 1;
            }
            const double down = __hiloint2double((1023 - l + room + e) << 20, 0);
            if (live)
                for (int i = sub; i < Ne; i += 4) {
                    const int4 v = y[i * nu];
                    emit(m, perm[i], down * (double)fx_join(v.x, v.y));
                }
        }
    bad = __syncthreads_or(bad);
    if (bad) {
        for (int idx = tid; idx < Ne * Ne; idx += blockDim.x) A[idx] = saved[idx];
        for (int i = tid; i < Ne; i += blockDim.x) {  // (exact)
            const double sc = __hiloint2double((1023 + unit[i]) << 20, 0);
            dinv[i] = make_double2(dinv[i].x * sc, dinv[i].y * sc);
        }
    }
    __syncthreads();
    return !bad;
}

}  // namespace iesh
