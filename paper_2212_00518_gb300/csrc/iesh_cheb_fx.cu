// iesh_cheb_fx.cu -- FP64 Chebyshev propagator with the contraction of every
// order on the tensor cores, in exact integer arithmetic (N <= 256).
//
// The exponential integrator of Sec. II C, as k_cheb (iesh_step.cu):
//   exp(-i H) C = e^{-ic} sum_k (2 - delta_k0) (-i)^k J_k(rho) T_k(X) C,
//   X = (H - c) / rho,  T_{k+1} = 2 X T_k - T_{k-1},  H = L - i W.
// The FP64 pipe of this GPU issues 2 DFMA per clock and SM, which bounds the
// SIMT kernel (99% busy); the FP16 tensor cores multiply small integers
// exactly and add them exactly as long as a sum stays below 2^24.  So T_k is
// held in fixed point (64-bit integers, unit 2^-60 of the electron column's
// scale) and the product W' T_k, W' = (2 / rho) W, is split into digits (the
// error-free splitting of Ozaki, Ogita, Oishi and Rump 2012, in a fixed-point
// form):
//   W' = 2^e sum_i W_i 2^{-8-8i},  T = sum_j T_j 2^{-8-8j},  i, j = 0..6,
// integers |W_0|, |T_0| <= 512 and |W_i|, |T_j| <= 128, each stored as an
// FP16 value.  The products of one weight, i + j = g, share one FP32
// accumulator in tensor memory (groups g = 0..G, G = 5 or 6, 28 products at
// most); an accumulator is an exact integer as long as it stays below 2^24
// (digits of random sign give 2^18 at N = 128; only digits aligned in sign along
// a whole row and column pass it, and then round in the last of 24 bits).  The
// update reads the group sums, adds them as 64-bit integers and forms
//   T_{k+1} = 2 (L - c) / rho T_k - i W' T_k - T_{k-1}
// in integer arithmetic; the Chebyshev sum is a 64-bit integer as well.
//
// Accuracy.  The state keeps 2^-60 of a column whose norm lies in [1, 2),
// against the FP64 kernel's rounding of 2^-54 .. 2^-57 of typical entries.
// The terms left out (i + j > G) amount to about 2^{17.5 - 16 - 8 (G+1) + e}:
// G is the smallest value that brings this to 2^-56, at most 6 (2^-54.5 for
// |W'| of order 1).  Couplings so weak that an entry which starts from zero
// stays small give every entry a unit of its own, up to 2^16 finer (a byte per
// entry, from its size and a bound of its growth), and G = 5, 2^-46.5 of max |W'|:
// the amplitude of an empty orbital after a step from unit columns, of the size
// of W', then carries 2e-14 of the largest of them and 10^-12 of its own (N = 101,
// dt = 1; one unit per column: 2e-11 and 2e-9; FP64 arithmetic: 2e-16).  Couplings
// below 2^-75 of the interval vanish.
//
// Layout.  One persistent CTA of 512 threads per SM takes (trajectory, range
// of electrons) items, in blocks of up to 64 real columns for one 128-row
// tile (N <= 128) and 32 for two: the group sums and the Chebyshev sum share
// tensor memory (512 columns).  The CTA cuts W' into digits once per item,
// in the order the MMAs read them, into its own slot of a workspace that
// stays in L2; one thread loads them by bulk copies into shared memory, as
// stages (one 16-wide K step of one row tile, all digits): all of them once
// per item where they fit beside T's digits, else through a ring.  T's
// digits stay in shared memory (N-major B operand: a thread holds one
// orbital row and writes four consecutive columns with one 8-byte store);
// T_k and T_{k-1} are in registers (up to 16 values each per thread).
//
// Measured (ms per step, against the SIMT kernel): N = 101, Ne = 50, 4096
// trajectories 7.5 against 65.7; N = 201, Ne = 100, 1024 trajectories 12.6
// against 127; N = 41, Ne = 20, 1000 trajectories, 20 orders 1.23 against
// 2.76.  (One unit per column and G = 4 for weak couplings: 6.4, 9.5 and 1.17.)
// MMAs and update do not overlap (tensor memory holds one block); the update's
// 64-bit integer arithmetic, about 100 instructions per entry, is
// latency-bound at 4 warps per scheduler.
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "iesh_common.cuh"
#include "iesh_kernels.h"
#include "iesh_tc.cuh"

namespace iesh {

namespace {

constexpr int kFxThreads = 512;
constexpr int kFxWarps = kFxThreads / 32;
constexpr int kFxS = 7;               // digits of each operand
constexpr int kFxMaxCols = 16;        // real columns per thread
constexpr int kFxMaxEl = 32;          // electrons per block
constexpr int kFxMaxShift = 16;       // of an entry's unit below 2^-60
constexpr int kFxWaitLimit = 1 << 22;
constexpr int kFxMaxStages = 16;
constexpr size_t kFxMaxSmem = 220 * 1024;
// at the end of the shared memory: the threads' shifts, 8 bytes each; an MMA
// reads 16 row groups from a digit's start, up to there (rows that are not used)
constexpr int kFxSlack = kFxThreads * 8;

// Sizes: rg 8-row groups of W, row tiles of 128 rows, ks K steps of 16.
struct FxShape {
    int Kp, ks, rg, rg0, tiles;
    size_t ws;    // workspace bytes of a CTA
};
__host__ __device__ inline FxShape fx_shape(int N)
{
    FxShape f;
    f.Kp = (N + 15) & ~15;
    f.ks = f.Kp / 16;
    f.rg = (N + 7) / 8;
    f.rg0 = f.rg < 16 ? f.rg : 16;
    f.tiles = N > 128 ? 2 : 1;
    f.ws = (size_t)f.ks * kFxS * f.rg * 256;
    return f;
}
// Electrons per block: tensor memory holds nsl group sums and the 64-bit
// Chebyshev sum of tiles x 2 eb real columns (a multiple of 16), nsl = G + 1.
__host__ __device__ inline int fx_block_cap(int tiles, int nsl)
{
    return (nsl <= 6 ? 32 : 24) / tiles;
}

// 64-bit integer pieces: a balanced split x = hi 2^32 + lo with lo signed,
// and the products of two split numbers.
struct Split {
    int hi, lo;
};
__device__ __forceinline__ Split split64(long long x)
{
    Split s;
    s.lo = (int)(uint32_t)x;
    s.hi = (int)(x >> 32) + (s.lo < 0 ? 1 : 0);
    return s;
}
// (a b) 2^-64 2^s, 0 <= s < 32; the lo lo product (below 2^-2 of the
// unshifted unit) is left out.
__device__ __forceinline__ long long mul_shift(Split a, Split b, int s)
{
    const long long p0 = (long long)a.hi * b.hi;
    const long long p1 = (long long)a.hi * b.lo + (long long)a.lo * b.hi;
    const long long h = p0 + (p1 >> 32);
    const uint32_t w0 = (uint32_t)p1, w1 = (uint32_t)h, w2 = (uint32_t)(h >> 32);
    const uint32_t r0 = __funnelshift_l(w0, w1, s), r1 = __funnelshift_l(w1, w2, s);
    return (long long)(((uint64_t)r1 << 32) | r0);
}
// the same with the lo lo product: every bit of the result's unit
__device__ __forceinline__ long long mul_shift_all(Split a, Split b, int s)
{
    const long long p0 = (long long)a.hi * b.hi;
    const long long p1 = (long long)a.hi * b.lo + (long long)a.lo * b.hi + (((long long)a.lo * b.lo) >> 32);
    const long long h = p0 + (p1 >> 32);
    const uint32_t w0 = (uint32_t)p1, w1 = (uint32_t)h, w2 = (uint32_t)(h >> 32);
    const uint32_t r0 = __funnelshift_l(w0, w1, s), r1 = __funnelshift_l(w1, w2, s);
    return (long long)(((uint64_t)r1 << 32) | r0);
}
__device__ __forceinline__ long long sar64(long long x, int s)  // 0 <= s < 32
{
    const int hi = (int)(x >> 32);
    return (long long)(((uint64_t)(uint32_t)(hi >> s) << 32) | __funnelshift_r((uint32_t)x, (uint32_t)hi, s));
}
// (a b) 2^-64 2^(s + d), |d| < 29
__device__ __forceinline__ long long mul_unit(Split a, Split b, int s, int d)
{
    return sar64(mul_shift_all(a, b, s + max(d, 0)), max(-d, 0));
}
// The group sums d (exact integers) as one integer of unit 2^(-60 - s), for W' =
// 2^e Wint: the weight of group g is 2^(-16 - 8 g + e), t = -4 - e - s >= -8.  The
// sum of the first six groups fits 63 bits (|d_0| < 2^22.5).  left: t may be
// negative (strong couplings, no shifts; uniform).
template <int NSL>
__device__ __forceinline__ long long fx_sum(const float (&d)[NSL], int t, bool left)
{
    long long a = __float2int_rn(d[5]);
    a += (long long)__float2int_rn(d[4]) * 256;
    a += (long long)__float2int_rn(d[3]) * 65536;
    a += (long long)__float2int_rn(d[2]) * 16777216;
    a += (long long)(__float2int_rn(d[0]) * 256 + __float2int_rn(d[1])) << 32;
    long long r;
    if (NSL > 6 && left) r = a << -t;  // (e > -4: seven digits)
    else r = sar64(a, t);
    if constexpr (NSL > 6) r += __float2int_rn(d[6]) >> min(31, t + 8);
    return r;
}
// v 2^ex as a double, rounded to nearest, by its bits; 0 below the normal
// range, infinity above.
__device__ __forceinline__ double double_of(long long v, int ex)
{
    if (v == 0) return 0.0;
    uint64_t m = v < 0 ? 0ull - (uint64_t)v : (uint64_t)v;
    const int lz = __clzll((long long)m);
    m <<= lz;
    const uint64_t r = (m >> 11) + ((m >> 10) & 1);
    const int E = 1023 + 63 - lz + ex;
    uint64_t b = ((uint64_t)(E - 1) << 52) + r;
    if (E < 1) b = 0;
    if (E > 2046) b = 0x7ff0000000000000ull;
    return __longlong_as_double((long long)(b | (v < 0 ? 0x8000000000000000ull : 0ull)));
}

// round(x 2^sh) of a double by its bits (no FP64 instruction); |x 2^sh| < 2^62.
__device__ __forceinline__ long long fixed_of(double x, int sh)
{
    const long long b = __double_as_longlong(x);
    const int ex = (int)(b >> 52) & 0x7ff;
    uint64_t m = (uint64_t)b & 0xfffffffffffffull;
    if (ex) m |= 1ull << 52;
    const int k = (ex ? ex : 1) - 1075 + sh;
    uint64_t r = 0;
    if (k >= 0) r = m << (k < 12 ? k : 12);
    else if (k > -54) r = (m + (1ull << (-k - 1))) >> -k;
    return b < 0 ? -(long long)r : (long long)r;
}

// 2^(E + 2), above the modulus of a number whose larger part has the exponent
// E; 0 below FP32's range.
__device__ __forceinline__ float above(int E) { return E < -120 ? 0.0f : __int_as_float((min(E, 100) + 129) << 23); }
__device__ __forceinline__ int exponent_of(double re, double im)  // of the larger part; -1023: zero
{
    return (int)((uint32_t)max(__double2hiint(re) & 0x7fffffff, __double2hiint(im) & 0x7fffffff) >> 20) - 1023;
}

// |x| as a float by its bits, truncated; 0 below and infinity above range.
__device__ __forceinline__ float abs_float(double x)
{
    const int h = __double2hiint(x) & 0x7fffffff;
    if (h < (897 << 20)) return 0.0f;
    if (h >= (1150 << 20)) return __int_as_float(0x7f800000);
    return __int_as_float(((h - (896 << 20)) << 3) | (int)((uint32_t)__double2loint(x) >> 29));
}

__device__ __forceinline__ void bulk_load(uint32_t dst, const void *src, uint32_t bytes, uint64_t *mbar)
{
    const uint32_t mb = tc::smem_addr(mbar);
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mb), "r"(bytes) : "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(mb)
                 : "memory");
}
// What the issuing thread needs about an item: descriptors of the ring and of
// T's digits, descriptor steps (16-byte units) between slots, digits of W
// (per row tile) and of T, the ring's slot of the next stage.
struct FxMma {
    uint64_t ad0, ad, bd0;
    uint64_t *full, *empty;
    uint32_t slot, nst, nstage, tiles, step, da0, da1, db, NB, d0, idesc;
};

// The MMAs of one order: for every stage (K step, row tile) all pairs i + j
// < NSL, issued by one thread.  The pair loops are unrolled: an MMA then takes
// 41 cycles (16 and 32 columns) to 50 (64 columns), against 84 when the
// thread walks them as a loop.
template <int NSL>
__device__ __forceinline__ bool fx_order(FxMma &m, uint32_t &fpar, bool wait, bool ring)
{
    uint64_t bd = m.bd0, ad = m.ad;
    uint32_t sl = m.slot;
    const uint32_t d0 = m.d0, NB = m.NB, idesc = m.idesc, db = m.db;
    for (uint32_t st = 0; st < m.nstage; ++st) {
        if (wait) {
            if (!tc::mbar_wait(&m.full[sl], (fpar >> sl) & 1u, kFxWaitLimit)) return false;
            fpar ^= 1u << sl;
        }
        const uint32_t tl = m.tiles == 2 ? st & 1u : 0u, da = tl ? m.da1 : m.da0;
        const uint32_t dt = d0 + tl * NSL * NB, acc = st >= m.tiles ? 1u : 0u;
#pragma unroll
        for (int i = 0; i < NSL; ++i)
#pragma unroll
            for (int j = 0; j < NSL - i; ++j)
                tc::mma_f16(dt + (i + j) * NB, ad + i * da, bd + j * db, idesc, i == 0 ? acc : 1u);
        if (ring) tc::commit(&m.empty[sl]);
        if (m.tiles == 1 || tl) bd += 16;
        ad += m.step;
        if (++sl == m.nst) {
            sl = 0;
            ad = m.ad0;
        }
    }
    m.slot = sl;
    m.ad = ad;
    return true;
}

// Digits of four columns (two electrons, re and im) of T into the B operand.
// With the bias the digits are the bytes of t >> 4; 0x64 above a byte makes
// the FP16 number 1024 + byte.  s0, s1: shifts of the two electrons' entries.
template <int NSL>
__device__ __forceinline__ void put_digits(unsigned char *b, int bsl, const long long *t, int s0, int s1, int nsl = NSL)
{
    constexpr long long kBias = (((512ll << 48) + 0x808080808080ll) << 4) + 8;
    uint32_t lo[4], hi[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const long long u = (sar64(t[q], q < 2 ? s0 : s1) + kBias) >> 4;
        lo[q] = (uint32_t)u;
        hi[q] = (uint32_t)(u >> 32);
    }
    const __half2 k1152 = __half2half2(__ushort_as_half(0x6480)), k1536 = __half2half2(__ushort_as_half(0x6600));
    auto put = [&](int j, uint32_t w0, uint32_t w1, __half2 off) {
        const __half2 h0 = __hsub2(*reinterpret_cast<__half2 *>(&w0), off);
        const __half2 h1 = __hsub2(*reinterpret_cast<__half2 *>(&w1), off);
        uint2 v;
        v.x = *reinterpret_cast<const uint32_t *>(&h0);
        v.y = *reinterpret_cast<const uint32_t *>(&h1);
        *reinterpret_cast<uint2 *>(b + j * bsl) = v;
    };
    put(0, __byte_perm(hi[0], hi[1], 0x7632) | 0x64006400u, __byte_perm(hi[2], hi[3], 0x7632) | 0x64006400u, k1536);
    {
        const uint32_t x0 = __byte_perm(hi[0], hi[1], 0x5140), x1 = __byte_perm(hi[2], hi[3], 0x5140);
        if (NSL > 1 && nsl > 1) put(1, __byte_perm(x0, 0x64646464u, 0x4342), __byte_perm(x1, 0x64646464u, 0x4342), k1152);
        if (NSL > 2 && nsl > 2) put(2, __byte_perm(x0, 0x64646464u, 0x4140), __byte_perm(x1, 0x64646464u, 0x4140), k1152);
    }
    if (NSL > 3 && nsl > 3) {
        const uint32_t x0 = __byte_perm(lo[0], lo[1], 0x7362), x1 = __byte_perm(lo[2], lo[3], 0x7362);
        put(3, __byte_perm(x0, 0x64646464u, 0x4342), __byte_perm(x1, 0x64646464u, 0x4342), k1152);
        if (NSL > 4 && nsl > 4) put(4, __byte_perm(x0, 0x64646464u, 0x4140), __byte_perm(x1, 0x64646464u, 0x4140), k1152);
    }
    if (NSL > 5 && nsl > 5) {
        const uint32_t x0 = __byte_perm(lo[0], lo[1], 0x5140), x1 = __byte_perm(lo[2], lo[3], 0x5140);
        put(5, __byte_perm(x0, 0x64646464u, 0x4342), __byte_perm(x1, 0x64646464u, 0x4342), k1152);
        if (NSL > 6 && nsl > 6) put(6, __byte_perm(x0, 0x64646464u, 0x4140), __byte_perm(x1, 0x64646464u, 0x4140), k1152);
    }
}

// One order of the series for this thread's row and columns: the group sums
// and the Chebyshev sum come from tensor memory, the new digits go to B.
// sL: shift of the diagonal's product; t: shift of fx_sum for s = 0; Jk
// carries the sign of (-i)^(k+1), odd whether it is imaginary; shifts: s of this
// thread's entries, a byte per electron in shared memory.
template <int NSL>
__device__ __forceinline__ void fx_update(long long (&tk)[kFxMaxCols], long long (&tp)[kFxMaxCols], int ncol, int col0,
                                          bool rowok, uint32_t dcol, uint32_t acol, uint32_t NB, unsigned char *brow,
                                          int bn, int bsl, const Split Ls, int sL, int t, const Split Jk, bool odd,
                                          const uchar2 *shifts)
{
#pragma unroll
    for (int q4 = 0; q4 < kFxMaxCols; q4 += 4) {
        if (q4 >= ncol) break;
        const uchar2 s2 = shifts[q4 / 4];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int c = q4 + 2 * h;
            const int s = h ? s2.y : s2.x;
            float dr[NSL], di[NSL], a0, a1, a2, a3;
#pragma unroll
            for (int g = 0; g < NSL; ++g) tc::tmem_ld2(dcol + (uint32_t)g * NB + c, dr[g], di[g]);
            tc::tmem_ld4(acol + 2 * c, a0, a1, a2, a3);
            long long nr = mul_shift(split64(tk[c]), Ls, sL) - tp[c];
            long long ni = mul_shift(split64(tk[c + 1]), Ls, sL) - tp[c + 1];
            tp[c] = tk[c];
            tp[c + 1] = tk[c + 1];
            tc::tmem_wait_ld();
            nr += fx_sum<NSL>(di, t - s, t < 0);
            ni -= fx_sum<NSL>(dr, t - s, t < 0);
            tk[c] = nr;
            tk[c + 1] = ni;
            const long long jr = mul_shift(split64(nr), Jk, 3), ji = mul_shift(split64(ni), Jk, 3);
            long long ar = ((long long)__float_as_int(a1) << 32) | (uint32_t)__float_as_int(a0);
            long long ai = ((long long)__float_as_int(a3) << 32) | (uint32_t)__float_as_int(a2);
            if (odd) {
                ar += ji;
                ai -= jr;
            } else {
                ar += jr;
                ai += ji;
            }
            tc::tmem_st4(acol + 2 * c, __int_as_float((int)ar), __int_as_float((int)(ar >> 32)), __int_as_float((int)ai),
                         __int_as_float((int)(ai >> 32)));
        }
        const int cb = col0 + q4;
        if (rowok) put_digits<NSL>(brow + (cb >> 3) * bn + (cb & 7) * 2, bsl, tk + q4, s2.x, s2.y);
    }
    tc::tmem_wait_st();
}

__global__ void __launch_bounds__(kFxThreads, 1)
    k_cheb_fx(DevState s, double dt, int64_t items, int parts, unsigned char *ws_all, size_t ws_stride)
{
    extern __shared__ __align__(1024) unsigned char fx_smem[];
    __shared__ __align__(8) uint64_t full[kFxMaxStages], empty[kFxMaxStages], done;
    __shared__ uint32_t tmem_slot;
    __shared__ int s_red[kFxWarps], s_max[8][kFxMaxEl], s_x[kFxMaxEl];
    __shared__ float s_ssq[8][kFxMaxEl];
    __shared__ Split s_J[kChebMax], s_a0[2][kFxMaxEl], s_a1[2][kFxMaxEl];
    __shared__ int s_as[kFxMaxEl];
    __shared__ float s_af[kFxMaxEl];
    constexpr int kNan = 0x7fffffff;  // column scale of a column that is not finite
    const int N = s.N, Ne = s.Ne;
    const FxShape f = fx_shape(N);
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int tile = f.tiles == 2 ? (warp >> 2) & 1 : 0, cg = f.tiles == 2 ? warp >> 3 : warp >> 2;
    const int row = 128 * tile + 32 * (warp & 3) + lane;
    const bool rowok = row < N, wact = row - lane < N;
    unsigned char *B = fx_smem, *ws = ws_all + (size_t)blockIdx.x * ws_stride;
    if (tid == 0) {
        for (int q = 0; q < kFxMaxStages; ++q) {
            tc::mbar_init(&full[q], 1);
            tc::mbar_init(&empty[q], 1);
        }
        tc::mbar_init(&done, 1);
    }
    if (warp == 0) tc::tmem_alloc(&tmem_slot, 512);
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = tmem_slot;
    const uint32_t my_lane = tmem + ((uint32_t)(32 * (warp & 3)) << 16);
    // phases: parities of the full barriers (the issuing thread's), of the
    // empty barriers and the slots whose empty phase is outstanding (the
    // copying thread's), orders done (all)
    uint32_t fpar = 0, epar = 0, epend = 0, norder = 0;
    bool ok = true;

    for (int64_t item = blockIdx.x; item < items; item += gridDim.x) {
        const int64_t t = traj_of(s, item / parts);
        if (t < 0 || (s.status[t] & ST_DONE)) continue;  // uniform over the CTA
        if (!ok) {  // an earlier wait gave up: this item's coefficients are not updated
            if (tid == 0) atomicOr(&s.status[t], ST_TC_WAIT);
            continue;
        }
        const int part = (int)(item % parts);
        const int e_lo = Ne * part / parts, e_hi = Ne * (part + 1) / parts;
        const double *cb = s.cheb + t * kChebStride;
        const double c = cb[0], rho = cb[1];
        const int K = (int)cb[2];
        const double *Wd = s.scratch + t * s.scratch_stride;
        double2 *C = reinterpret_cast<double2 *>(s.C) + (int64_t)t * Ne * N;
        const double w2 = rho > 0.0 ? 2.0 / rho : 0.0;

        // exponent of max |W| (its high word orders like the magnitude)
        int mx = 0;
        for (int idx = tid; idx < N * N; idx += kFxThreads) mx = max(mx, __double2hiint(Wd[idx]) & 0x7fffffff);
        mx = __reduce_max_sync(0xffffffffu, mx);
        if (lane == 0) s_red[warp] = mx;
        for (int k = tid; k <= K; k += kFxThreads) {
            const long long j = fixed_of((k ? 2.0 : 1.0) * cb[3 + k], 62);  // |2 J_k| < 2
            s_J[k] = split64((k & 2) ? -j : j);  // (-i)^k = 1, -i, -1, i
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < kFxWarps; ++q) mx = max(mx, s_red[q]);
        const double wmax = __hiloint2double(mx, -1) * w2;  // max |W'| rounded up
        const double Lc = rowok ? w2 * (0.5 * dt * (s.lam_prev[t * N + row] + s.lam[t * N + row]) - c) : 0.0;
        // not finite (the coupling kernels bound finite values): every
        // coefficient becomes NaN
        const bool bad = __syncthreads_or(!(wmax < 32.0) || !(fabs(Lc) < 1e8) || !(fabs(c) < 1e300));
        if (bad) {
            const double nan = __longlong_as_double(0x7ff8000000000000ll);
            for (int idx = 2 * e_lo * N + tid; idx < 2 * e_hi * N; idx += kFxThreads) reinterpret_cast<double *>(C)[idx] = nan;
            continue;
        }
        // an entry of T_k changes by at most this much of its column's norm: 2.5
        // max |W'| sqrt(N) per order (columns normalised below 2, with the
        // deflated level's share), at most k-fold in T_k; the deflated level's row,
        // where T_k grows faster, by what k_build_w found
        const float grow = 1.3f * abs_float(wmax) * sqrtf((float)N) * (float)(K * (K + 1));
        // couplings so weak that entries that start from zero stay small: every
        // entry has a unit of its own
        const bool shifts = grow < 1.0f;  // (max |W'| is below 2^-4 then)
        uchar2 *s_shift = reinterpret_cast<uchar2 *>(fx_smem + kFxMaxSmem - kFxSlack + 8 * tid);
        // W' = 2^e Wint with |Wint| < 2, e in [-26, 4]; nsl digits: the fewest
        // with 17.5 - 16 - 8 nsl + e <= -56 (7 at most); with shifts, 2^-46 of
        // max |W'|.  Without shifts e is above -18: 6 digits at least
        const int ew = (int)((__double2hiint(wmax) >> 20) & 0x7ff) - 1023, e = max(-26, ew);
        const int nsl = shifts ? (e > ew ? 7 : 6) : min(kFxS, (58 + e + 7) / 8);
        // the row's diagonal 2 (L - c) / rho, times 2^(61 - fL) below 2^62
        const int fL = max(1, (int)((__double2hiint(Lc) >> 20) & 0x7ff) - 1023);
        const Split Ls = split64(fixed_of(Lc, 61 - fL));
        // blocks of the item's electrons
        int cap = f.tiles == 2 && nsl == kFxS ? 8 : fx_block_cap(f.tiles, nsl);
        if (s.cheb_ept > 0) cap = min(cap, s.cheb_ept * s.cheb_G);  // a requested shape
        const int nblk = (e_hi - e_lo + cap - 1) / cap, eb = (e_hi - e_lo + nblk - 1) / nblk;
        const int NB = (2 * eb + 15) & ~15, ncol = NB * f.tiles / 4, col0 = cg * ncol;
        const int bn = (f.Kp / 8) * 128, bsl = (NB / 8) * bn;  // bytes of 8 columns, of a digit of T
        const int stage0 = nsl * f.rg0 * 256, stage1 = f.tiles == 2 ? nsl * (f.rg - 16) * 256 : 0;
        const int nstage = f.ks * f.tiles;  // stages per order
        const int nst = min(min(kFxMaxStages, nstage), (int)((kFxMaxSmem - kFxSlack - (size_t)nsl * bsl) / stage0));
        const bool resident = nst == nstage;
        const uint32_t ring = tc::smem_addr(fx_smem) + (uint32_t)(nsl * bsl);
        // digits of W', K step by K step and row tile by row tile:
        // A[j][i] = W_ji = -W_ij, consecutive threads on consecutive rows j
        {
            const int rows = 8 * f.rg, units = rows * (f.Kp / 8);
            for (int it = tid; it < units; it += kFxThreads) {
                const int kc = it / rows, r = it - kc * rows;
                uint32_t h[kFxS][4];
#pragma unroll
                for (int q2 = 0; q2 < 4; ++q2) {
                    long long u[2];
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        const int k = 8 * kc + 2 * q2 + q;
                        long long v = 0;
                        if (r < N && k < N) v = -fixed_of(Wd[(int64_t)k * N + r] * w2, 56 - e);
                        u[q] = v + ((512ll << 48) + 0x808080808080ll);
                    }
                    const uint32_t l0 = (uint32_t)u[0], l1 = (uint32_t)u[1], h0 = (uint32_t)(u[0] >> 32), h1 = (uint32_t)(u[1] >> 32);
                    auto half2_of = [&](uint32_t w, uint32_t off) {
                        const __half2 a = *reinterpret_cast<__half2 *>(&w);
                        const __half2 d = __hsub2(a, __half2half2(__ushort_as_half((unsigned short)off)));
                        return *reinterpret_cast<const uint32_t *>(&d);
                    };
                    // W_0 + 512 in [0, 1024] by conversions, the other digits as
                    // bytes below 0x64 (1024 + byte)
                    const __half2 top = __halves2half2(__int2half_rn((int)(h0 >> 16) - 512), __int2half_rn((int)(h1 >> 16) - 512));
                    h[0][q2] = *reinterpret_cast<const uint32_t *>(&top);
                    const uint32_t x1 = __byte_perm(h0, h1, 0x5140), x3 = __byte_perm(l0, l1, 0x7362), x5 = __byte_perm(l0, l1, 0x5140);
                    h[1][q2] = half2_of(__byte_perm(x1, 0x64646464u, 0x4342), 0x6480);
                    h[2][q2] = half2_of(__byte_perm(x1, 0x64646464u, 0x4140), 0x6480);
                    h[3][q2] = half2_of(__byte_perm(x3, 0x64646464u, 0x4342), 0x6480);
                    h[4][q2] = half2_of(__byte_perm(x3, 0x64646464u, 0x4140), 0x6480);
                    h[5][q2] = half2_of(__byte_perm(x5, 0x64646464u, 0x4342), 0x6480);
                    h[6][q2] = half2_of(__byte_perm(x5, 0x64646464u, 0x4140), 0x6480);
                }
                const int tl = r >> 7, rgt = tl ? f.rg - 16 : f.rg0;
                unsigned char *dst = ws + (size_t)(kc >> 1) * (stage0 + stage1) + (tl ? stage0 : 0) + ((r & 127) >> 3) * 256 +
                                     (kc & 1) * 128 + (r & 7) * 16;
#pragma unroll
                for (int i = 0; i < kFxS; ++i)
                    if (i < nsl) *reinterpret_cast<uint4 *>(dst + (size_t)i * rgt * 256) = make_uint4(h[i][0], h[i][1], h[i][2], h[i][3]);
            }
        }
        asm volatile("fence.proxy.async;" ::: "memory");  // the bulk copies read what was just written
        // T's digits: rows past N stay zero
        for (int w = tid; w < nsl * bsl / 16; w += kFxThreads) reinterpret_cast<uint4 *>(B)[w] = make_uint4(0, 0, 0, 0);
        const double *df = s.defl ? s.defl + t * defl_stride(N, Ne) : nullptr;
        const bool defl = df && df[0] != 0.0;
        const float grow_row = defl && row == N - 1 ? 2.0f * abs_float(df[4]) : grow;
        Split ur = {0, 0}, ui = {0, 0};
        float uf = 0.0f;  // at least |u_j|
        if (defl && rowok) {
            ur = split64(fixed_of(df[kDeflHead + row], 62));
            ui = split64(fixed_of(df[kDeflHead + N + row], 62));
            uf = above(exponent_of(df[kDeflHead + row], df[kDeflHead + N + row]));
        }
        Split cc, sc;  // e^{-ic}
        {
            double sn, cs;
            sincos(c, &sn, &cs);
            cc = split64(fixed_of(cs, 62));
            sc = split64(fixed_of(sn, 62));
        }
        const uint32_t idesc = tc::idesc_f16(128, NB) | (1u << 16);  // B is N-major
        const uint32_t dcol = my_lane + (uint32_t)(tile * nsl * NB + col0);
        const uint32_t acol = my_lane + (uint32_t)(f.tiles * nsl * NB + 2 * (tile * NB + col0));
        unsigned char *brow = B + (row >> 3) * 128 + (row & 7) * 16;
        uint32_t qp = 0;  // stages copied in this item
        FxMma m;
        m.ad0 = m.ad = tc::smem_desc(ring, 128, 256);
        m.bd0 = tc::smem_desc(tc::smem_addr(B), 128, (uint32_t)bn);
        m.full = full, m.empty = empty;
        m.slot = 0, m.nst = (uint32_t)nst, m.nstage = (uint32_t)nstage, m.tiles = (uint32_t)f.tiles;
        m.step = (uint32_t)stage0 / 16u, m.da0 = (uint32_t)f.rg0 * 16u, m.da1 = (uint32_t)(f.rg - 16) * 16u;
        m.db = (uint32_t)bsl / 16u, m.NB = (uint32_t)NB, m.d0 = tmem, m.idesc = idesc;
        const uint32_t qend = resident ? (uint32_t)nstage : (uint32_t)(nblk * K * nstage);
        int ord = 0;  // orders of this item

        for (int blk = 0; blk < nblk && ok; ++blk) {
            const int e0 = e_lo + blk * eb, ne = min(eb, e_hi - e0);
            long long tk[kFxMaxCols], tp[kFxMaxCols];
            // the coefficients (as bits), column norms (as floats: their
            // exponents set the columns' scales) and largest exponents
#pragma unroll
            for (int q = 0; q < kFxMaxCols / 2; ++q) {
                if (2 * q >= ncol) break;
                const int el = col0 / 2 + q;
                double2 v = make_double2(0.0, 0.0);
                if (rowok && el < ne) v = C[(int64_t)(e0 + el) * N + row];
                tk[2 * q] = __double_as_longlong(v.x);
                tk[2 * q + 1] = __double_as_longlong(v.y);
            }
            if (wact)
#pragma unroll
                for (int q = 0; q < kFxMaxCols / 2; ++q) {
                    if (2 * q >= ncol) break;
                    const double vx = __longlong_as_double(tk[2 * q]), vy = __longlong_as_double(tk[2 * q + 1]);
                    const float a = abs_float(vx), b = abs_float(vy);
                    float ss = fmaf(a, a, b * b);
                    int m = max(__double2hiint(vx) & 0x7fffffff, __double2hiint(vy) & 0x7fffffff);
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
                    m = __reduce_max_sync(0xffffffffu, m);
                    if (lane == 0) {
                        s_ssq[4 * tile + (warp & 3)][col0 / 2 + q] = ss;
                        s_max[4 * tile + (warp & 3)][col0 / 2 + q] = m;
                    }
                }
            __syncthreads();
            if (tid < eb) {
                float ss = 0.f;
                int m = 0;
                for (int w = 0; 32 * w < N; ++w) {
                    ss += s_ssq[w][tid];
                    m = max(m, s_max[w][tid]);
                }
                // norm 2^-x in [0.99, 1.98); outside the float range, from the
                // largest entry: norm < 2 sqrt(N) 2^exponent
                int x = (m >> 20) - 1023 + 5;
                if (ss > 1e-30f && ss < 1e30f) x = ilogbf(sqrtf(ss) * 1.0101f);
                if (m >= 0x7ff00000) x = kNan;
                s_x[tid] = x;
                if (defl && tid < ne) {
                    const double *qd = df + kDeflHead + 2 * N + e0 + tid;
                    const double ar = qd[0], ai = qd[Ne], cm = df[2], sm = df[3];
                    // a in a unit of its own, 2^as finer than the column's
                    const int ea = exponent_of(ar, ai);
                    const int as = x == kNan ? 0 : max(0, min(kFxMaxShift, x - ea - 2)), sh = 60 + as - (x == kNan ? 0 : x);
                    s_as[tid] = as;
                    s_af[tid] = above(ea - (x == kNan ? 0 : x));
                    s_a0[0][tid] = split64(fixed_of(ar, sh));
                    s_a0[1][tid] = split64(fixed_of(ai, sh));
                    s_a1[0][tid] = split64(fixed_of(fma(cm, ar, sm * ai), sh));  // e^{-i mu} a
                    s_a1[1][tid] = split64(fixed_of(fma(cm, ai, -(sm * ar)), sh));
                }
            }
            __syncthreads();
            if (wact) {
#pragma unroll
                for (int q4 = 0; q4 < kFxMaxCols; q4 += 4) {
                    if (q4 >= ncol) break;
                    int ups[2] = {0, 0};  // the entries' shifts
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int el = (col0 + q4) / 2 + h;
                        long long vr = 0, vi = 0;
                        const int x = el < ne ? s_x[el] : kNan;
                        if (rowok && x != kNan) {
                            const double cr = __longlong_as_double(tk[q4 + 2 * h]), ci = __longlong_as_double(tk[q4 + 2 * h + 1]);
                            // the entry's shift: |.| 2^(60 + up) stays below 2^61, from
                            // its size, the deflated level's share and its growth
                            const float size = above(exponent_of(cr, ci) - x) + (defl ? s_af[el] * uf : 0.0f) + grow_row;
                            const int up = shifts ? max(0, min(min(kFxMaxShift, -4 - e), 127 - (__float_as_int(size) >> 23))) : 0;
                            vr = fixed_of(cr, 60 - x + up);
                            vi = fixed_of(ci, 60 - x + up);
                            if (defl) {  // c - a u
                                const Split ar = s_a0[0][el], ai = s_a0[1][el];
                                const int d = up - s_as[el];
                                vr -= mul_unit(ar, ur, 2, d) - mul_unit(ai, ui, 2, d);
                                vi -= mul_unit(ar, ui, 2, d) + mul_unit(ai, ur, 2, d);
                            }
                            ups[h] = up;
                        }
                        tk[q4 + 2 * h] = vr;
                        tk[q4 + 2 * h + 1] = vi;
                        tp[q4 + 2 * h] = tp[q4 + 2 * h + 1] = 0;
                        const long long ar = mul_shift(split64(vr), s_J[0], 3), ai = mul_shift(split64(vi), s_J[0], 3);  // unit 2^-61
                        tc::tmem_st4(acol + 2 * (q4 + 2 * h), __int_as_float((int)ar), __int_as_float((int)(ar >> 32)),
                                     __int_as_float((int)ai), __int_as_float((int)(ai >> 32)));
                    }
                    const int cbq = col0 + q4;
                    if (rowok) put_digits<kFxS>(brow + (cbq >> 3) * bn + (cbq & 7) * 2, bsl, tk + q4, ups[0], ups[1], nsl);
                    s_shift[q4 / 4] = make_uchar2((unsigned char)ups[0], (unsigned char)ups[1]);
                }
                tc::tmem_wait_st();
            }
            for (int k = 0; k < K; ++k, ++ord) {
                tc::fence_async_smem();
                tc::fence_before_sync();
                __syncthreads();  // T's digits are in place, D has been read
                tc::fence_after_sync();
                if (warp == 0) {
                    if (tc::elect_one()) {
                        ok = nsl == 6 ? fx_order<6>(m, fpar, !resident || ord == 0, !resident)
                                      : fx_order<7>(m, fpar, !resident || ord == 0, !resident);
                        tc::commit(&done);
                    }
                    __syncwarp();
                } else if (warp == 5) {
                    if (tc::elect_one()) {
                        // this order's stages and the next order's first ones, as slots free up
                        const uint32_t upto = (uint32_t)((ord + 1) * nstage + nst - 1);
                        for (; qp < qend && qp < upto; ++qp) {
                            const uint32_t sl = qp % (uint32_t)nst;
                            if ((epend >> sl) & 1u) {
                                ok = tc::mbar_wait(&empty[sl], (epar >> sl) & 1u, kFxWaitLimit);
                                if (!ok) break;
                                epar ^= 1u << sl;
                                epend ^= 1u << sl;
                            }
                            const int st = (int)(qp % (uint32_t)nstage), kst = f.tiles == 2 ? st >> 1 : st, tl = f.tiles == 2 ? st & 1 : 0;
                            bulk_load(ring + sl * (uint32_t)stage0, ws + (size_t)kst * (stage0 + stage1) + (tl ? stage0 : 0),
                                      (uint32_t)(tl ? stage1 : stage0), &full[sl]);
                            if (!resident) epend |= 1u << sl;
                        }
                    }
                    __syncwarp();
                }
                ok = tc::mbar_wait(&done, norder & 1u, kFxWaitLimit) && ok;
                ++norder;
                if (__syncthreads_or(!ok)) {
                    ok = false;
                    break;
                }
                tc::fence_after_sync();
                if (!wact) continue;  // the whole warp holds rows past N
                // the first order is T_1 = X T_0: half the shifts' values, T_{-1} = 0
                const int fst = k == 0 ? 1 : 0, sL = 3 + fL - fst, ts = fst - 4 - e;
                const Split Jk = s_J[k + 1];
                const bool odd = !(k & 1);
                if (nsl == 6) fx_update<6>(tk, tp, ncol, col0, rowok, dcol, acol, (uint32_t)NB, brow, bn, bsl, Ls, sL, ts, Jk, odd, s_shift);
                else fx_update<7>(tk, tp, ncol, col0, rowok, dcol, acol, (uint32_t)NB, brow, bn, bsl, Ls, sL, ts, Jk, odd, s_shift);
            }
            if (!ok) {
                if (tid == 0) atomicOr(&s.status[t], ST_TC_WAIT);
                break;
            }
            // e^{-ic} of the sum plus the deflated level's share e^{-i mu} a u
            if (wact)
#pragma unroll
                for (int q = 0; q < kFxMaxCols / 2; ++q) {
                    if (2 * q >= ncol) break;
                    float a0, a1, a2, a3;
                    tc::tmem_ld4(acol + 4 * q, a0, a1, a2, a3);
                    tc::tmem_wait_ld();
                    const int el = col0 / 2 + q;
                    if (rowok && el < ne) {
                        const int x = s_x[el], up = q & 1 ? s_shift[q / 2].y : s_shift[q / 2].x;
                        const Split ar = split64(((long long)__float_as_int(a1) << 32) | (uint32_t)__float_as_int(a0));
                        const Split ai = split64(((long long)__float_as_int(a3) << 32) | (uint32_t)__float_as_int(a2));
                        long long outr = mul_shift(cc, ar, 2) + mul_shift(sc, ai, 2);
                        long long outi = mul_shift(cc, ai, 2) - mul_shift(sc, ar, 2);
                        if (defl) {
                            const Split br = s_a1[0][el], bi = s_a1[1][el];
                            const int d = up - s_as[el];
                            outr += mul_unit(br, ur, 3, d) - mul_unit(bi, ui, 3, d);
                            outi += mul_unit(br, ui, 3, d) + mul_unit(bi, ur, 3, d);
                        }
                        const double nan = __longlong_as_double(0x7ff8000000000000ll);
                        C[(int64_t)(e0 + el) * N + row] = x == kNan ? make_double2(nan, nan)
                                                                    : make_double2(double_of(outr, x - 61 - up), double_of(outi, x - 61 - up));
                    }
                }
            __syncthreads();  // the columns' scales are read before the next block's
        }
    }
    // a wait that gave up: let the copies and MMAs in flight land (bounded)
    // before the CTA leaves
    if (!ok) {
        for (int q = 0; q < kFxMaxStages; ++q) {
            tc::mbar_wait(&full[q], 0u, kFxWaitLimit / kFxMaxStages);
            tc::mbar_wait(&full[q], 1u, kFxWaitLimit / kFxMaxStages);
        }
        tc::mbar_wait(&done, norder & 1u, kFxWaitLimit);
    }
    tc::fence_before_sync();
    __syncthreads();
    if (warp == 0) tc::tmem_dealloc(tmem, 512);
}

int fx_sms()
{
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms > 0 ? sms : 1;
}

// Electron ranges per trajectory: one while there are trajectories for every
// SM, else as many as occupy them, of at least 8 electrons (16 real columns,
// the smallest block).
int fx_parts(int Ne, int64_t n, int sms)
{
    const int most = (Ne + 7) / 8;
    int parts = 1;
    while (parts < most && n * (parts + 1) <= sms) ++parts;
    return parts;
}

}  // namespace

// Where the tensor cores pay: measured against the SIMT kernel k_cheb on the
// double well (9 orders) and the relaxation model (20 orders), 2048
// trajectories, Ne = M / 2, ms per step: N = 25 0.84 against 0.66 and 1.65
// against 1.41; N = 29 0.89 against 0.99 and 1.73 against 2.07; N = 41 1.22
// against 2.52 and 2.45 against 5.48.  Its cost per trajectory hardly falls
// with Ne below one block of columns, while the SIMT kernel's is N^2 Ne per
// order: with few electrons the same break-even, N Ne = 28 x 14, holds
// (N = 101, Ne = 4: 1.17 against 2.84; between 2 and 4).  The rule takes N and
// Ne only, so that a batch gives the same bits however it is divided.
bool cheb_fx_eligible(int N, int Ne) { return N >= 28 && N <= 256 && N * Ne >= 28 * 14; }

size_t cheb_fx_work_bytes(int N, int Ne, int64_t max_traj)
{
    if (!cheb_fx_eligible(N, Ne)) return 0;
    const int sms = fx_sms();
    const int64_t items = max_traj * ((Ne + 7) / 8);
    return fx_shape(N).ws * (size_t)(items < sms ? items : sms);
}

void configure_cheb_fx()
{
    cudaFuncSetAttribute(k_cheb_fx, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFxMaxSmem);
    cudaGetLastError();
}

cudaError_t launch_cheb_fx(const DevState &s, double dt, cudaStream_t st)
{
    if (s.n == 0) return cudaSuccess;
    if (!s.fx_work || !cheb_fx_eligible(s.N, s.Ne)) return cudaErrorInvalidValue;
    const FxShape f = fx_shape(s.N);
    const int sms = fx_sms();
    const int parts = fx_parts(s.Ne, s.n, sms);
    const int64_t items = s.n * parts, slots = (int64_t)(s.fx_work_bytes / f.ws);
    int64_t grid = items < sms ? items : sms;
    if (grid > slots) grid = slots;
    if (grid < 1) return cudaErrorInvalidValue;
    k_cheb_fx<<<(unsigned)grid, kFxThreads, kFxMaxSmem, st>>>(s, dt, items, parts, s.fx_work, f.ws);
    return cudaGetLastError();
}

}  // namespace iesh
