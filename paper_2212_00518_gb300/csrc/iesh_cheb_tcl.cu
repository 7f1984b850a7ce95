// iesh_cheb_tcl.cu -- mixed-precision Chebyshev propagator on the tensor cores
// for 128 < N <= 256 (two row tiles).
//
// The exponential integrator of Sec. II C in FP32, as k_cheb_f32t
// (iesh_step.cu): T_{k+1} = 2 X T_k - T_{k-1} with T_k, T_{k-1} and the
// Chebyshev sum in FP32; the contraction (2 / rho) W T_k of every order runs
// as FP16 MMAs with FP32 accumulation.  Both operands are FP32 numbers split
// into FP16 digits of 11 bits (x = x_0 + x_1 + x_2, each the FP16 rounding of
// what is left), scaled so that the largest entry of W' = (2 / rho) W and
// every electron column's norm lie near the top of the FP16 range.  Two digits
// of both operands (three products) hold 24 bits: the amplitude of an empty
// orbital, which W' T makes, then has FP32's accuracy however weak the
// couplings are (one step from unit columns, N = 201: hop probabilities within
// 3e-7 of the largest, as FP32 products give; one digit gave 5e-4).  With |W'| <
// 2^(e+1) the product of digits i and j is about 2^(e - 11 (i + j)) of T, and
// what is left out stays below 2^-28 of a column's norm: three digits (six
// products) from |W'| = 2^-6 up.  The SIMT kernel rounds T_k to 2^-25 of its
// entries.
//
// Two persistent CTAs of 256 threads (one per row) per SM take (trajectory,
// electron range) items in blocks of up to 16 electrons (32 real columns), in
// the layouts of k_cheb_fx (iesh_cheb_fx.cu).  T_k and T_{k-1} are in registers
// (32 values each per thread), the product and the Chebyshev sum in tensor
// memory, T's digits in shared memory.  W' is cut into digits once per item:
// where they fit (N up to about 135) straight into shared memory, where they
// stay for all blocks and orders; otherwise into the CTA's slot of a workspace
// that stays in L2, streamed back by bulk copies through a ring of two or three
// slots of several K steps.
//
// What bounds it: the chain of an order -- barrier, MMAs (78 of 128 x 32 x 16
// at N = 201, 41 cycles each), commit, wait, update of the registers and
// digits -- of two CTAs that fill each other's waits.  Measured at N = 201,
// Ne = 100, 8192 trajectories, 5 orders: 17.0 ms per step for the SIMT kernel
// (50% of the FP32 peak) -> 8.4 ms (7.35 with one digit, 11.8 with three, which
// is not more accurate).  One CTA of 512 threads per SM took 17.6 ms
// with a commit per K step and row tile, 10.9 ms with several K steps per slot.
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "iesh_common.cuh"
#include "iesh_kernels.h"
#include "iesh_tc.cuh"

namespace iesh {

namespace {

constexpr int kTlThreads = 256;       // a thread per row
constexpr int kTlWarps = kTlThreads / 32;
constexpr int kTlS = 3;               // digits of each operand
constexpr int kTlMaxCols = 32;        // real columns of a block
constexpr int kTlMaxEl = 16;          // electrons of a block
constexpr int kTlWaitLimit = 1 << 22;
constexpr int kTlMaxStages = 16;
constexpr size_t kTlMaxSmem = 104 * 1024;  // two CTAs per SM

// Sizes: rg 8-row groups of W in two row tiles of 128 rows, ks K steps of 16.
struct TlShape {
    int Kp, ks, rg;
    size_t ws;    // workspace bytes of a CTA
};
__host__ __device__ inline TlShape tl_shape(int N)
{
    TlShape f;
    f.Kp = (N + 15) & ~15;
    f.ks = f.Kp / 16;
    f.rg = (N + 7) / 8;
    f.ws = (size_t)f.ks * kTlS * f.rg * 256;
    return f;
}

__device__ __forceinline__ void bulk_load(uint32_t dst, const void *src, uint32_t bytes, uint64_t *mbar)
{
    const uint32_t mb = tc::smem_addr(mbar);
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mb), "r"(bytes) : "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(mb)
                 : "memory");
}
// What the issuing thread needs about an item, as FxMma of iesh_cheb_fx.cu.
struct TlMma {
    uint64_t ad0, bd0;
    uint64_t *full, *empty;
    uint32_t slot, nst, ks, kps, kstep, tstep, da0, da1, db, d0, idesc;
};

// The MMAs of one order: for every K step and row tile all pairs i + j < NSL
// into one accumulator per row tile, unrolled, issued by one thread.
template <int NSL>
__device__ __forceinline__ bool tl_order(TlMma &m, uint32_t &fpar, bool ring)
{
    uint64_t bd = m.bd0;
    uint32_t sl = m.slot;
    for (uint32_t k0 = 0; k0 < m.ks; k0 += m.kps) {
        if (ring) {
            if (!tc::mbar_wait(&m.full[sl], (fpar >> sl) & 1u, kTlWaitLimit)) return false;
            fpar ^= 1u << sl;
        }
        uint64_t ak = m.ad0 + sl * (m.kps * m.kstep);
        const uint32_t k1 = min(m.ks, k0 + m.kps);
#pragma unroll 1
        for (uint32_t k = k0; k < k1; ++k, ak += m.kstep, bd += 16)
#pragma unroll
            for (int tl = 0; tl < 2; ++tl)
#pragma unroll
                for (int i = 0; i < NSL; ++i)
#pragma unroll
                    for (int j = 0; j < NSL - i; ++j)
                        tc::mma_f16(m.d0 + tl * kTlMaxCols, ak + tl * m.tstep + i * (tl ? m.da1 : m.da0), bd + j * m.db, m.idesc,
                                    i == 0 && j == 0 ? (k ? 1u : 0u) : 1u);
        if (ring) tc::commit(&m.empty[sl]);
        sl = sl + 1 == m.nst ? 0u : sl + 1;
    }
    m.slot = sl;
    return true;
}

// FP16 digits of a pair: the FP16 rounding of what is left, three times.
__device__ __forceinline__ void digits2(float x, float y, uint32_t *d, int n)
{
#pragma unroll
    for (int i = 0; i < kTlS; ++i)
        if (i < n) {
            const __half2 h = __floats2half2_rn(x, y);
            d[i] = *reinterpret_cast<const uint32_t *>(&h);
            const float2 f = __half22float2(h);
            x -= f.x;
            y -= f.y;
        }
}
// Digits of eight columns of T (scaled) into the B operand.
__device__ __forceinline__ void tl_put(unsigned char *b, int bsl, const float *t, int nsl)
{
    uint32_t d[4][kTlS];
#pragma unroll
    for (int q = 0; q < 4; ++q) digits2(t[2 * q], t[2 * q + 1], d[q], nsl);
#pragma unroll
    for (int i = 0; i < kTlS; ++i)
        if (i < nsl) *reinterpret_cast<uint4 *>(b + i * bsl) = make_uint4(d[0][i], d[1][i], d[2][i], d[3][i]);
}

__global__ void __launch_bounds__(kTlThreads, 2)
    k_cheb_tcl(DevState s, double dt, int64_t items, int parts, unsigned char *ws_all, size_t ws_stride, int dfl)
{
    extern __shared__ __align__(1024) unsigned char tl_smem[];
    __shared__ __align__(8) uint64_t full[kTlMaxStages], empty[kTlMaxStages], done;
    __shared__ uint32_t tmem_slot;
    __shared__ int s_red[kTlWarps], s_max[kTlMaxEl];
    __shared__ float s_cj[kChebMax], s_sc[4];
    __shared__ float2 s_a[kTlMaxEl];
    const int N = s.N, Ne = s.Ne, Np = (N + 3) & ~3;
    const TlShape f = tl_shape(N);
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int tile = warp >> 2, row = tid;
    const bool rowok = row < N, wact = row - lane < N;
    unsigned char *ws = ws_all + (size_t)blockIdx.x * ws_stride;
    if (tid == 0) {
        for (int q = 0; q < kTlMaxStages; ++q) {
            tc::mbar_init(&full[q], 1);
            tc::mbar_init(&empty[q], 1);
        }
        tc::mbar_init(&done, 1);
    }
    if (warp == 0) tc::tmem_alloc(&tmem_slot, 128);
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
        const float *Wf = reinterpret_cast<const float *>(s.scratch + t * s.scratch_stride);  // [N][Np]
        float2 *C = reinterpret_cast<float2 *>(s.C) + (int64_t)t * Ne * N;
        const double w2d = rho > 0.0 ? 2.0 / rho : 0.0;
        const float w2 = (float)w2d;
        const double *df = dfl ? s.defl + t * defl_stride(N, Ne) : nullptr;
        const bool defl = df && df[0] != 0.0;
        const float *dq = reinterpret_cast<const float *>(df + kDeflHead);  // u, then a
        float ur = 0.f, ui = 0.f;
        if (defl && rowok) {
            ur = dq[row];
            ui = dq[N + row];
        }

        // exponent of max |W'|
        int mx = 0;
#pragma unroll 8
        for (int idx = tid; idx < N * Np / 4; idx += kTlThreads) {
            const int4 w = reinterpret_cast<const int4 *>(Wf)[idx];
            mx = max(max(mx, w.x & 0x7fffffff), w.y & 0x7fffffff);
            mx = max(max(mx, w.z & 0x7fffffff), w.w & 0x7fffffff);
        }
        mx = __reduce_max_sync(0xffffffffu, mx);
        if (lane == 0) s_red[warp] = mx;
        if (tid < kTlMaxEl) s_max[tid] = 0;
        for (int k = tid; k <= K; k += kTlThreads) s_cj[k] = (float)((k ? 2.0 : 1.0) * cb[3 + k]);
        if (tid == 0) {
            double sn, cs;
            sincos(c, &sn, &cs);
            s_sc[0] = (float)sn;
            s_sc[1] = (float)cs;
            s_sc[2] = defl ? (float)df[3] : 0.f;  // e^{-i mu}
            s_sc[3] = defl ? (float)df[2] : 1.f;
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < kTlWarps; ++q) mx = max(mx, s_red[q]);
        const float wmax = __int_as_float(mx) * w2;
        // W' = 2^e Wn, |Wn| < 2 (not finite: e = 0, and NaN in every column)
        int e = (int)((__float_as_int(wmax) >> 23) & 0xff) - 127;
        if (e > 100) e = 0;
        if (e < -60) e = -60;
        const int nsl = e >= -6 ? kTlS : 2;
        const float ws_scale = w2 * __int_as_float((127 + 13 - e) << 23);  // digits of 2^(13 - e) W'
        const float dscale = __int_as_float((127 + e - 27) << 23);         // D of 2^14 T from the accumulator: 2^(e - 13)
        const float d14 = dscale * 16384.0f;
        const float Lc = rowok ? (float)(w2d * (0.5 * dt * (s.lam_prev[t * N + row] + s.lam[t * N + row]) - c)) : 0.0f;
        // blocks of the item's electrons
        const int cap = s.cheb_ept > 0 ? min(kTlMaxEl, 4 * s.cheb_G) : kTlMaxEl;  // (a requested shape)
        const int eb = cap, nblk = (e_hi - e_lo + eb - 1) / eb;
        const int NB0 = (2 * min(eb, e_hi - e_lo) + 15) & ~15;  // columns of a full block
        const int bn = (f.Kp / 8) * 128, bsl = (NB0 / 8) * bn;  // bytes of 8 columns, of a digit of T
        const int stage0 = nsl * 16 * 256, stage1 = nsl * (f.rg - 16) * 256;
        // the ring: kps K steps per slot; all of W' where it fits (loaded once
        // per item), else three slots, or two
        const int kb = stage0 + stage1, avail = (int)kTlMaxSmem - nsl * bsl;
        const bool resident = f.ks * kb <= avail;
        const int kps = resident ? (f.ks + 3) / 4 : max(1, avail / (3 * kb));
        const int nstage = (f.ks + kps - 1) / kps;  // stages per order
        const int nst = resident ? nstage : min(nstage, avail / (kps * kb));
        // (an MMA reads 16 row groups from a digit's start: past the ring, T's
        // digits, into rows that are not used)
        const uint32_t ring = tc::smem_addr(tl_smem);
        unsigned char *B = tl_smem + min(nst * kps, f.ks) * kb;
        // digits of W': A[j][i] = W_ji = -W_ij, consecutive threads on
        // consecutive rows j
        {
            unsigned char *wd = resident ? tl_smem : ws;
            const int rows = 8 * f.rg, units = rows * (f.Kp / 8);
#pragma unroll 2
            for (int it = tid; it < units; it += kTlThreads) {
                const int kc = it / rows, r = it - kc * rows;
                uint32_t h[kTlS][4];
#pragma unroll
                for (int q2 = 0; q2 < 4; ++q2) {
                    float v[2];
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        const int k = 8 * kc + 2 * q2 + q;
                        v[q] = (r < N && k < N) ? -ws_scale * Wf[(int64_t)k * Np + r] : 0.0f;
                    }
                    uint32_t d[kTlS] = {0, 0, 0};
                    digits2(v[0], v[1], d, nsl);
#pragma unroll
                    for (int i = 0; i < kTlS; ++i) h[i][q2] = d[i];
                }
                const int tl = r >> 7, rgt = tl ? f.rg - 16 : 16;
                unsigned char *dst = wd + (kc >> 1) * kb + (tl ? stage0 : 0) + ((r & 127) >> 3) * 256 +
                                     (kc & 1) * 128 + (r & 7) * 16;
#pragma unroll
                for (int i = 0; i < kTlS; ++i)
                    if (i < nsl) *reinterpret_cast<uint4 *>(dst + (size_t)i * rgt * 256) = make_uint4(h[i][0], h[i][1], h[i][2], h[i][3]);
            }
        }
        if (!resident) asm volatile("fence.proxy.async;" ::: "memory");  // the bulk copies read what was just written
        // T's digits: rows past N stay zero
        for (int w = tid; w < nsl * bsl / 16; w += kTlThreads) reinterpret_cast<uint4 *>(B)[w] = make_uint4(0, 0, 0, 0);
        const uint32_t dcol = my_lane + (uint32_t)(tile * kTlMaxCols);
        const uint32_t acol = my_lane + (uint32_t)((2 + tile) * kTlMaxCols);
        unsigned char *brow = B + (row >> 3) * 128 + (row & 7) * 16;
        uint32_t qp = 0;  // stages copied in this item
        TlMma m;
        m.ad0 = tc::smem_desc(ring, 128, 256);
        m.bd0 = tc::smem_desc(tc::smem_addr(B), 128, (uint32_t)bn);
        m.full = full, m.empty = empty;
        m.slot = 0, m.nst = (uint32_t)nst, m.ks = (uint32_t)f.ks, m.kps = (uint32_t)kps;
        m.kstep = (uint32_t)kb / 16u, m.tstep = (uint32_t)stage0 / 16u;
        m.da0 = 16u * 16u, m.da1 = (uint32_t)(f.rg - 16) * 16u;
        m.db = (uint32_t)bsl / 16u, m.d0 = tmem;
        const uint32_t qend = resident ? 0u : (uint32_t)(nblk * K * nstage);
        int ord = 0;  // orders of this item
        // log2 of the scale of a column with largest entry mm: its norm is below
        // 2 sqrt(N / 2) 2^exponent
        auto col_log2 = [](int mm) { return mm == 0 || mm >= 0x7f800000 ? 0 : max(-100, min(100, (mm >> 23) - 122)); };

        for (int blk = 0; blk < nblk && ok; ++blk) {
            const int e0 = e_lo + blk * eb, ne = min(eb, e_hi - e0);
            const int ncol = (2 * ne + 15) & ~15;
            m.idesc = tc::idesc_f16(128, ncol) | (1u << 16);
            float tk[kTlMaxCols], tp[kTlMaxCols];  // in the unit 2^-14 of the column's scale
#pragma unroll
            for (int q = 0; q < kTlMaxCols / 2; ++q) {
                float2 v = make_float2(0.f, 0.f);
                if (rowok && q < ne) v = C[(int64_t)(e0 + q) * N + row];
                tk[2 * q] = v.x;
                tk[2 * q + 1] = v.y;
            }
            if (defl && tid < ne) s_a[tid] = make_float2(dq[2 * N + e0 + tid], dq[2 * N + Ne + e0 + tid]);
            __syncthreads();  // (s_max is zero)
            if (wact) {
                int mm[kTlMaxEl];
#pragma unroll
                for (int q = 0; q < kTlMaxEl; ++q)
                    mm[q] = __reduce_max_sync(0xffffffffu, max(__float_as_int(tk[2 * q]) & 0x7fffffff,
                                                               __float_as_int(tk[2 * q + 1]) & 0x7fffffff));
                int mine = 0;
#pragma unroll
                for (int q = 0; q < kTlMaxEl; ++q) mine = lane == q ? mm[q] : mine;
                if (lane < kTlMaxEl) atomicMax(&s_max[lane], mine);
            }
            if (defl)  // c - a u (the scales are those of c: the share along u grows)
#pragma unroll
                for (int q = 0; q < kTlMaxCols / 2; ++q)
                    if (rowok && q < ne) {
                        const float2 a = s_a[q];
                        tk[2 * q] -= fmaf(a.x, ur, -(a.y * ui));
                        tk[2 * q + 1] -= fmaf(a.x, ui, a.y * ur);
                    }
            __syncthreads();
            if (wact) {
                const float J0 = s_cj[0];
#pragma unroll
                for (int q8 = 0; q8 < kTlMaxCols; q8 += 8) {
                    if (q8 >= ncol) break;
                    float a[8];
#pragma unroll
                    for (int h = 0; h < 8; ++h) {
                        const int el = (q8 + h) / 2;
                        const float sc = __int_as_float((127 + 14 - col_log2(s_max[el])) << 23);
                        tk[q8 + h] *= sc;
                        tp[q8 + h] = 0.f;
                        a[h] = J0 * tk[q8 + h];
                    }
                    tc::tmem_st8(acol + q8, a);
                    if (rowok) tl_put(brow + (q8 >> 3) * bn, bsl, tk + q8, nsl);
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
                        ok = nsl == 2 ? tl_order<2>(m, fpar, !resident) : tl_order<3>(m, fpar, !resident);
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
                                ok = tc::mbar_wait(&empty[sl], (epar >> sl) & 1u, kTlWaitLimit);
                                if (!ok) break;
                                epar ^= 1u << sl;
                                epend ^= 1u << sl;
                            }
                            const int k0 = (int)(qp % (uint32_t)nstage) * kps;
                            bulk_load(ring + sl * (uint32_t)(kps * kb), ws + (size_t)k0 * kb,
                                      (uint32_t)(min(kps, f.ks - k0) * kb), &full[sl]);
                            if (!resident) epend |= 1u << sl;
                        }
                    }
                    __syncwarp();
                }
                ok = tc::mbar_wait(&done, norder & 1u, kTlWaitLimit) && ok;
                ++norder;
                if (__syncthreads_or(!ok)) {
                    ok = false;
                    break;
                }
                tc::fence_after_sync();
                if (!wact) continue;  // the whole warp holds rows past N
                const float cj = s_cj[k + 1];
                const int ph = (k + 1) & 3;  // (-i)^(k+1) = (1, 0), (0, -1), (-1, 0), (0, 1)
                const float cs = ph >= 2 ? -cj : cj;
                const bool odd = ph & 1;
                const float hf = k == 0 ? 0.5f : 1.0f;  // T_1 = X T_0
                const float Lh = hf * Lc, dh = hf * d14;
#pragma unroll
                for (int q8 = 0; q8 < kTlMaxCols; q8 += 8) {
                    if (q8 >= ncol) break;
                    float d[8], a[8];
                    tc::tmem_ld8(dcol + q8, d);
                    tc::tmem_ld8(acol + q8, a);
                    float n[8];
#pragma unroll
                    for (int h = 0; h < 8; ++h) n[h] = fmaf(Lh, tk[q8 + h], -tp[q8 + h]);
                    tc::tmem_wait_ld();
#pragma unroll
                    for (int h = 0; h < 8; h += 2) {
                        // 2 (X t)_j = 2 ((L_j - c) t_j - i (W t)_j) / rho
                        const float nr = fmaf(d[h + 1], dh, n[h]), ni = fmaf(-d[h], dh, n[h + 1]);
                        tp[q8 + h] = tk[q8 + h];
                        tp[q8 + h + 1] = tk[q8 + h + 1];
                        tk[q8 + h] = nr;
                        tk[q8 + h + 1] = ni;
                        a[h] = fmaf(cs, odd ? ni : nr, a[h]);
                        a[h + 1] = fmaf(odd ? -cs : cs, odd ? nr : ni, a[h + 1]);
                    }
                    tc::tmem_st8(acol + q8, a);
                    if (rowok) tl_put(brow + (q8 >> 3) * bn, bsl, tk + q8, nsl);
                }
                tc::tmem_wait_st();
            }
            if (!ok) {
                if (tid == 0) atomicOr(&s.status[t], ST_TC_WAIT);
                break;
            }
            // e^{-ic} of the sum plus the deflated level's share e^{-i mu} a u
            if (wact) {
                const float sc = s_sc[0], cc = s_sc[1];
                const float sm = s_sc[2], cm = s_sc[3];
#pragma unroll
                for (int q8 = 0; q8 < kTlMaxCols; q8 += 8) {
                    if (q8 >= ncol) break;
                    float a[8];
                    tc::tmem_ld8(acol + q8, a);
                    tc::tmem_wait_ld();
#pragma unroll
                    for (int h = 0; h < 4; ++h) {
                        const int el = q8 / 2 + h;
                        if (rowok && el < ne) {
                            const float us = __int_as_float((127 - 14 + col_log2(s_max[el])) << 23);
                            const float ar = us * a[2 * h], ai = us * a[2 * h + 1];
                            float2 o = make_float2(fmaf(cc, ar, sc * ai), fmaf(cc, ai, -(sc * ar)));
                            if (defl) {
                                const float2 a2 = s_a[el];
                                const float br = fmaf(a2.x, ur, -(a2.y * ui)), bi = fmaf(a2.x, ui, a2.y * ur);  // a u_j
                                o.x += fmaf(cm, br, sm * bi);
                                o.y += fmaf(cm, bi, -(sm * br));
                            }
                            C[(int64_t)(e0 + el) * N + row] = o;
                        }
                    }
                }
            }
            __syncthreads();  // the columns' scales are read before they are reset for the next block
            if (tid < kTlMaxEl) s_max[tid] = 0;
        }
    }
    // a wait that gave up: let the copies and MMAs in flight land (bounded)
    // before the CTA leaves
    if (!ok) {
        for (int q = 0; q < kTlMaxStages; ++q) {
            tc::mbar_wait(&full[q], 0u, kTlWaitLimit / kTlMaxStages);
            tc::mbar_wait(&full[q], 1u, kTlWaitLimit / kTlMaxStages);
        }
        tc::mbar_wait(&done, norder & 1u, kTlWaitLimit);
    }
    tc::fence_before_sync();
    __syncthreads();
    if (warp == 0) tc::tmem_dealloc(tmem, 128);
}

int tl_sms()
{
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms > 0 ? sms : 1;
}

}  // namespace

// Few electrons: cutting W' costs as much as the SIMT kernel's whole product.
// Measured per step at 2048 trajectories, SIMT -> tensor cores: N = 131: Ne = 12
// .320 -> .325 ms, 16 .428 -> .333; N = 201: Ne = 4 .367 -> .360, 6 .515 ->
// .367, 12 .750 -> .449; N = 255: Ne = 8 .892 -> .599.  The rule takes N and Ne only, so
// that a batch gives the same bits however it is divided.
bool cheb_tcl_eligible(int N, int Ne) { return N > 128 && N <= 256 && (Ne >= 16 || (N >= 192 && Ne >= 6)); }

size_t cheb_tcl_work_bytes(int N, int Ne, int64_t max_traj)
{
    if (!cheb_tcl_eligible(N, Ne)) return 0;
    const int sms = tl_sms();
    const int64_t items = max_traj * ((Ne + 7) / 8);
    return tl_shape(N).ws * (size_t)(items < 2 * sms ? items : 2 * sms);
}

void configure_cheb_tcl()
{
    cudaFuncSetAttribute(k_cheb_tcl, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTlMaxSmem);
    cudaGetLastError();
}

cudaError_t launch_cheb_tcl(const DevState &s, double dt, cudaStream_t st)
{
    if (s.n == 0) return cudaSuccess;
    if (!s.fx_work || !cheb_tcl_eligible(s.N, s.Ne)) return cudaErrorInvalidValue;
    const TlShape f = tl_shape(s.N);
    const int sms = tl_sms(), most = (s.Ne + 7) / 8;
    // electron ranges per trajectory: as many as occupy the SMs in a small batch
    int parts = 1;
    while (parts < most && s.n * (parts + 1) <= 2 * sms) ++parts;
    const int64_t items = s.n * parts, slots = (int64_t)(s.fx_work_bytes / f.ws);
    int64_t grid = items < 2 * sms ? items : 2 * sms;
    if (grid > slots) grid = slots;
    if (grid < 1) return cudaErrorInvalidValue;
    k_cheb_tcl<<<(unsigned)grid, kTlThreads, kTlMaxSmem, st>>>(s, dt, items, parts, s.fx_work, f.ws, mixed_deflates(s) ? 1 : 0);
    return cudaGetLastError();
}

}  // namespace iesh
