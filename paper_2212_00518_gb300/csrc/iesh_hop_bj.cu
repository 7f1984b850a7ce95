// iesh_hop_bj.cu -- hop probabilities of the mixed-precision path by blocked
// Gauss-Jordan column elimination in shared memory.
//
// The candidate that puts orbital m in slot a has amplitude det S *
// R_{m a}, R = C_u S^{-1} (Sec. II B, determinant ratios).  Right-multiplying
// the N x Ne matrix Z = C^T (Z_{o e} = C_e(o): the rows of the occupied
// orbitals form S, the others C_u) by S^{-1} turns the S rows into the
// identity and leaves R in the unoccupied rows.  Eliminating slot i's
// orbital s_i chooses the pivot column j among the columns not chosen yet by
// the largest |Z_{s_i j}| (partial pivoting); after all Ne slots column j(i)
// belongs to slot i: R_{m i} = Z_{m j(i)}.
//
// The slots are eliminated four at a time.  One warp takes the block's four
// rows P of Z (4 x Ne, in registers) through an in-place Gauss-Jordan row
// elimination, pivots chosen as above: with J the four pivot columns it
// ends with P_J^{-1} P outside J and P_J^{-1} inside, which are (up to sign)
// the rows M of the column transformation,
//   Z' = Z (columns J zeroed) + Z_J M,
// and the whole CTA then applies that rank-4 update, tile by tile in
// registers: four complex rank-one updates per pass over Z, in packed FP32
// pairs, and three barriers per four slots.  One pivot per barrier (k_hop_gj) leaves the SM
// waiting for each slot's pivot search.  Measured, ms per step: N = 51, Ne =
// 25, 1821 trajectories 0.185 -> 0.083 (k_hop_gj before); the limits of its
// range stand at hop_bj_eligible.  Also measured at N = 101: blocks of eight
// with scalar FMAs 0.84, Z in registers with the panels one block ahead in a
// warp of their own 1.0, against k_hop_gj's 0.775.
//
// FP32 throughout (the coefficients are FP32 in the mixed path), the
// couplings d_{m, s_a} included: their numerators from lam - h rounded once
// from FP64, their eigenvalue gaps from double-float (hi, lo) eigenvalues, so
// nearly degenerate pairs keep FP32 relative accuracy.  The running sum of
// the selection is exact in 64-bit integers of 2^-60 (each probability
// counted up to 1, where every uniform lies below): an FP64 instruction
// takes a warp 64 cycles of its scheduler, conversions included.  The
// rescale is FP64 as in k_hop.  The skip bound of Sec. II C saves no work
// here (the elimination is the ratio solve) and is not applied; hop
// decisions are the same either way.
#include <cuda_runtime.h>
#include <stdint.h>

#include "iesh_common.cuh"
#include "iesh_hop.cuh"
#include "iesh_kernels.h"

namespace iesh {

namespace {

constexpr int kBjB = 4;            // slots per block
constexpr int kBjRPT = 4;          // rows per thread: tr + TR k, TR = ceil(N / 4)
constexpr int kBjTC = 8;           // column classes: tc + 8 q within a pass
constexpr int kBjZs = kBjB + 1;    // row stride of the pivot columns (conflict-free 16-byte reads)
constexpr int kBjMaxN = 96, kBjMaxNe = 48, kBjMaxThreads = 192;

// Sizes: g8 groups of 8 columns, row stride CP = 8 (mod 16) entries (two rows
// of a half warp's 64-byte reads fall on distinct banks).
struct BjShape {
    int TR, threads, g8, CP;
    size_t z, zj, pm, orb, part, total;  // bytes of Z, Z_J, P and M, orbital data, slot sums
};
__host__ __device__ inline BjShape bj_shape(int N, int Ne, bool ext)
{
    BjShape b;
    b.TR = (N + kBjRPT - 1) / kBjRPT;
    b.threads = (b.TR * kBjTC + 31) & ~31;
    if (b.threads < 128) b.threads = 128;  // (the panel's warp is one of four)
    b.g8 = (Ne + 7) / 8;
    b.CP = 8 * b.g8;
    if (b.CP % 16 != 8) b.CP += 8;
    b.z = (size_t)N * b.CP * sizeof(float2);
    b.zj = (size_t)kBjRPT * b.TR * kBjZs * sizeof(float4);
    b.pm = (size_t)kBjB * b.CP * sizeof(float4);
    b.orb = (size_t)(N + b.CP) * (ext ? 6 : 4) * sizeof(float);
    b.part = (size_t)(b.threads / 32) * b.CP * sizeof(long long);
    b.orb = (b.orb + 15) & ~(size_t)15;
    // the slot sums reuse Z_J and M (the elimination is over)
    const size_t tail = b.zj + b.pm > b.part ? b.zj + b.pm : b.part;
    b.total = b.z + tail + b.orb;
    return b;
}

// A probability as an integer of 2^-60, counted up to 1.
__device__ __forceinline__ long long prob_fixed(float g)
{
    if (!(g > 0.f)) return 0;
    if (g >= 1.f) return 1ll << 60;
    const int b = __float_as_int(g), sh = (b >> 23) - 150 + 60;
    const long long m = (b & 0x7fffff) | 0x800000;
    return sh >= 0 ? m << sh : (sh > -25 ? m >> -sh : 0);
}
__device__ __forceinline__ long long sat1(long long v) { return v < (1ll << 60) ? v : 1ll << 60; }

// 1/a of a complex pivot: the FP32 reciprocal of |a|^2 with a Newton step.
__device__ __forceinline__ float2 bj_rcp(float2 a)
{
    const float m = fmaf(a.x, a.x, a.y * a.y);
    // |a|^2 outside the estimate's range: the division
    const float d = m > 1e-30f && m < 1e30f ? pole_recip<float>(m) : 1.0f / m;
    return make_float2(a.x * d, -a.y * d);
}

// Packed pairs of FP32 (re, im): one instruction for two FMAs, which halves
// the issue slots of a complex rank-one update,
//   u += w m = (w.x, w.x) (m.x, m.y) + (w.y, w.y) (-m.y, m.x).
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c)
{
    f32x2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ f32x2 pack2(float x, float y)
{
    f32x2 d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(x), "f"(y));
    return d;
}
__device__ __forceinline__ float2 unpack2(f32x2 v)
{
    float2 d;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(d.x), "=f"(d.y) : "l"(v));
    return d;
}

// Z += Z_J M on rows tr + TR k and columns c0 + 8 q: zj holds (x, x, y, y) of
// the pivot columns' entries, M (x, y, -y, x) of the transformation's.
template <int CPT>
__device__ __forceinline__ void bj_update(f32x2 *Z, const ulonglong2 *zj, const ulonglong2 *M, int N, int TR, int CP, int tr,
                                          int c0)
{
    f32x2 v[kBjRPT][CPT];
#pragma unroll
    for (int k = 0; k < kBjRPT; ++k)
#pragma unroll
        for (int q = 0; q < CPT; ++q) {
            const int r = tr + TR * k;
            v[k][q] = r < N ? Z[r * CP + c0 + kBjTC * q] : 0ull;
        }
#pragma unroll
    for (int kk = 0; kk < kBjB; ++kk) {
        ulonglong2 w[kBjRPT];
#pragma unroll
        for (int k = 0; k < kBjRPT; ++k) w[k] = zj[(tr + TR * k) * kBjZs + kk];
#pragma unroll
        for (int q = 0; q < CPT; ++q) {
            const ulonglong2 m = M[kk * CP + c0 + kBjTC * q];
#pragma unroll
            for (int k = 0; k < kBjRPT; ++k) v[k][q] = fma2(w[k].x, m.x, fma2(w[k].y, m.y, v[k][q]));
        }
    }
#pragma unroll
    for (int k = 0; k < kBjRPT; ++k)
#pragma unroll
        for (int q = 0; q < CPT; ++q) {
            const int r = tr + TR * k;
            if (r < N) Z[r * CP + c0 + kBjTC * q] = v[k][q];
        }
}

template <bool EXT>
__global__ void __launch_bounds__(kBjMaxThreads, 4) k_hop_bj(DevState s, double dt, double mass, uint64_t seed, double *g_out)
{
    constexpr int CPW = 2;  // panel columns per lane
    constexpr unsigned kFull = 0xffffffffu;
    extern __shared__ __align__(16) unsigned char bj_smem[];
    const int64_t t = traj_of(s, blockIdx.x);
    if (t < 0 || (s.status[t] & ST_DONE)) return;
    const int N = s.N, Ne = s.Ne, nthr = blockDim.x;
    const BjShape b = bj_shape(N, Ne, EXT);
    const int TR = b.TR, CP = b.CP;
    const int tid = threadIdx.x, tr = tid >> 3, tc = tid & 7, lane = tid & 31, warp = tid >> 5, nwarp = nthr >> 5;
    const bool act = tr < TR;
    float2 *Z = reinterpret_cast<float2 *>(bj_smem);                 // [N][CP]
    float4 *zj = reinterpret_cast<float4 *>(bj_smem + b.z);          // [4 TR][kBjZs] pivot columns (x, x, y, y)
    float4 *M = reinterpret_cast<float4 *>(bj_smem + b.z + b.zj);    // [4][CP] the transformation (x, y, -y, x)
    long long *part = reinterpret_cast<long long *>(bj_smem + b.z);  // [warps][CP] slot sums (afterwards)
    // FP32 coupling data per orbital, then per column (of its slot's orbital):
    // adsorbate component, lam - h, lam as (hi, lo); EXT: the other orbital's
    float4 *od = reinterpret_cast<float4 *>(bj_smem + b.total - b.orb);  // [N + CP]
    float2 *od2 = reinterpret_cast<float2 *>(od + N + CP);                // [N + CP] (EXT)
    __shared__ double red[64];
    __shared__ int occ_s[kBjMaxNe], slot_of[kBjMaxNe + 8], col_of[kBjMaxNe], s_J[kBjB], s_hop_a, s_hop_m, s_sing;
    __shared__ unsigned occ_bits[kBjMaxN / 32];
    __shared__ float s_fac[5];
    __shared__ long long s_zeta;
    const double *gv = EXT ? s.geo2 + t * 8 : s.geo + t * 4;  // h, h', kappa (EXT: h_0, h_1, projections)

    // Z = C^T, zero columns past Ne: a warp takes 4 rows of 8 columns (whole
    // 32-byte sectors of C, no bank conflicts in Z)
    const float2 *Ct = reinterpret_cast<const float2 *>(s.C) + (int64_t)t * Ne * N;
    for (int c0 = 0; c0 < CP; c0 += 8) {
        const int c = c0 + (lane >> 2);
#pragma unroll 4
        for (int r = 4 * warp + (lane & 3); r < N; r += 4 * nwarp)
            Z[r * CP + c] = c < Ne ? Ct[(int64_t)c * N + r] : make_float2(0.f, 0.f);
    }
    if (tid < kBjMaxN / 32) occ_bits[tid] = 0;
    if (tid == 0) {
        s_hop_a = -1;
        s_hop_m = -1;
        s_sing = 0;
        // -2 dt v (the six-coordinate coupling carries its velocity) and the
        // numerators' factors h' + kappa (.) (EXT: the two orbitals' projections)
        const double v = EXT ? 1.0 : s.p[t] / mass;
        s_fac[0] = (float)(-2.0 * dt * v);
        s_fac[1] = (float)(EXT ? gv[2] : gv[1]);
        s_fac[2] = (float)(EXT ? gv[4] : gv[2]);
        s_fac[3] = (float)(EXT ? gv[3] : 0.0);
        s_fac[4] = (float)(EXT ? gv[5] : 0.0);
    }
    if (tid == nthr - 1) {  // the uniform, 53 bits, in units of 2^-60
        const U4 rn = draw_traj(s, seed, t, kStreamHop, (uint64_t)s.nstep[t]);
        s_zeta = (((long long)(rn.v[0] >> 5) << 26) | (rn.v[1] >> 6)) << 7;
    }
    __syncthreads();
    for (int a = tid; a < Ne; a += nthr) {
        const int o = s.occ[t * Ne + a];
        occ_s[a] = o;
        atomicOr(&occ_bits[o >> 5], 1u << (o & 31));
    }
    const double h0 = gv[0], h1 = EXT ? gv[1] : 0.0;
    for (int i = tid; i < N; i += nthr) {
        const double l = s.lam[t * N + i];
        const float lh = (float)l;
        od[i] = make_float4((float)s.q0[t * N + i], (float)(l - h0), lh, (float)(l - (double)lh));
        if constexpr (EXT) od2[i] = make_float2((float)s.q2[t * N + i], (float)(l - h1));
    }
    __syncthreads();

    // ---- elimination, four slots per block, three barriers
    // the panel's warp: CTAs of one SM take warps of different schedulers
    const int pw = (int)(blockIdx.x & 3u);
    unsigned used = 0;  // warp pw: bit h: panel column lane + 32 h is a pivot column already
    bool singular = false;
    f32x2 *Z2 = reinterpret_cast<f32x2 *>(Z);
    const ulonglong2 *zj2 = reinterpret_cast<const ulonglong2 *>(zj), *M2 = reinterpret_cast<const ulonglong2 *>(M);
    for (int i0 = 0; i0 < Ne; i0 += kBjB) {
        const int nb = min(kBjB, Ne - i0);
        if (warp == pw) {
            f32x2 a[kBjB][CPW];
#pragma unroll
            for (int r = 0; r < kBjB; ++r) {
                const f32x2 *row = reinterpret_cast<const f32x2 *>(Z) + (r < nb ? occ_s[i0 + r] : 0) * CP;
#pragma unroll
                for (int h = 0; h < CPW; ++h) {
                    const int c = lane + 32 * h;
                    a[r][h] = (r < nb && c < CP) ? row[c] : 0ull;
                }
            }
            unsigned mine = 0;  // bit h: a pivot column of this block
            int ok = 1;
#pragma unroll
            for (int i = 0; i < kBjB; ++i) {
                if (i < nb && ok) {  // uniform
                    // the largest entry among the free columns: |.| to 15
                    // mantissa bits with the column below it (lower columns win)
                    int best = 0;
#pragma unroll
                    for (int h = 0; h < CPW; ++h) {
                        const int key = pivot_key(unpack2(a[i][h]));
                        if (key > 0xff && !((used >> h) & 1u)) best = max(best, (key & ~0xff) | (255 - (lane + 32 * h)));
                    }
                    const int m = __reduce_max_sync(kFull, best);
                    if (m <= 0) {  // the row is zero in every free column
                        ok = 0;
                    } else {
                        const int j = 255 - (m & 0xff), jl = j & 31, jh = j >> 5;
                        float2 f[kBjB];
#pragma unroll
                        for (int r = 0; r < kBjB; ++r) {
                            f32x2 v = a[r][0];
#pragma unroll
                            for (int h = 1; h < CPW; ++h) v = jh == h ? a[r][h] : v;
                            f[r] = unpack2(__shfl_sync(kFull, v, jl));
                        }
#pragma unroll
                        for (int h = 0; h < CPW; ++h) {
                            const bool pc = lane == jl && jh == h;
                            used |= pc ? 1u << h : 0u;
                            mine |= pc ? 1u << h : 0u;
#pragma unroll
                            for (int r = 0; r < kBjB; ++r) a[r][h] = pc ? (r == i ? 0x3f800000ull : 0ull) : a[r][h];
                        }
                        const float2 pinv = bj_rcp(f[i]);
                        const f32x2 px = pack2(pinv.x, pinv.x), py = pack2(-pinv.y, pinv.y);
                        f32x2 fx[kBjB], fy[kBjB];
#pragma unroll
                        for (int r = 0; r < kBjB; ++r) {
                            fx[r] = pack2(-f[r].x, -f[r].x);
                            fy[r] = pack2(f[r].y, -f[r].y);
                        }
#pragma unroll
                        for (int h = 0; h < CPW; ++h) {
                            // the pivot row times 1 / pivot, then the others minus
                            // f times it: (x, y) and (y, x) of the row
                            float2 u = unpack2(a[i][h]);
                            const f32x2 sc = fma2(px, a[i][h], fma2(py, pack2(u.y, u.x), 0ull));
                            a[i][h] = sc;
                            u = unpack2(sc);
                            const f32x2 sw = pack2(u.y, u.x);
#pragma unroll
                            for (int r = 0; r < kBjB; ++r)
                                if (r != i) a[r][h] = fma2(fx[r], sc, fma2(fy[r], sw, a[r][h]));
                        }
                        if (lane == 0) {
                            s_J[i] = j;
                            slot_of[j] = i0 + i;
                            col_of[i0 + i] = j;
                        }
                    }
                }
            }
            // the rows of the transformation: P_J^{-1} in the pivot columns,
            // minus P_J^{-1} P elsewhere
#pragma unroll
            for (int r = 0; r < kBjB; ++r)
#pragma unroll
                for (int h = 0; h < CPW; ++h) {
                    const int c = lane + 32 * h;
                    const float2 u = unpack2(a[r][h]);
                    const float sg = (mine >> h) & 1u ? 1.f : -1.f;
                    if (c < CP) M[r * CP + c] = make_float4(sg * u.x, sg * u.y, -(sg * u.y), sg * u.x);
                }
            if (lane == 0 && !ok) s_sing = 1;
        }
        __syncthreads();
        if (s_sing) {  // uniform
            singular = true;
            break;
        }
        // the pivot columns, and their place in Z cleared (rows past N and
        // slots past nb: zeros)
        for (int r = tid; r < kBjRPT * TR; r += nthr) {
#pragma unroll
            for (int kk = 0; kk < kBjB; ++kk) {
                float2 v = make_float2(0.f, 0.f);
                if (r < N && kk < nb) {
                    float2 *e = Z + r * CP + s_J[kk];
                    v = *e;
                    *e = make_float2(0.f, 0.f);
                }
                zj[r * kBjZs + kk] = make_float4(v.x, v.x, v.y, v.y);
            }
        }
        __syncthreads();
        if (act) {
            switch (b.g8) {
            case 1: bj_update<1>(Z2, zj2, M2, N, TR, CP, tr, tc); break;
            case 2: bj_update<2>(Z2, zj2, M2, N, TR, CP, tr, tc); break;
            case 3: bj_update<3>(Z2, zj2, M2, N, TR, CP, tr, tc); break;
            case 4: bj_update<4>(Z2, zj2, M2, N, TR, CP, tr, tc); break;
            case 5: bj_update<5>(Z2, zj2, M2, N, TR, CP, tr, tc); break;
            default: bj_update<6>(Z2, zj2, M2, N, TR, CP, tr, tc); break;
            }
        }
        __syncthreads();
    }
    if (singular && tid == 0) atomicOr(&s.status[t], ST_SINGULAR);

    // ---- probabilities g_{a->m} = max(0, -2 dt v Re(R_ma) d_{m, s_a})
    auto occupied = [&](int m) { return (occ_bits[m >> 5] >> (m & 31)) & 1u; };
    // orbital data of m and of the column's slot (index N + c)
    auto prob = [&](const float4 &om, const float2 &om2, int c, float zr) -> float {
        // T_{m s_a} (times v for EXT) and lam_{s_a} - lam_m in FP32
        const float4 oc = od[N + c];
        float Tn = om.x * oc.x * fmaf(s_fac[2], om.y + oc.y, s_fac[1]);
        if constexpr (EXT) {
            const float2 oc2 = od2[N + c];
            Tn = fmaf(om2.x * oc2.x, fmaf(s_fac[4], om2.y + oc2.y, s_fac[3]), Tn);
        }
        const float gap = (oc.z - om.z) + (oc.w - om.w);
        const float g = s_fac[0] * zr * __fdividef(Tn, gap);  // at most 2 ulp
        return g > 0.f ? g : 0.f;
    };
    auto orb2 = [&](int m) { return EXT ? od2[m] : make_float2(0.f, 0.f); };
    if (!singular) {
        for (int c = tid; c < CP; c += nthr) {
            const int o = c < Ne ? occ_s[slot_of[c]] : 0;
            od[N + c] = od[o];
            if constexpr (EXT) od2[N + c] = od2[o];
        }
    }
    __syncthreads();
    if (g_out) {
        double *G = g_out + (int64_t)t * Ne * N;
        for (int a = warp; a < Ne; a += nwarp) {
            const int c = singular ? 0 : col_of[a];
            for (int m = lane; m < N; m += 32)
                G[(int64_t)a * N + m] = (singular || occupied(m)) ? 0.0 : (double)prob(od[m], orb2(m), c, Z[m * CP + c].x);
        }
        return;
    }
    if (!singular) {
        // per-slot sums over the unoccupied orbitals: thread (tr, tc) takes the
        // columns tc + 8 q of its rows
        // (the row's data stay in registers)
        float4 om[kBjRPT];
        float2 om2[kBjRPT];
        bool free_row[kBjRPT];
#pragma unroll
        for (int k = 0; k < kBjRPT; ++k) {
            const int m = tr + TR * k;
            free_row[k] = act && m < N && !occupied(m);
            om[k] = od[free_row[k] ? m : 0];
            om2[k] = orb2(free_row[k] ? m : 0);
        }
        for (int c = tc; c < CP; c += kBjTC) {
            long long acc = 0;
            if (c < Ne) {
#pragma unroll
                for (int k = 0; k < kBjRPT; ++k)
                    if (free_row[k]) acc += prob_fixed(prob(om[k], om2[k], c, Z[(tr + TR * k) * CP + c].x));
            }
            acc = sat1(acc);
#pragma unroll
            for (int o = kBjTC; o < 32; o <<= 1) acc = sat1(acc + __shfl_xor_sync(kFull, acc, o));
            if (lane < kBjTC) part[warp * CP + c] = acc;
        }
        __syncthreads();
        // the first slot (ascending), then the first orbital (ascending) whose
        // running sum exceeds zeta: warp 0, a run of slots (orbitals) per lane
        if (warp == 0) {
            const long long zeta = s_zeta;
            auto scan_excl = [&](long long v) {  // sum over the lanes below
                long long inc = v;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const long long w = __shfl_up_sync(kFull, inc, o);
                    if (lane >= o) inc = sat1(inc + w);
                }
                const long long ex = __shfl_up_sync(kFull, inc, 1);
                return lane == 0 ? 0 : ex;
            };
            constexpr int PA = 2;
            long long v[PA], loc = 0;
#pragma unroll
            for (int q = 0; q < PA; ++q) {
                const int a = lane * PA + q;
                v[q] = 0;
                if (a < Ne) {
                    const int c = col_of[a];
                    for (int w = 0; w < nwarp; ++w) v[q] = sat1(v[q] + part[w * CP + c]);
                }
                loc = sat1(loc + v[q]);
            }
            long long cum = scan_excl(loc), base = 0;
            int hit = -1;
#pragma unroll
            for (int q = 0; q < PA; ++q) {
                if (hit < 0 && cum + v[q] > zeta) {
                    hit = lane * PA + q;
                    base = cum;
                }
                cum = sat1(cum + v[q]);
            }
            const unsigned ba = __ballot_sync(kFull, hit >= 0);
            if (ba) {  // the slot; then its orbital
                const int src = __ffs(ba) - 1;
                const int ah = __shfl_sync(kFull, hit, src);
                base = __shfl_sync(kFull, base, src);
                const int ch = col_of[ah];
                const int pu = (N + 31) / 32, u0 = lane * pu, u1 = min(N, u0 + pu);
                auto g_of = [&](int m) { return occupied(m) ? 0ll : prob_fixed(prob(od[m], orb2(m), ch, Z[m * CP + ch].x)); };
                long long l2 = 0;
                for (int u = u0; u < u1; ++u) l2 = sat1(l2 + g_of(u));
                long long c2 = base + scan_excl(l2);
                int mh = -1;
                for (int u = u0; u < u1; ++u) {
                    c2 += g_of(u);
                    if (mh < 0 && c2 > zeta) mh = u;
                }
                const unsigned bm = __ballot_sync(kFull, mh >= 0);
                const int m_sel = bm ? __shfl_sync(kFull, mh, __ffs(bm) - 1) : -1;
                if (lane == 0 && m_sel >= 0) {
                    s_hop_a = ah;
                    s_hop_m = m_sel;
                }
            }
        }
        __syncthreads();
    }
    if constexpr (EXT) {  // rescale and bookkeeping in the six-coordinate acceptance kernel
        if (tid == 0) s.hop_pair[t] = s_hop_a >= 0 ? s_hop_a * N + s_hop_m : -1;
    } else {
        hop_apply<float2>(s, t, mass, red, occ_s, gv[0], gv[1], gv[2], s_hop_a, s_hop_m, Ct);
    }
}

}  // namespace

// Where it is the faster one (2048 trajectories, Ne = M / 2, ms per step, against
// the slot-by-slot kernel): N = 21 0.047 against 0.105, N = 51 0.10 against
// 0.22, N = 91 0.27 against 0.38; at N = 101 its passes over shared memory and
// its footprint bring it level, 0.42.
bool hop_bj_eligible(int N, int Ne) { return N <= kBjMaxN && Ne >= 1 && Ne <= kBjMaxNe && Ne < N; }

void configure_hop_bj()
{
    // the largest matrix (N = 96, Ne = 48) with its pivot columns: 58 KB, three CTAs
    // per SM (four up to N = 91, Ne = 45)
    const int most = (int)bj_shape(kBjMaxN, kBjMaxNe, true).total;
    cudaFuncSetAttribute(k_hop_bj<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
    cudaFuncSetAttribute(k_hop_bj<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
    cudaGetLastError();
}

cudaError_t launch_hop_bj(const DevState &s, double dt, double mass, uint64_t seed, double *g_out, cudaStream_t st,
                          bool ext)
{
    if (s.n == 0) return cudaSuccess;
    if (!hop_bj_eligible(s.N, s.Ne)) return cudaErrorInvalidValue;
    const BjShape b = bj_shape(s.N, s.Ne, ext);
    if (ext) k_hop_bj<true><<<(unsigned)s.n, b.threads, b.total, st>>>(s, dt, mass, seed, g_out);
    else k_hop_bj<false><<<(unsigned)s.n, b.threads, b.total, st>>>(s, dt, mass, seed, g_out);
    return cudaGetLastError();
}

}  // namespace iesh
