// Exact kNN affinity graph of Section 4.2 (k nearest neighbours q != p by
// Euclidean distance, ascending by (distance, index)), brute force.
//
// Pipeline
//  1. prep: centre the features (x - mu, mu the column mean: distances are
//     translation invariant) and round them to the candidate operand type
//     (float32 or bfloat16).  Per point keep ||xt_p||^2 and the rounding
//     perturbation rho_p >= ||xt_p - (x_p - mu)|| (float32 lane sums with
//     their rounding bounds, lanes added as 2Sum float pairs).
//  2. candidates: a distance-tile kernel evaluates
//     dt(p, q) = ||xt_p||^2 + ||xt_q||^2 - 2 xt_p . xt_q.  float32: for all pairs,
//     keeping per row and per column split the KC smallest (KC > k), sorted.
//     bfloat16 (knn_sweep.cu): keeping what a threshold from the k-th smallest
//     lets through, unsorted; above a work size over points sorted by region
//     (knn_group.cu) and only the tiles that can hold a neighbour.
//  3. rerank + certificate (one warp per row; knn_rerank_kernel, for the sweep's
//     slots knn_select_kernel): rank the candidates, recompute exactly in float32, from the original features, the distances
//     of the candidates whose lower bound can still reach the k nearest, keep
//     the k smallest.  With T the KC-th smallest dt, every other point q
//     satisfies dt(p,q) >= T, hence (rounding bounds below) its true distance
//     is at least LB = (sqrt(T - delta) - rho_p - rho_max)^2.  The row is
//     certified when the k-th exact distance, inflated by its own rounding
//     bound, is below LB; then the row equals a full float32 scan.
//  4. fallback: with bfloat16 candidates, the rows that fail the certificate
//     get two-term bfloat16 tiles from 100000 points on, then float32 candidate
//     tiles, each under its own certificate; rows that fail that (or the float32 certificate of a
//     float32 pass) are rescanned exactly.
#include <cuda_bf16.h>
#include <math.h>

#include <stdint.h>

#include <algorithm>

#include "knn_cert.cuh"
#include "knn_group.cuh"
#include "knn_sweep.cuh"
#include "pair32.cuh"
#include "slk_internal.cuh"

namespace {

constexpr int BM = 128, BN = 128, BK = 16, KT = 256;
constexpr int MAXE = 16;    // merge entries per lane (splits * KC <= 512)
#define kInf __int_as_float(0x7f800000)
constexpr int kNoIdx = 0x7fffffff;

__device__ __forceinline__ bool lex_less(float d, int i, float d2, int i2) {
    return d < d2 || (d == d2 && i < i2);
}

// Rows the exact rescan takes together, in registers (1: long rows).
__host__ __device__ __forceinline__ int exact_rows(int D) {
    const int dpl = (D + 31) / 32;
    return dpl <= 4 ? 16 : dpl <= 8 ? 8 : dpl <= 16 ? 4 : dpl <= 32 ? 2 : 1;
}
// Open rows at or below this count skip the float32 tiles (whose 128-row
// blocks they would leave mostly empty) and go to the exact scan.
constexpr long long kExactDirectRows = 256;

// Longest row the wide exact rescan stages in shared memory (bytes).
constexpr size_t kWideSmemMax = 200 * 1024;

// Column splits of the float32 stage for F open rows: as many as a buffer of
// cap floats holds at F rows per list of KC, at most 16 (the rerank stages
// 16 lists of 32 per row).  Host and device compute it from the same count.
__host__ __device__ __forceinline__ int query_splits(long long F, long long cap, int kc) {
    if (F <= 0) return 1;
    long long sp = cap / (F * (long long)kc);
    if (sp > 16) sp = 16;
    if (sp < 1) sp = 1;
    return (int)sp;
}

// Column splits of the exact scan for F rows, `together` at a time, on `ctas`
// CTAs: one item (rows, column range) per CTA, or 16 ranges where that leaves
// less than four, but no range below 64 columns and no more partial lists of k
// entries per (row, split) than cap entries hold.  A split costs an item's own
// merge and the final one k entries per row: with as many as the buffer held, at
// most 1024, the fallback took 1.18 ms for 22 rows of 9000 x 100, k = 24 (now 0.22),
// 3.55 for 219 rows of 9000 x 900, k = 6 (0.56), 11.0 for 762 after 9000 float32
// rows there (8.7).
__host__ __device__ __forceinline__ int exact_splits(long long F, int together, int ctas, int64_t N,
                                                     long long cap, int k) {
    if (F <= 0) return 1;
    const long long items = (F + together - 1) / together;
    long long sp = 4 * items <= ctas ? ctas / items : 16;
    if (sp > (N + 63) / 64) sp = (N + 63) / 64;
    if (sp > cap / (F * (long long)k)) sp = cap / (F * (long long)k);
    return sp < 1 ? 1 : (int)sp;
}

// -------------------------------------------------------------------- prep

// Column sums (the centring mean mu only has to be some float vector:
// distances are translation invariant): float32 sums of 64 rows, added in
// float64.  Each lane sums V adjacent columns (V = 4: 16-byte loads, when D
// is a multiple of 4 and X is 16-byte aligned); the rows and their order do
// not depend on V.
template <int V>
__global__ void col_sum_kernel(const float* __restrict__ X, int64_t N, int D,
                               double* __restrict__ colsum) {
    __shared__ double sm[8][32 * V + 1];
    const int DV = D / V;
    const int c = blockIdx.x * 32 + threadIdx.x;   // column group
    const int64_t per = (N + gridDim.y - 1) / gridDim.y;
    const int64_t r0 = (int64_t)blockIdx.y * per;
    const int64_t r1 = (r0 + per < N) ? r0 + per : N;
    double acc[V];
#pragma unroll
    for (int q = 0; q < V; ++q) acc[q] = 0.0;
    if (c < DV) {
        // rows r0 + y, r0 + y + 8, ... in increasing order; each chunk of 64
        // of them summed in float32 (8 loads in flight), the chunks in
        // float64 outside the inner loops (a float64 add predicated into
        // every iteration would occupy GB300's narrow float64 pipe)
        for (int64_t cb = r0 + threadIdx.y; cb < r1; cb += 512) {
            float part[V];
#pragma unroll
            for (int q = 0; q < V; ++q) part[q] = 0.f;
#pragma unroll 2
            for (int b = 0; b < 8; ++b) {
                float v[8][V];
#pragma unroll
                for (int t = 0; t < 8; ++t) {
                    const int64_t r = cb + 64 * b + 8 * t;
                    if constexpr (V == 4) {
                        const float4 w = (r < r1) ? __ldg(reinterpret_cast<const float4*>(X + r * D) + c)
                                                  : make_float4(0.f, 0.f, 0.f, 0.f);
                        v[t][0] = w.x; v[t][1] = w.y; v[t][2] = w.z; v[t][3] = w.w;
                    } else {
                        v[t][0] = (r < r1) ? X[r * D + c] : 0.f;
                    }
                }
#pragma unroll
                for (int t = 0; t < 8; ++t)
#pragma unroll
                    for (int q = 0; q < V; ++q) part[q] += v[t][q];
            }
#pragma unroll
            for (int q = 0; q < V; ++q) acc[q] += (double)part[q];
        }
    }
#pragma unroll
    for (int q = 0; q < V; ++q) sm[threadIdx.y][threadIdx.x * V + q] = acc[q];
    __syncthreads();
    if (threadIdx.y == 0 && c < DV) {
#pragma unroll
        for (int q = 0; q < V; ++q) {
            double t = 0.0;
            for (int i = 0; i < 8; ++i) t += sm[i][threadIdx.x * V + q];
            atomicAdd(&colsum[c * V + q], t);
        }
    }
}

// Column means of the centring: mu_j = (float)(colsum_j / N).
__global__ void mu_kernel(const double* __restrict__ colsum, int64_t N, int D, float* __restrict__ mu) {
    const double inv_n = 1.0 / (double)N;
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < D; j += gridDim.x * blockDim.x)
        mu[j] = (float)(colsum[j] * inv_n);
}

// rho >= sqrt(e2 bound) + u sqrt(v2 bound) and kappa >= rho / ||v|| with
// ||v|| >= sqrt(v2 / bound), from the float pairs (eh, el) = e2 and (vh, vl)
// = v2 (lane sums of e^2 and v^2); every step rounded toward the bound.
// kappa = 0 when v2 = 0 (then e = 0 and rho = 0), +inf when ||v|| underflows.
__device__ __forceinline__ void rho_kappa(float eh, float el, float vh, float vl, float bound_u,
                                          float& rho, float& kappa) {
    const float e2 = __fadd_ru(eh, el), v2 = __fadd_ru(vh, vl);
    const float t1 = __fsqrt_ru(__fmul_ru(e2, bound_u));
    const float t2 = __fmul_ru(5.9604644775390625e-08f, __fsqrt_ru(__fmul_ru(v2, bound_u)));
    rho = __fadd_ru(t1, t2);
    const float vlo = __fsqrt_rd(__fdiv_rd(__fadd_rd(vh, vl), bound_u));
    kappa = (v2 > 0.f) ? (vlo > 0.f ? __fdiv_ru(rho, vlo) : __int_as_float(0x7f800000)) : 0.f;
}

// Form of the candidate operand: bfloat16 or float32 rows, or float32 tiles of
// 128 rows by feature ([Np / 128][Dp][128]), as the float32 kernel stages them.
enum class Operand { bf16, f32_rows, f32_tiles };

// One warp per padded row: xt = round(v), v = fl(x - mu), with
//   norms[p] = ||xt_p||^2: lane sums of xt^2 in float32, lanes added as float
//     pairs (within a few u^2 of the exact sum);
//   rho[p] >= ||xt_p - (x_p - mu)||: with e = xt - v (exact in float32) and
//     |v - (x - mu)| <= u |v|, rho <= ||e|| + u ||v||, both norms from float32
//     lane sums inflated by their summation bound and rounded up.
// Every square of a lane sum passes through at most Dp/32 roundings (u =
// 2^-24): V = 1 sums the lane's Dp/32 columns in one accumulator; V = 4
// (16-byte loads, D a multiple of 4, X 16-byte aligned, Dp >= 128) keeps one
// accumulator per column of its 4-column groups, ceil(Dp/128) terms each,
// added pairwise at the end: ceil(Dp/128) + 2 <= Dp/32 roundings.  Each
// bfloat16 square is exact.
// The row maxima go to st with one atomic per block, with that of
// kappa_p = rho_p / ||v_p|| (||v_p|| from below), so that rho_q <= kappa ||v_q||
// for every row.
// aug (nullable, Np x 32 bfloat16): the folded-norm columns of the
// tensor-core tiles, [1, 1, 1, a_p, 0...] in columns 0..15 and [a_p, 1, 1, 1,
// 0...] in 16..31 (perm nullable: row p is point perm[p]; norms32 stays by
// point), a_p = (t1, t2, t3) the bfloat16 terms of -norms[p] / 2
// (t1 = bf16(x), t2 = bf16(x - t1), t3 = bf16(x - t1 - t2), each difference
// exact in float32, so t1 + t2 + t3 is within 2^-24 (1.02) |x| of x); a
// padding row has a_p = (-inf, 0, 0).
template <int V>
__global__ void __launch_bounds__(256)
prep_rows_kernel(const float* __restrict__ X, int64_t N, int D, int Dp,
                 int64_t Np, const float* __restrict__ mu, Operand to,
                 float* __restrict__ xt32, __nv_bfloat16* __restrict__ xt16,
                 float* __restrict__ norms, float* __restrict__ rho,
                 float* __restrict__ norms32, __nv_bfloat16* __restrict__ aug,
                 const int32_t* __restrict__ perm, DevState* st) {
    __shared__ unsigned bmax_n, bmax_r, bmax_n32, bmax_k;
    if (threadIdx.x == 0) { bmax_n = 0u; bmax_r = 0u; bmax_n32 = 0u; bmax_k = 0u; }
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int64_t nw = (int64_t)gridDim.x * (blockDim.x >> 5);
    // 1 + (Dp/32 + 2) u, rounded up: the lane sums' relative error bound
    const float bound_u = __double2float_ru(1.0 + (double)(Dp / 32 + 2) * 5.9604644775390625e-08);
    unsigned my_n = 0u, my_r = 0u, my_n32 = 0u, my_k = 0u;
    for (int64_t p = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); p < Np;
         p += nw) {
        const int64_t src = (perm && p < N) ? (int64_t)perm[p] : p;
        float n2v[V], e2v[V], v2v[V];
#pragma unroll
        for (int q = 0; q < V; ++q) { n2v[q] = 0.f; e2v[q] = 0.f; v2v[q] = 0.f; }
#pragma unroll 4
        for (int j = lane * V; j < Dp; j += 32 * V) {
            float v[V], vv[V];
#pragma unroll
            for (int q = 0; q < V; ++q) v[q] = 0.f;
            if (p < N && j < D) {
                if constexpr (V == 4) {
                    const float4 x = __ldg(reinterpret_cast<const float4*>(X + src * D + j));
                    const float4 m = __ldg(reinterpret_cast<const float4*>(mu + j));
                    v[0] = x.x - m.x; v[1] = x.y - m.y; v[2] = x.z - m.z; v[3] = x.w - m.w;
                } else {
                    v[0] = X[src * D + j] - __ldg(mu + j);
                }
            }
            if (to == Operand::bf16) {
                if constexpr (V == 4) {
                    const __nv_bfloat162 b01 = __floats2bfloat162_rn(v[0], v[1]);
                    const __nv_bfloat162 b23 = __floats2bfloat162_rn(v[2], v[3]);
                    uint2 w;
                    w.x = *reinterpret_cast<const unsigned*>(&b01);
                    w.y = *reinterpret_cast<const unsigned*>(&b23);
                    *reinterpret_cast<uint2*>(xt16 + p * Dp + j) = w;
                    vv[0] = __low2float(b01); vv[1] = __high2float(b01);
                    vv[2] = __low2float(b23); vv[3] = __high2float(b23);
                } else {
                    const __nv_bfloat16 b = __float2bfloat16_rn(v[0]);
                    xt16[p * Dp + j] = b;
                    vv[0] = __bfloat162float(b);
                }
            } else {
                if (to == Operand::f32_tiles)
#pragma unroll
                    for (int q = 0; q < V; ++q) xt32[((p / BM) * Dp + j + q) * BM + p % BM] = v[q];
                else if constexpr (V == 4)
                    *reinterpret_cast<float4*>(xt32 + p * Dp + j) = make_float4(v[0], v[1], v[2], v[3]);
                else
                    xt32[p * Dp + j] = v[0];
#pragma unroll
                for (int q = 0; q < V; ++q) vv[q] = v[q];
            }
#pragma unroll
            for (int q = 0; q < V; ++q) {
                n2v[q] = fmaf(vv[q], vv[q], n2v[q]);
                const float e = vv[q] - v[q];
                e2v[q] = fmaf(e, e, e2v[q]);
                v2v[q] = fmaf(v[q], v[q], v2v[q]);
            }
        }
        float n2 = n2v[0], e2 = e2v[0], v2 = v2v[0];
        if constexpr (V == 4) {
            n2 = (n2v[0] + n2v[1]) + (n2v[2] + n2v[3]);
            e2 = (e2v[0] + e2v[1]) + (e2v[2] + e2v[3]);
            v2 = (v2v[0] + v2v[1]) + (v2v[2] + v2v[3]);
        }
        // butterfly sums of the lane sums as unevaluated float pairs (2Sum):
        // within a few u^2 of the exact sum, and off the slow float64 pipe
        float nh = n2, nl = 0.f, eh = e2, el = 0.f, vh = v2, vl = 0.f;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            fpair_add(nh, nl, __shfl_xor_sync(0xffffffffu, nh, o), __shfl_xor_sync(0xffffffffu, nl, o));
            fpair_add(eh, el, __shfl_xor_sync(0xffffffffu, eh, o), __shfl_xor_sync(0xffffffffu, el, o));
            fpair_add(vh, vl, __shfl_xor_sync(0xffffffffu, vh, o), __shfl_xor_sync(0xffffffffu, vl, o));
        }
        if (lane == 0) {
            // the pair sums rounded to nearest (norms), up and down (bounds);
            // float32 with directed rounding keeps the bounds off the slow
            // float64 pipe
            const float nf = __fadd_rn(nh, nl);
            float rf, kf;
            rho_kappa(eh, el, vh, vl, bound_u, rf, kf);
            // padding rows get an infinite norm: no distance to them can pass a filter
            norms[p] = (p < N) ? nf : __int_as_float(0x7f800000);
            rho[p] = rf;
            const float n32 = __fadd_rn(vh, vl);   // ||v||^2 of the float32 operand v
            if (norms32) norms32[src] = (p < N) ? n32 : __int_as_float(0x7f800000);
            if (p < N) {
                my_n = max(my_n, __float_as_uint(nf));
                my_r = max(my_r, __float_as_uint(rf));
                my_n32 = max(my_n32, __float_as_uint(n32));
                my_k = max(my_k, __float_as_uint(kf));
            }
        }
        if (aug) {
            // lanes 0..3 write 8 columns each (16-byte stores)
            const float nfa = __shfl_sync(0xffffffffu, __fadd_rn(nh, nl), 0);
            if (lane < 4) {
                const float x = -0.5f * nfa;
                const __nv_bfloat16 t1 = __float2bfloat16_rn(x);
                const float r1 = x - __bfloat162float(t1);
                const __nv_bfloat16 t2 = __float2bfloat16_rn(r1);
                const __nv_bfloat16 t3 = __float2bfloat16_rn(r1 - __bfloat162float(t2));
                const __nv_bfloat16 one = __float2bfloat16_rn(1.f), zero = __float2bfloat16_rn(0.f);
                const __nv_bfloat16 a1 = (p < N) ? t1 : __float2bfloat16_rn(-__int_as_float(0x7f800000));
                const __nv_bfloat16 a2 = (p < N) ? t2 : zero, a3 = (p < N) ? t3 : zero;
                __nv_bfloat16 w[8];
#pragma unroll
                for (int q = 0; q < 8; ++q) w[q] = zero;
                if (lane == 0) {          // columns 0..7: 1, 1, 1, a1, a2, a3
                    w[0] = one; w[1] = one; w[2] = one; w[3] = a1; w[4] = a2; w[5] = a3;
                } else if (lane == 2) {   // columns 16..23: a1, a2, a3, 1, 1, 1
                    w[0] = a1; w[1] = a2; w[2] = a3; w[3] = one; w[4] = one; w[5] = one;
                }
                *reinterpret_cast<uint4*>(aug + p * 32 + 8 * lane) = *reinterpret_cast<const uint4*>(w);
            }
        }
    }
    if (lane == 0) {
        atomicMax(&bmax_n, my_n);
        atomicMax(&bmax_r, my_r);
        atomicMax(&bmax_n32, my_n32);
        atomicMax(&bmax_k, my_k);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        atomicMax(&st->knn_max_norm_bits, bmax_n);
        atomicMax(&st->knn_max_rho_bits, bmax_r);
        atomicMax(&st->knn_max_norm32_bits, bmax_n32);
        atomicMax(&st->knn_max_kappa_bits, bmax_k);
    }
}

// ------------------------------------------------- two-term bfloat16 operand

// One warp per padded row p < Np, for the rows the bfloat16 certificate
// leaves open (nothing runs when *open_count is 0): with v = fl(x - mu) and
// h = bf16(v) (the candidate operand xt), the second term l = bf16(v - h)
// (v - h is exact), so that s = h + l carries 16 significant bits of v:
//   xh[p]      = h (nullable: only where the operand xt is in another order),
//   xl[p]      = l,
//   norms_s[p] = ||s||^2 (s = h + l is exact in float32: l either equals
//                v - h, then s = v, or has its last bit above v's),
//   rho_s[p]  >= ||s - (x_p - mu)||, from e = s - v (exact) and
//                |v - (x - mu)| <= u |v|, as for the other operands.
// Sums as in prep_rows_kernel (the same lane split and float-pair butterfly,
// so the same summation bound); row maxima to st.
template <int V>
__global__ void __launch_bounds__(256)
prep_split_kernel(const float* __restrict__ X, int64_t N, int D, int Dp, int64_t Np,
                  const float* __restrict__ mu, const long long* __restrict__ open_count,
                  __nv_bfloat16* __restrict__ xh, __nv_bfloat16* __restrict__ xl,
                  float* __restrict__ norms_s, float* __restrict__ rho_s, DevState* st) {
    if (*open_count == 0) return;
    __shared__ unsigned bmax_n, bmax_r, bmax_k;
    if (threadIdx.x == 0) { bmax_n = 0u; bmax_r = 0u; bmax_k = 0u; }
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int64_t nw = (int64_t)gridDim.x * (blockDim.x >> 5);
    // 1 + (Dp/32 + 2) u, rounded up: the lane sums' relative error bound
    const float bound_u = __double2float_ru(1.0 + (double)(Dp / 32 + 2) * 5.9604644775390625e-08);
    unsigned my_n = 0u, my_r = 0u, my_k = 0u;
    for (int64_t p = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); p < Np;
         p += nw) {
        float n2v[V], e2v[V], v2v[V];
#pragma unroll
        for (int q = 0; q < V; ++q) { n2v[q] = 0.f; e2v[q] = 0.f; v2v[q] = 0.f; }
#pragma unroll 4
        for (int j = lane * V; j < Dp; j += 32 * V) {
            float v[V];
#pragma unroll
            for (int q = 0; q < V; ++q) v[q] = 0.f;
            if (p < N && j < D) {
                if constexpr (V == 4) {
                    const float4 x = __ldg(reinterpret_cast<const float4*>(X + p * D + j));
                    const float4 m = __ldg(reinterpret_cast<const float4*>(mu + j));
                    v[0] = x.x - m.x; v[1] = x.y - m.y; v[2] = x.z - m.z; v[3] = x.w - m.w;
                } else {
                    v[0] = X[p * D + j] - __ldg(mu + j);
                }
            }
            __nv_bfloat16 hb[V], lb[V];
            float sv[V];
#pragma unroll
            for (int q = 0; q < V; ++q) {
                hb[q] = __float2bfloat16_rn(v[q]);
                const float h = __bfloat162float(hb[q]);
                lb[q] = __float2bfloat16_rn(v[q] - h);
                sv[q] = h + __bfloat162float(lb[q]);
            }
            if constexpr (V == 4) {
                __nv_bfloat162 b01, b23;
                b01.x = lb[0]; b01.y = lb[1]; b23.x = lb[2]; b23.y = lb[3];
                uint2 w;
                w.x = *reinterpret_cast<const unsigned*>(&b01);
                w.y = *reinterpret_cast<const unsigned*>(&b23);
                *reinterpret_cast<uint2*>(xl + p * Dp + j) = w;
                if (xh) {
                    b01.x = hb[0]; b01.y = hb[1]; b23.x = hb[2]; b23.y = hb[3];
                    w.x = *reinterpret_cast<const unsigned*>(&b01);
                    w.y = *reinterpret_cast<const unsigned*>(&b23);
                    *reinterpret_cast<uint2*>(xh + p * Dp + j) = w;
                }
            } else {
                xl[p * Dp + j] = lb[0];
                if (xh) xh[p * Dp + j] = hb[0];
            }
#pragma unroll
            for (int q = 0; q < V; ++q) {
                n2v[q] = fmaf(sv[q], sv[q], n2v[q]);
                const float e = sv[q] - v[q];
                e2v[q] = fmaf(e, e, e2v[q]);
                v2v[q] = fmaf(v[q], v[q], v2v[q]);
            }
        }
        float n2 = n2v[0], e2 = e2v[0], v2 = v2v[0];
        if constexpr (V == 4) {
            n2 = (n2v[0] + n2v[1]) + (n2v[2] + n2v[3]);
            e2 = (e2v[0] + e2v[1]) + (e2v[2] + e2v[3]);
            v2 = (v2v[0] + v2v[1]) + (v2v[2] + v2v[3]);
        }
        float nh = n2, nl = 0.f, eh = e2, el = 0.f, vh = v2, vl = 0.f;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            fpair_add(nh, nl, __shfl_xor_sync(0xffffffffu, nh, o), __shfl_xor_sync(0xffffffffu, nl, o));
            fpair_add(eh, el, __shfl_xor_sync(0xffffffffu, eh, o), __shfl_xor_sync(0xffffffffu, el, o));
            fpair_add(vh, vl, __shfl_xor_sync(0xffffffffu, vh, o), __shfl_xor_sync(0xffffffffu, vl, o));
        }
        if (lane == 0) {
            const float nf = __fadd_rn(nh, nl);
            float rf, kf;
            rho_kappa(eh, el, vh, vl, bound_u, rf, kf);
            norms_s[p] = (p < N) ? nf : __int_as_float(0x7f800000);
            rho_s[p] = rf;
            if (p < N) {
                my_n = max(my_n, __float_as_uint(nf));
                my_r = max(my_r, __float_as_uint(rf));
                my_k = max(my_k, __float_as_uint(kf));
            }
        }
    }
    if (lane == 0) {
        atomicMax(&bmax_n, my_n);
        atomicMax(&bmax_r, my_r);
        atomicMax(&bmax_k, my_k);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        atomicMax(&st->knn_max_norm_s_bits, bmax_n);
        atomicMax(&st->knn_max_rho_s_bits, bmax_r);
        atomicMax(&st->knn_max_kappa_s_bits, bmax_k);
    }
}

// Query rows of the two-term stage: row f < min(*count, Fcap) of qh / ql /
// qnorm is row fb[f] of xh / xl / norms_s; the rest of its 128-row block is
// zero with an infinite norm.  One warp per row, 16-byte copies (Dp is a
// multiple of 64).
__global__ void __launch_bounds__(256)
gather_split_kernel(const __nv_bfloat16* __restrict__ xh, const __nv_bfloat16* __restrict__ xl,
                    const float* __restrict__ norms_s, int Dp, const int32_t* __restrict__ fb,
                    const long long* __restrict__ count, int64_t Fcap,
                    __nv_bfloat16* __restrict__ qh, __nv_bfloat16* __restrict__ ql,
                    float* __restrict__ qnorm) {
    long long c = *count;
    if (c > Fcap) c = Fcap;
    const int64_t rows = (c + 127) / 128 * 128;
    const int lane = threadIdx.x & 31;
    const int64_t nw = (int64_t)gridDim.x * (blockDim.x >> 5);
    const int n16 = Dp / 8;   // 16-byte words per row
    for (int64_t f = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); f < rows;
         f += nw) {
        const bool live = f < c;
        const int64_t p = live ? (int64_t)fb[f] : 0;
        const uint4* sh = reinterpret_cast<const uint4*>(xh + p * Dp);
        const uint4* sl = reinterpret_cast<const uint4*>(xl + p * Dp);
        uint4* dh = reinterpret_cast<uint4*>(qh + f * Dp);
        uint4* dl = reinterpret_cast<uint4*>(ql + f * Dp);
        const uint4 z = make_uint4(0u, 0u, 0u, 0u);
        for (int j = lane; j < n16; j += 32) {
            dh[j] = live ? __ldg(sh + j) : z;
            dl[j] = live ? __ldg(sl + j) : z;
        }
        if (lane == 0) qnorm[f] = live ? norms_s[p] : __int_as_float(0x7f800000);
    }
}

// ------------------------------------------------------- fp32 candidate tiles

constexpr int kFStages = 4;   // operand chunks staged (as large as the tile of distances)

// Shared-memory layout of the candidate kernels (dynamic).  The tile of
// distances takes the operands' place once the products are done; lists are
// keys (tile_key) in increasing order.
template <int KC>
struct CandSmem {
    union {
        struct {
            float As[kFStages][BK][BM];
            float Bs[kFStages][BK][BN];
        } op;
        float dt[BM][BN];
    };
    unsigned long long list[BM][KC];
    float nrow[BM];
    float ncol[BN];
};

// (distance, index) as one integer of the same order.
__device__ __forceinline__ unsigned long long tile_key(float d, int i) {
    const uint32_t u = __float_as_uint(d + 0.f);   // -0 as 0: equal distances go by index
    return (unsigned long long)(u ^ ((uint32_t)((int)u >> 31) | 0x80000000u)) << 32 | (uint32_t)i;
}
__device__ __forceinline__ float key_dist(unsigned long long key) {
    const uint32_t u = (uint32_t)(key >> 32);
    return __uint_as_float(u >> 31 ? u ^ 0x80000000u : ~u);
}
__device__ __forceinline__ unsigned long long empty_key() { return tile_key(kInf, kNoIdx); }

// One step of the tiles' products: features kk of 8 x 8 rows and columns of a
// thread, two columns per instruction.
template <int KC>
__device__ __forceinline__ void tile_products(const CandSmem<KC>& s, int buf, int ty, int tx,
                                              pair32 (&acc)[8][4]) {
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
        const float4 a0 = *reinterpret_cast<const float4*>(&s.op.As[buf][kk][4 * ty]);
        const float4 a1 = *reinterpret_cast<const float4*>(&s.op.As[buf][kk][64 + 4 * ty]);
        const ulonglong2 b0 = *reinterpret_cast<const ulonglong2*>(&s.op.Bs[buf][kk][4 * tx]);
        const ulonglong2 b1 = *reinterpret_cast<const ulonglong2*>(&s.op.Bs[buf][kk][64 + 4 * tx]);
        const float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
        const pair32 b[4] = {b0.x, b0.y, b1.x, b1.y};
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const pair32 aa = pack2(a[i], a[i]);
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[i][j] = fma2(aa, b[j], acc[i][j]);
        }
    }
}

__device__ __forceinline__ void tile_copy16(float* dst, const float* src) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void tile_copies_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void tile_copies_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(kFStages - 2) : "memory");
}

// Sorts one key per lane (up: increasing with the lane).
template <int V>
__device__ __forceinline__ void warp_sort(unsigned long long (&x)[V], const bool (&up)[V], int lane,
                                          int from) {
#pragma unroll
    for (int n = 2; n <= 32; n <<= 1) {
        if (n < from) continue;
#pragma unroll
        for (int o = n >> 1; o > 0; o >>= 1)
#pragma unroll
            for (int v = 0; v < V; ++v) {
                const unsigned long long y = __shfl_xor_sync(0xffffffffu, x[v], o);
                const bool asc = n == 32 ? up[v] : (lane & n) == 0;
                const bool keep_min = ((lane & o) == 0) == asc;
                x[v] = (y < x[v]) == keep_min ? y : x[v];
            }
    }
}

// Distances of the tile (products acc; n_p + n_q - 2 dot) into shared memory,
// NaN (never a candidate) where ok refuses the pair, and each row's list
// brought up to date: a warp takes 16 rows, four columns per lane.  A row with
// many hits (the first tiles) sorts the tile's 128 keys and merges; one with
// few inserts them one by one, the bound falling with each.  Queues filled by
// atomics and merged by one thread per row made the whole block wait for the
// longest: candidates of 2000 x 16 points 200 us, now 51 us; of 30011 x 200,
// k = 12, 11.8 ms, now 8.5 (7.6 with the operand in tiles, below).
constexpr int kSortHits = 20;
template <int KC, class Ok>
__device__ __forceinline__ void tile_select(CandSmem<KC>& s, const pair32 (&acc)[8][4], int64_t col0,
                                            int ty, int tx, Ok ok) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int r = (i < 4) ? 4 * ty + i : 64 + 4 * ty + (i - 4);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float d[4];
            unpack2(acc[i][2 * h], d[0], d[1]);
            unpack2(acc[i][2 * h + 1], d[2], d[3]);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int c = 64 * h + 4 * tx + j;
                d[j] = ok(r, c) ? fmaf(-2.f, d[j], s.nrow[r] + s.ncol[c]) : __int_as_float(0x7fffffff);
            }
            *reinterpret_cast<float4*>(&s.dt[r][64 * h + 4 * tx]) = make_float4(d[0], d[1], d[2], d[3]);
        }
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int RW = BM / (KT / 32);
    for (int r = warp * RW; r < (warp + 1) * RW; ++r) {
        const float4 x = *reinterpret_cast<const float4*>(&s.dt[r][4 * lane]);
        const float v[4] = {x.x, x.y, x.z, x.w};
        float thr = key_dist(s.list[r][KC - 1]);
        int hits = 0;
        unsigned m[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            m[j] = __ballot_sync(0xffffffffu, v[j] <= thr);
            hits += __popc(m[j]);
        }
        if (hits == 0) continue;
        unsigned long long l = lane < KC ? s.list[r][lane] : empty_key();
        if (hits > kSortHits) {
            unsigned long long k[4];
#pragma unroll
            for (int j = 0; j < 4; ++j)
                k[j] = v[j] <= thr ? tile_key(v[j], (int)col0 + 4 * lane + j) : empty_key();
            warp_sort<4>(k, {true, false, true, false}, lane, 2);
            unsigned long long h[2] = {min(k[0], k[1]), min(k[2], k[3])};
            warp_sort<2>(h, {true, false}, lane, 32);
            unsigned long long q[1] = {min(h[0], h[1])};
            warp_sort<1>(q, {false}, lane, 32);
            q[0] = min(l, q[0]);
            warp_sort<1>(q, {true}, lane, 32);
            l = q[0];
        } else {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                unsigned left = m[j];
                while (left) {
                    const int src = __ffs(left) - 1;
                    const float d = __shfl_sync(0xffffffffu, v[j], src);
                    left &= left - 1;
                    if (d > thr) continue;
                    const unsigned long long key = tile_key(d, (int)col0 + 4 * src + j);
                    const unsigned long long up = __shfl_up_sync(0xffffffffu, l, 1);
                    // entries above the new key move one lane on
                    if (l > key) l = lane > 0 && up > key ? up : key;
                    thr = key_dist(__shfl_sync(0xffffffffu, l, KC - 1));
                }
            }
        }
        if (lane < KC) s.list[r][lane] = l;
    }
}

// Bound by the float32 units (2 N^2 Dp operations: 49 of 80 TFLOP/s at 30011 x
// 200).  The operand comes in tiles of 128 points by feature, so that a chunk of
// either side is one contiguous run: four chunks under way by asynchronous copies
// and no registers held for them (row by row through registers, transposed on the
// way: 8.5 ms, now 7.6; the rows' values doubled in shared memory to save the
// packing: 9.9).
// Grid: (row blocks of 128, column splits).  Thread (ty, tx) = (t / 16, t % 16)
// owns rows {4ty..4ty+3, 64+4ty..64+4ty+3} and the same pattern of columns.
template <int KC>
__global__ void __launch_bounds__(KT, 2)
knn_cand_fp32_kernel(const float* __restrict__ xt, const float* __restrict__ norms, int64_t N,
                     int Dp, int n_tiles, int64_t Np, float* __restrict__ cand_d,
                     int32_t* __restrict__ cand_i) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    CandSmem<KC>& s = *reinterpret_cast<CandSmem<KC>*>(smem_raw);
    const int t = threadIdx.x, ty = t >> 4, tx = t & 15;
    const int64_t row0 = (int64_t)blockIdx.x * BM;
    const int sp = blockIdx.y, splits = gridDim.y;
    const int tile0 = (int)((int64_t)sp * n_tiles / splits);
    const int tile1 = (int)((int64_t)(sp + 1) * n_tiles / splits);
    if (t < BM) {
        for (int j = 0; j < KC; ++j) s.list[t][j] = empty_key();
        s.nrow[t] = norms[row0 + t];
    }
    const int nk = Dp / BK;
    // chunk kt of a tile: BK x 128 floats, contiguous in the tiled operand
    const float* pa = xt + row0 * Dp + 4 * t;
    for (int tile = tile0; tile < tile1; ++tile) {
        const int64_t col0 = (int64_t)tile * BN;
        __syncthreads();  // previous epilogue finished with ncol / buffers
        if (t < BN) s.ncol[t] = norms[col0 + t];
        pair32 acc[8][4];
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[i][j] = 0ull;
        const float* pb = xt + col0 * Dp + 4 * t;
        auto fetch = [&](int kt) {
            if (kt < nk) {
                float* a = &s.op.As[kt % kFStages][0][0] + 4 * t;
                float* b = &s.op.Bs[kt % kFStages][0][0] + 4 * t;
#pragma unroll
                for (int h = 0; h < BK * BM / (4 * KT); ++h) {
                    tile_copy16(a + 4 * KT * h, pa + kt * (BK * BM) + 4 * KT * h);
                    tile_copy16(b + 4 * KT * h, pb + kt * (BK * BN) + 4 * KT * h);
                }
            }
            tile_copies_commit();   // (an empty group keeps the wait count uniform)
        };
#pragma unroll
        for (int kt = 0; kt < kFStages - 1; ++kt) fetch(kt);
        for (int kt = 0; kt < nk; ++kt) {
            tile_copies_wait();     // this thread's copies of chunk kt have landed
            __syncthreads();        // ... every thread's, and chunk kt - 1 is read
            fetch(kt + kFStages - 1);
            tile_products<KC>(s, kt % kFStages, ty, tx, acc);
        }
        __syncthreads();            // the operands are read: the tile may take their place
        tile_select<KC>(s, acc, col0, ty, tx, [&](int r, int c) {
            const int64_t p = row0 + r, q = col0 + c;
            return p < N && q < N && q != p;
        });
    }
    __syncthreads();
    if (t < BM) {
        const int64_t o = ((int64_t)sp * Np + row0 + t) * KC;
        for (int j = 0; j < KC; ++j) {
            cand_d[o + j] = key_dist(s.list[t][j]);
            cand_i[o + j] = (int)(uint32_t)s.list[t][j] == kNoIdx ? -1 : (int)(uint32_t)s.list[t][j];
        }
    }
}

// Float32 distance tiles for listed query rows (the rows the earlier
// certificates left open): rows fb_list[f], f < F = *count, against every
// point.  Both operands are centred on the fly, v = fl(x - mu) -- the float32
// operand the float32 path would hold -- and the norms are its norms.  Work
// items (query row block, column split) are taken persistently, so the grid
// does not depend on the count; the split count is query_splits(F, cap, KC)
// and lists go to ((split F + f) KC).  Nothing runs for F <=
// kExactDirectRows (those rows go to the exact scan).
template <int KC>
__global__ void __launch_bounds__(KT, 2)
knn_cand_query_kernel(const float* __restrict__ X, int64_t N, int D, int Dp,
                      const float* __restrict__ mu, const float* __restrict__ norms32,
                      const int32_t* __restrict__ fb_list, const long long* count_ptr,
                      long long cap, int n_tiles, float* __restrict__ cand_d,
                      int32_t* __restrict__ cand_i) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    CandSmem<KC>& s = *reinterpret_cast<CandSmem<KC>*>(smem_raw);
    __shared__ int64_t prow[BM];
    const int t = threadIdx.x, ty = t >> 4, tx = t & 15;
    const long long F = *(const volatile long long*)count_ptr;
    if (F <= kExactDirectRows) return;
    const int splits = query_splits(F, cap, KC);
    const int64_t items = (F + BM - 1) / BM * splits;
    const int nk = Dp / BK;
    const int lr0 = t & 127, lq0 = t >> 7, lq1 = lq0 + 2;
    for (int64_t item = blockIdx.x; item < items; item += gridDim.x) {
        const int64_t rb = item / splits;
        const int sp = (int)(item % splits);
        const int tile0 = (int)((int64_t)sp * n_tiles / splits);
        const int tile1 = (int)((int64_t)(sp + 1) * n_tiles / splits);
        __syncthreads();   // the previous item is done with the lists
        if (t < BM) {
            const int64_t f = rb * BM + t;
            const int64_t p = (f < F) ? (int64_t)fb_list[f] : -1;
            prow[t] = p;
            for (int j = 0; j < KC; ++j) s.list[t][j] = empty_key();
            s.nrow[t] = (p >= 0) ? norms32[p] : kInf;
        }
        __syncthreads();
        const int64_t pa_row = prow[lr0];
        for (int tile = tile0; tile < tile1; ++tile) {
            const int64_t col0 = (int64_t)tile * BN;
            __syncthreads();  // previous epilogue finished with ncol / buffers
            if (t < BN) s.ncol[t] = (col0 + t < N) ? norms32[col0 + t] : kInf;
            const int64_t qb_row = (col0 + lr0 < N) ? col0 + lr0 : -1;
            pair32 acc[8][4];
#pragma unroll
            for (int i = 0; i < 8; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = 0ull;
            float ra[8], rbv[8];
            // 16-byte loads when every row starts on a 16-byte boundary and the
            // four features of a chunk are all inside the row (D % 4 == 0)
            const bool v4 = (D & 3) == 0 && ((reinterpret_cast<uintptr_t>(X) & 15) == 0);
            auto fetch = [&](int k0) {
                if (v4) {
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int d = k0 + 4 * (h == 0 ? lq0 : lq1);
                        const bool in = d < D;
                        const float4 m4 = in ? __ldg(reinterpret_cast<const float4*>(mu + d))
                                             : make_float4(0.f, 0.f, 0.f, 0.f);
                        const float4 xa = (pa_row >= 0 && in)
                                              ? __ldg(reinterpret_cast<const float4*>(X + pa_row * D + d))
                                              : m4;
                        const float4 xb = (qb_row >= 0 && in)
                                              ? __ldg(reinterpret_cast<const float4*>(X + qb_row * D + d))
                                              : m4;
                        ra[4 * h + 0] = xa.x - m4.x; ra[4 * h + 1] = xa.y - m4.y;
                        ra[4 * h + 2] = xa.z - m4.z; ra[4 * h + 3] = xa.w - m4.w;
                        rbv[4 * h + 0] = xb.x - m4.x; rbv[4 * h + 1] = xb.y - m4.y;
                        rbv[4 * h + 2] = xb.z - m4.z; rbv[4 * h + 3] = xb.w - m4.w;
                    }
                    return;
                }
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    const int d = k0 + 4 * (c < 4 ? lq0 : lq1) + (c & 3);
                    const float m = (d < D) ? mu[d] : 0.f;
                    ra[c] = (pa_row >= 0 && d < D) ? X[pa_row * D + d] - m : 0.f;
                    rbv[c] = (qb_row >= 0 && d < D) ? X[qb_row * D + d] - m : 0.f;
                }
            };
            auto stash = [&](int buf) {
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    const int kk = 4 * (c < 4 ? lq0 : lq1) + (c & 3);
                    s.op.As[buf][kk][lr0] = ra[c];
                    s.op.Bs[buf][kk][lr0] = rbv[c];
                }
            };
            fetch(0);
            stash(0);
            __syncthreads();
            for (int kt = 0; kt < nk; ++kt) {
                const int buf = kt & 1;
                if (kt + 1 < nk) fetch((kt + 1) * BK);
                tile_products<KC>(s, buf, ty, tx, acc);
                if (kt + 1 < nk) stash(buf ^ 1);
                __syncthreads();
            }
            tile_select<KC>(s, acc, col0, ty, tx, [&](int r, int c) {
                const int64_t p = prow[r], q = col0 + c;
                return p >= 0 && q < N && q != p;
            });
        }
        __syncthreads();
        if (t < BM) {
            const int64_t f = rb * BM + t;
            if (f < F) {
                const int64_t o = ((int64_t)sp * F + f) * KC;
                for (int j = 0; j < KC; ++j) {
                    cand_d[o + j] = key_dist(s.list[t][j]);
                    cand_i[o + j] = (int)(uint32_t)s.list[t][j] == kNoIdx ? -1 : (int)(uint32_t)s.list[t][j];
                }
            }
        }
    }
}

// ------------------------------------------------------ rerank + certificate

// Exact float32 squared distance, lane-strided over features, xor-butterfly
// sum: every lane gets the same bits, and the fallback scan uses the same
// formula so both paths agree bit for bit.
__device__ __forceinline__ float exact_d2(const float* __restrict__ xp,
                                          const float* __restrict__ xq, int D, int lane) {
    float part = 0.f;
    for (int j = lane; j < D; j += 32) {
        const float df = xp[j] - xq[j];
        part = fmaf(df, df, part);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
    return part;
}

// Feature-loop unrolling of the rerank's exact distances (gathers in flight;
// measured at 1e6 x 128: 4 gives 10.0 ms against 9.0 for 1)
#ifndef SLK_RERANK_UNROLL
#define SLK_RERANK_UNROLL 1
#endif
constexpr int kRerankUnroll = SLK_RERANK_UNROLL;

// Rerank + certificate of the float32 tiles, one warp per row.  Lists hold KC
// entries each; the KC best of their union are the candidates whose last one
// bounds the rest.  gam bounds the error of a tile's dot product relative to
// |xt_p| |xt_q| (with the norms' roundings added here).
//   MODE 0: every row p < N, the lists of the candidate kernels at
//           ((list Np + p) KC), failures appended to fb_list.
//   MODE 1: the rows fb_in[f], f < F = *count_in, their float32 query lists
//           at ((split F + f) KC), query_splits(F, Np, KC) of them (Np: the
//           list buffer's capacity in floats), norms of the float32 operand
//           (rho <= u ||v||), failures appended to fb_list / *count_out; for
//           F <= kExactDirectRows every row is appended (no lists were made).
template <int KC, int MODE, int E = MAXE>
__global__ void __launch_bounds__(256, 4)
knn_rerank_kernel(const float* __restrict__ X, int64_t N, int D, int Dp, int k, int splits_in,
                  int64_t Np, const float* __restrict__ cand_d, const int32_t* __restrict__ cand_i,
                  const float* __restrict__ norms, const float* __restrict__ rho, double gam,
                  int64_t* __restrict__ row_ptr, int32_t* __restrict__ col_idx,
                  float* __restrict__ dist2, int32_t* __restrict__ fb_list, DevState* st,
                  const int32_t* __restrict__ fb_in = nullptr, const long long* count_in = nullptr,
                  long long* count_out = nullptr) {
    constexpr bool Q = MODE != 0;
    constexpr int SEL = KC;
    __shared__ float s_d[8][32 * E];   // each warp's staged lists (256 threads)
    __shared__ int s_i[8][32 * E];
    __shared__ float s_od[8][SEL];     // and its SEL selected candidates
    __shared__ int s_oi[8][SEL];
    const int lane = threadIdx.x & 31;
    const int64_t nw = (int64_t)gridDim.x * (blockDim.x >> 5);
    const double u = 5.9604644775390625e-08;  // 2^-24
    const double nmax = (double)__uint_as_float(MODE == 0 ? st->knn_max_norm_bits : st->knn_max_norm32_bits);
    const double rmax = MODE == 1 ? u * sqrt(nmax) * (1.0 + 1e-6)
                                  : (double)__uint_as_float(st->knn_max_rho_bits);
    // rho_q <= kappa ||v_q|| for every row q
    const double kappa = MODE == 1 ? u * (1.0 + 1e-5)
                                   : (double)__uint_as_float(st->knn_max_kappa_bits);
    const double err_exact = 1.01 * (double)(D + 8) * u;
    // float32 copies of the bound's constants for the candidate pruning
    // (margins of 1e-6 .. 1e-5 cover the float rounding of the bounds)
    const float coef_f = (float)((gam + (double)(Dp / 32 + 5) * u) * (1.0 + 1e-6));
    const float rmax_f = (float)(rmax * (1.0 + 1e-6));
    const float snmax_f = (float)(sqrt(nmax) * (1.0 + 1e-6));
    const float keep_f = (float)((1.0 + 2.02 * err_exact) / (1.0 - 2.02 * err_exact) * (1.0 + 1e-5));
    const int64_t rows = Q ? (int64_t)(*(const volatile long long*)count_in) : N;
    const int splits = MODE == 1 ? query_splits(rows, Np, KC) : splits_in;
    const int64_t stride = MODE == 1 ? rows : Np;
    if (MODE == 1 && rows <= kExactDirectRows) {
        // too few rows for the float32 tiles: all of them to the exact scan
        for (int64_t f = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; f < rows;
             f += (int64_t)gridDim.x * blockDim.x) {
            const unsigned long long slot = atomicAdd((unsigned long long*)count_out, 1ull);
            fb_list[slot] = fb_in[f];
        }
        return;
    }
    if (!Q && blockIdx.x == 0 && threadIdx.x == 0) row_ptr[N] = N * (int64_t)k;
    for (int64_t f = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); f < rows;
         f += nw) {
        const int64_t p = Q ? (int64_t)fb_in[f] : f;
        if (!Q && lane == 0) row_ptr[p] = p * (int64_t)k;
        // The splits' lists are sorted by (distance, index) and cover
        // disjoint columns, so the position of an entry in their union is its
        // position in its own list plus, for every other list, the number of
        // that list's entries ordered before it (a binary search; equal keys
        // count from earlier lists only, so positions stay distinct).  Empty
        // slots are (+inf, no index) and follow every entry.
        const int wib = threadIdx.x >> 5;
        float* sd = s_d[wib];
        int* si = s_i[wib];
        const int total = splits * KC;
#pragma unroll
        for (int m = 0; m < E; ++m) {
            const int e = lane + 32 * m;
            if (e < total) {
                const int64_t o = ((int64_t)(e / KC) * stride + f) * KC + (e % KC);
                const int i = cand_i[o];
                sd[e] = i >= 0 ? cand_d[o] : kInf;
                si[e] = i >= 0 ? i : kNoIdx;
            }
        }
        __syncwarp();
        int rk[E];   // E >= ceil(splits KC / 32) entries per lane
#pragma unroll
        for (int m = 0; m < E; ++m) {
            const int e = lane + 32 * m;
            rk[m] = 0x7fffffff;
            if (e >= total) continue;
            const float xd = sd[e];
            const int xi = si[e];
            if (xi == kNoIdx) continue;   // empty slots are never selected
            const int l = e / KC;
            int r = 0;
            for (int l2 = 0; l2 < splits; ++l2) {
                int c;
                if (l2 == l) {
                    c = e % KC;
                } else {
                    const float* bd = sd + l2 * KC;
                    const int* bi = si + l2 * KC;
                    const bool eq = l2 < l;
                    c = 0;
#pragma unroll
                    for (int w = KC / 2; w > 0; w >>= 1) {
                        const float od = bd[c + w - 1];
                        const int oi = bi[c + w - 1];
                        if (lex_less(od, oi, xd, xi) || (eq && od == xd && oi == xi)) c += w;
                    }
                    const float od = bd[c];
                    const int oi = bi[c];
                    if (lex_less(od, oi, xd, xi) || (eq && od == xd && oi == xi)) ++c;
                }
                r += c;
            }
            rk[m] = r;
        }
        // the row itself is not a neighbour: entries after it move up one
        int self_rank = 0x7fffffff;
#pragma unroll
        for (int m = 0; m < E; ++m)
            if (lane + 32 * m < total && si[lane + 32 * m] == (int)p) self_rank = rk[m];
        self_rank = __reduce_min_sync(0xffffffffu, self_rank);
        float* od_ = s_od[wib];
        int* oi_ = s_oi[wib];
        int nv = 0;
#pragma unroll
        for (int m = 0; m < E; ++m) {
            const int e = lane + 32 * m;
            const int xi = e < total ? si[e] : kNoIdx;
            const bool valid = xi != kNoIdx && xi != (int)p;
            nv += __popc(__ballot_sync(0xffffffffu, valid));
            const int r = rk[m] - (rk[m] > self_rank ? 1 : 0);
            if (valid && r < SEL) {
                od_[r] = sd[e];
                oi_[r] = xi;
            }
        }
        __syncwarp();
        // candidate c lives on lane c % 32, slot c / 32
        constexpr int CPL = (SEL + 31) / 32;
        const int nc = nv < SEL ? nv : SEL;
        int ci[CPL];
        float cd[CPL];
#pragma unroll
        for (int h = 0; h < CPL; ++h) {
            const int c = lane + 32 * h;
            ci[h] = c < nc ? oi_[c] : kNoIdx;
            cd[h] = c < nc ? od_[c] : kInf;
        }
        float T = nc == SEL ? od_[SEL - 1] : kInf;
        __syncwarp();   // read before the next row's lists are staged
        // Lower bound T on dt of every point that is not a candidate: a column
        // a split rejected has dt >= that split's last list entry (when its
        // list is full); an entry of the union left out has dt >= the SEL-th
        // selected one.
        {
            float ts = kInf;
            if (lane < splits) {
                const int64_t o = ((int64_t)lane * stride + f) * KC + (KC - 1);
                if (cand_i[o] >= 0) ts = cand_d[o];
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) ts = fminf(ts, __shfl_xor_sync(0xffffffffu, ts, o));
            T = fminf(T, ts);
        }
        // Candidates that cannot be among the k nearest need no exact
        // distance.  With |dt - |xt_p - xt_q|^2| <= delta_q =
        // coef (|xt_p| + |xt_q|)^2 and |xt - (x - mu)| <= rho, the exact
        // distance of candidate c = q lies in
        // [lb_c, ub_c] = [(sqrt(dt - delta_q) - rho_p - rho_q)^2,
        // (sqrt(dt + delta_q) + rho_p + rho_q)^2].  Every ub_c is at most the
        // same bound taken with the largest norm and rho of all rows, which
        // grows with dt, and the candidates come in increasing dt, so the
        // k-th smallest ub is at most that bound of candidate k - 1 (U); a
        // candidate whose own lb exceeds U (by more than the float32
        // rounding of the exact sums) is beaten by k candidates whatever the
        // rounding.  Skipped candidates keep an infinite distance, so they
        // rank after every computed one and the k nearest, their distances
        // and the certificate are unchanged.
        unsigned need[CPL];
        {
            const float npf = norms[p];
            const float rp = MODE == 1 ? 5.9604645e-08f * 1.000001f * sqrtf(npf) : rho[p] * 1.000001f;
            const float snp = sqrtf(npf) * 1.000001f;   // the row's own terms
            const float rr = rp + rmax_f;
            const float snf = snp + snmax_f;
            const float dl = coef_f * snf * snf;
            float U = kInf;
            if (nc >= k) {
                float dkt = kInf;
#pragma unroll
                for (int h = 0; h < CPL; ++h)
                    if ((k - 1) / 32 == h) dkt = __shfl_sync(0xffffffffu, cd[h], (k - 1) % 32);
                const float a = sqrtf(dkt + dl) + rr;
                U = a * a * 1.00001f;
            }
            const float lim = U * keep_f;
#pragma unroll
            for (int h = 0; h < CPL; ++h) {
                bool keep = false;
                if (lane + 32 * h < nc) {
                    const int q = ci[h];
                    const float nqf = norms[q];
                    const float rq = (MODE == 1 ? 5.9604645e-08f * 1.000001f * sqrtf(nqf) : rho[q] * 1.000001f);
                    const float snq = snp + sqrtf(nqf) * 1.000001f;
                    const float lo = cd[h] - coef_f * snq * snq;
                    const float r = lo > 0.f ? sqrtf(lo) * 0.99999f - (rp + rq) : 0.f;
                    const float lb = r > 0.f ? r * r * 0.99999f : 0.f;
                    keep = !(lb > lim);
                }
                need[h] = __ballot_sync(0xffffffffu, keep);
            }
        }
        // exact float32 distances of the remaining candidates
        const float* xp = X + p * D;
        float myd[CPL];
#pragma unroll
        for (int h = 0; h < CPL; ++h) myd[h] = kInf;
#pragma unroll
        for (int h = 0; h < CPL; ++h) {
            if (D > 256) {
                // long rows: a candidate's own loads already overlap
                for (unsigned msk = need[h]; msk != 0u; msk &= msk - 1u) {   // warp-uniform
                    const int b = __ffs(msk) - 1;
                    const int q = __shfl_sync(0xffffffffu, ci[h], b);
                    const float d = exact_d2(xp, X + (int64_t)q * D, D, lane);
                    if (lane == b) myd[h] = d;
                }
                continue;
            }
            // short rows: four candidates at a time, their row gathers overlap;
            // each one's sum has exact_d2's per-lane order and butterfly (the
            // same bits)
            unsigned msk = need[h];   // warp-uniform
            while (msk != 0u) {
                int b[4], q[4];
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    b[c] = msk != 0u ? __ffs(msk) - 1 : -1;
                    if (msk != 0u) msk &= msk - 1u;
                    q[c] = __shfl_sync(0xffffffffu, ci[h], b[c] < 0 ? 0 : b[c]);
                }
                float part[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll kRerankUnroll
                for (int j = lane; j < D; j += 32) {
                    const float a = xp[j];
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        if (b[c] >= 0) {
                            const float df = a - X[(int64_t)q[c] * D + j];
                            part[c] = fmaf(df, df, part[c]);
                        }
                    }
                }
#pragma unroll
                for (int c = 0; c < 4; ++c) {
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) part[c] += __shfl_xor_sync(0xffffffffu, part[c], o);
                    if (b[c] >= 0 && lane == b[c]) myd[h] = part[c];
                }
            }
        }
        // rank of each candidate by (exact distance, index) among the
        // computed ones; a skipped one (+inf) ranks after at least k of them
        int rank[CPL];
#pragma unroll
        for (int h = 0; h < CPL; ++h) rank[h] = 0;
#pragma unroll
        for (int hs = 0; hs < CPL; ++hs) {
            for (unsigned msk = need[hs]; msk != 0u; msk &= msk - 1u) {
                const int b = __ffs(msk) - 1;
                const float od = __shfl_sync(0xffffffffu, myd[hs], b);
                const int oi = __shfl_sync(0xffffffffu, ci[hs], b);
#pragma unroll
                for (int h = 0; h < CPL; ++h)
                    if (lex_less(od, oi, myd[h], ci[h])) ++rank[h];
            }
        }
        float dk = kInf;
#pragma unroll
        for (int h = 0; h < CPL; ++h) {
            const bool mine = lane + 32 * h < nc;
            if (mine && rank[h] < k) {
                col_idx[p * k + rank[h]] = ci[h];
                dist2[p * k + rank[h]] = myd[h];
            }
            const unsigned kth = __ballot_sync(0xffffffffu, mine && rank[h] == k - 1);
            if (kth) dk = __shfl_sync(0xffffffffu, myd[h], __ffs(kth) - 1);
        }
        if (lane == 0 && T < kInf) {
            bool ok = false;
            const double np_ = (double)norms[p];
            const double rp = MODE == 1 ? u * sqrt(np_) * (1.0 + 1e-6) : (double)rho[p];
            // every point q outside the candidates must be farther than
            // K = dk (1 + 2.02 err_exact), the k-th candidate's exact distance
            // inflated by its rounding.  With y = x - mu, a q with |y_q| >=
            // |y_p| + sqrt(K) is (|y_q| - |y_p| >= sqrt(K)); any other has
            // |y_q| < R = |xt_p| + rho_p + sqrt(K), hence rho_q <= kappa
            // ||v_q|| <= kappa (1 + u) R and |xt_q| < R + rho_q.  Its
            // distance is at least (sqrt(T - delta_q) - rho_p - rho_q)^2 with
            // delta_q = coef (|xt_p| + |xt_q|)^2 (tile arithmetic gam, the
            // norms' float32 lane sums and roundings), |xt_q| and rho_q taken
            // at the smaller of these bounds and the largest norm and rho of
            // all rows.
            const double K = (double)dk * (1.0 + 2.02 * err_exact);
            const double sp = sqrt(np_) * (1.0 + (double)(Dp / 32 + 4) * u);
            const double R = (sp + rp + sqrt(K)) * (1.0 + 1e-9);
            const double rq = fmin(rmax, kappa * (1.0 + u) * R * (1.0 + 1e-9));
            const double sn = fmin(sqrt(np_) + sqrt(nmax), sp + R + rq);
            const double delta = (gam + (double)(Dp / 32 + 5) * u) * sn * sn;
            const double tt = (double)T - delta;
            if (tt > 0.0) {
                const double root = sqrt(tt) - rp - rq;
                if (root > 0.0) {
                    const double lb = root * root * (1.0 - 1e-12);
                    ok = K < lb;
                }
            }
            if (!ok) {
                long long* cnt = Q ? count_out : &st->fallback_count;
                const unsigned long long slot = atomicAdd((unsigned long long*)cnt, 1ull);
                fb_list[slot] = (int32_t)p;
            }
        }
    }
}

// ------------------------------------------- selection from the sweep's lists

// The warp's need mask m over candidates (lane b holds candidate b, its point
// in q_of): exact distances, lane b receives that of candidate b.
__device__ __forceinline__ void exact_of(const float* __restrict__ X, const float* __restrict__ xp, int D,
                                         int lane, unsigned m, int q_of, float& mine) {
    if (D > 256) {
        // long rows: a candidate's own loads already overlap
        for (; m != 0u; m &= m - 1u) {
            const int b = __ffs(m) - 1;
            const int q = __shfl_sync(0xffffffffu, q_of, b);
            const float d = exact_d2(xp, X + (int64_t)q * D, D, lane);
            if (lane == b) mine = d;
        }
        return;
    }
    // short rows: four candidates at a time, their row gathers overlap; each
    // one's sum has exact_d2's per-lane order and butterfly (the same bits)
    while (m != 0u) {
        int b[4], q[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            b[c] = m != 0u ? __ffs(m) - 1 : -1;
            if (m != 0u) m &= m - 1u;
            q[c] = __shfl_sync(0xffffffffu, q_of, b[c] < 0 ? 0 : b[c]);
        }
        float part[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll kRerankUnroll
        for (int j = lane; j < D; j += 32) {
            const float a = xp[j];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                if (b[c] >= 0) {
                    const float df = a - X[(int64_t)q[c] * D + j];
                    part[c] = fmaf(df, df, part[c]);
                }
            }
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) part[c] += __shfl_xor_sync(0xffffffffu, part[c], o);
            if (b[c] >= 0 && lane == b[c]) mine = part[c];
        }
    }
}

struct SelectArgs {
    const float* X;
    int64_t N;
    int D, Dp, k;
    SweepWork w;
    SweepLists lists;
    const int32_t* perm;      // point of each operand column (NULL: the same)
    const float* norms;       // by operand column
    const float* rho;
    double gam;
    int64_t* row_ptr;
    int32_t* col_idx;
    float* dist2;
    int32_t* fb_list;         // rows left open, counted in *fb_count
    unsigned long long* fb_count;
    const DevState* st;
    // two-term stage: rows fb_in[f], f < *count_in; those from cap on are left open
    const int32_t* fb_in;
    const long long* count_in;
    int64_t cap;
};

// k-th smallest dt of a row over the lists of its pieces.  A piece's list holds
// the columns under its own threshold, its k smallest among them, so the
// entries up to the smallest k-th value of any piece (at most k per piece)
// contain the k smallest of the union; ranks by counting.
template <int NK>
__device__ __forceinline__ float union_kth(const SweepLists& ls, int64_t first, int segs,
                                           int64_t extra0, int fr, float kmin, int k, float* sk, int lane,
                                           bool& bad) {
    int m = 0;
    for (int s = 0; s < segs; ++s) {
        const int64_t row = s == 0 ? first : (extra0 + s) * 128 + fr;
        const uint2* src = ls.cand + row * ls.stride;
        const int n = sweep_count(src[0].x);
        for (int e0 = 0; e0 < n; e0 += 32) {
            const float d = e0 + lane < n ? __uint_as_float(src[1 + e0 + lane].x) : kInf;
            const unsigned take = __ballot_sync(0xffffffffu, d <= kmin && d < kInf);
            const int at = m + __popc(take & ((1u << lane) - 1u));
            if (d <= kmin && d < kInf && at < NK) sk[at] = d;
            m += __popc(take);
        }
    }
    if (m > NK || m < k) { bad = true; return kInf; }
    __syncwarp();
    float found = -kInf;
    for (int e = lane; e < m; e += 32) {
        const float d = sk[e];
        int less = 0, leq = 0;
        for (int c = 0; c < m; ++c) {
            less += sk[c] < d;
            leq += sk[c] <= d;
        }
        if (less < k && k <= leq) found = d;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) found = fmaxf(found, __shfl_xor_sync(0xffffffffu, found, o));
    __syncwarp();
    return found;
}

// The k nearest of each row from the candidates the sweep kept, one warp per
// row: the threshold of the k-th smallest dt over all pieces, exact float32
// distances of the candidates whose lower bound can still reach the k nearest,
// the k smallest by (distance, index).  Every column that is no candidate has
// dt >= T (or a squared operand distance >= T), which certifies the row unless
// its k-th exact distance is too close to that (knn_cert.cuh); it is also left
// open if a list gave up on ties or more than 64 candidates remain (128 in the
// two-term stage, whose row blocks come in more pieces).
template <bool SPLIT>
__global__ void __launch_bounds__(256, 4)
knn_select_kernel(const SelectArgs a) {
    constexpr int NK = kSweepMaxSeg * SLK_MAX_K;
    __shared__ float s_k[8][NK];
    constexpr int kSelMax = SPLIT ? 128 : 64, CPL = kSelMax / 32;
    __shared__ float s_d[8][kSelMax];
    __shared__ int s_i[8][kSelMax];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, k = a.k, D = a.D;
    const int64_t nw = (int64_t)gridDim.x * (blockDim.x >> 5);
    const DevState* st = a.st;
    const CertConsts cc = SPLIT ? cert_make(a.gam, a.Dp, D, st->knn_max_norm_s_bits, st->knn_max_rho_s_bits,
                                            st->knn_max_kappa_s_bits)
                                : cert_make(a.gam, a.Dp, D, st->knn_max_norm_bits, st->knn_max_rho_bits,
                                            st->knn_max_kappa_bits);
    SweepWork w = a.w;
    int64_t rows = a.N;
    if (SPLIT) {
        rows = (int64_t)(*(const volatile long long*)a.count_in);
        const int64_t in = rows < a.cap ? rows : a.cap;
        w.row_blocks = (int)((in + 127) / 128);
    }
    const int64_t chunk = sweep_chunk(w, sweep_total(w));
    if (!SPLIT && blockIdx.x == 0 && threadIdx.x == 0) a.row_ptr[a.N] = a.N * (int64_t)k;
    for (int64_t f = (int64_t)blockIdx.x * (blockDim.x >> 5) + wib; f < rows; f += nw) {
        const int64_t c0 = SPLIT ? (int64_t)a.fb_in[f] : f;   // the row's own operand column
        const int64_t p = a.perm ? (int64_t)a.perm[c0] : c0;
        bool bad = SPLIT && f >= a.cap;   // beyond the query stage's capacity: on to the next stage
        int nc = 0;
        float T = kInf, lim = kInf;   // columns that are no candidate have dt >= T
        const float np_ = a.norms[c0];
        const float sp = sqrtf(np_) * cc.sn_infl, rp = a.rho[c0] * 1.000001f;
        if (!SPLIT && lane == 0) a.row_ptr[p] = p * (int64_t)k;
        if (!bad) {
            const int rb = (int)(f >> 7), fr = (int)(f & 127);
            int64_t s0, s1;
            sweep_block(w, rb, s0, s1);
            const int64_t u0 = s0 / chunk;
            const int segs = s1 > s0 ? (int)((s1 - 1) / chunk - u0) + 1 : 1;
            const int64_t extra0 = (int64_t)a.w.row_blocks + u0;   // slot of piece s > 0: extra0 + s
            // headers of the pieces
            int n = 0;
            float kt = kInf, tc = kInf;
            if (lane < segs) {
                const int64_t row = lane == 0 ? f : (extra0 + lane) * 128 + fr;
                const uint2* src = a.lists.cand + row * a.lists.stride;
                const uint2 h = src[0];
                n = sweep_count(h.x);
                kt = __uint_as_float(h.y);
                if (sweep_capped(h.x)) tc = __uint_as_float(src[1 + n].x);
            }
            bad = __any_sync(0xffffffffu, n < 0);
            float dk = kt;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                dk = fminf(dk, __shfl_xor_sync(0xffffffffu, dk, o));
                tc = fminf(tc, __shfl_xor_sync(0xffffffffu, tc, o));
            }
            if (!bad && segs > 1)
                dk = union_kth<NK>(a.lists, f, segs, extra0, fr, dk, k, s_k[wib], lane, bad);
            if (!(dk < kInf)) bad = true;
            if (!bad) {
                T = fminf(tc, cert_thr(cc, sp, rp, dk));
                const float sk = cert_reach(cc, sp, rp, dk);
                lim = sk * sk * 1.00001f + 1e-30f;
                for (int s = 0; s < segs; ++s) {
                    const int64_t row = s == 0 ? f : (extra0 + s) * 128 + fr;
                    const uint2* src = a.lists.cand + row * a.lists.stride;
                    const int ns = __shfl_sync(0xffffffffu, n, s);
                    for (int e0 = 0; e0 < ns; e0 += 32) {
                        const bool in = e0 + lane < ns;
                        const uint2 v = in ? src[1 + e0 + lane] : make_uint2(0u, 0u);
                        const bool take = in && __uint_as_float(v.x) < T;
                        const unsigned tm = __ballot_sync(0xffffffffu, take);
                        const int at = nc + __popc(tm & ((1u << lane) - 1u));
                        if (take && at < kSelMax) {
                            s_d[wib][at] = __uint_as_float(v.x);
                            s_i[wib][at] = (int)v.y;
                        }
                        nc += __popc(tm);
                    }
                }
                if (nc > kSelMax || nc < k) bad = true;
            }
        }
        if (bad) {
            if (lane == 0) a.fb_list[atomicAdd(a.fb_count, 1ull)] = (int32_t)p;
            continue;
        }
        __syncwarp();
        // candidate c lives on lane c % 32, slot c / 32; one whose lower bound
        // (its own norm and rho) exceeds the reach of the k nearest needs no
        // exact distance
        int ci[CPL];
        float myd[CPL];
        unsigned need[CPL];
#pragma unroll
        for (int h = 0; h < CPL; ++h) {
            const int c = lane + 32 * h;
            bool keep = false;
            ci[h] = kNoIdx;
            myd[h] = kInf;
            need[h] = 0u;
            if (32 * h >= nc) continue;   // warp-uniform
            if (c < nc) {
                const int q = s_i[wib][c];
                ci[h] = a.perm ? a.perm[q] : q;
                const float rq = a.rho[q] * 1.000001f;
                const float snq = sp + sqrtf(a.norms[q]) * cc.sn_infl;
                const float lo = s_d[wib][c] - cc.coef * snq * snq;
                const float r = lo > 0.f ? sqrtf(lo) * 0.99999f - (rp + rq) : 0.f;
                const float lb = r > 0.f ? r * r * 0.99999f : 0.f;
                keep = !(lb > lim);
            }
            need[h] = __ballot_sync(0xffffffffu, keep);
        }
        __syncwarp();
        const float* xp = a.X + p * D;
#pragma unroll
        for (int h = 0; h < CPL; ++h) exact_of(a.X, xp, D, lane, need[h], ci[h], myd[h]);
        // rank of each candidate by (exact distance, index) among the computed
        // ones; a skipped one (+inf) ranks after at least k of them
        int rank[CPL];
#pragma unroll
        for (int h = 0; h < CPL; ++h) rank[h] = 0;
#pragma unroll
        for (int hs = 0; hs < CPL; ++hs) {
            for (unsigned m = need[hs]; m != 0u; m &= m - 1u) {
                const int b = __ffs(m) - 1;
                const float od = __shfl_sync(0xffffffffu, myd[hs], b);
                const int oi = __shfl_sync(0xffffffffu, ci[hs], b);
#pragma unroll
                for (int h = 0; h < CPL; ++h)
                    if (lex_less(od, oi, myd[h], ci[h])) ++rank[h];
            }
        }
        float dk = kInf;
#pragma unroll
        for (int h = 0; h < CPL; ++h) {
            if (lane + 32 * h < nc && rank[h] < k) {
                a.col_idx[p * k + rank[h]] = ci[h];
                a.dist2[p * k + rank[h]] = myd[h];
                if (rank[h] == k - 1) dk = myd[h];
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) dk = fminf(dk, __shfl_xor_sync(0xffffffffu, dk, o));
        if (lane == 0 && !cert_ok(cc, sp, rp, dk, T)) a.fb_list[atomicAdd(a.fb_count, 1ull)] = (int32_t)p;
    }
}

// ------------------------------------------------------------ exact fallback

// One block per listed row: 8 warps scan disjoint column subsets keeping a
// register top-k (lane i holds entry i), then warp 0 merges the 8 lists.
__global__ void __launch_bounds__(256)
knn_fallback_kernel(const float* __restrict__ X, int64_t N, int D, int k,
                    const int32_t* __restrict__ fb_list, const long long* count_ptr,
                    int32_t* __restrict__ col_idx, float* __restrict__ dist2) {
    __shared__ float md[8][32];
    __shared__ int mi[8][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long count = *(const volatile long long*)count_ptr;
    for (long long f = blockIdx.x; f < count; f += gridDim.x) {
        const int64_t p = fb_list[f];
        const float* xp = X + p * D;
        float ld = kInf;
        int li = kNoIdx;
        for (int64_t q = warp; q < N; q += 8) {
            if (q == p) continue;
            const float d = exact_d2(xp, X + q * D, D, lane);
            const float lastd = __shfl_sync(0xffffffffu, ld, k - 1);
            const int lasti = __shfl_sync(0xffffffffu, li, k - 1);
            if (!lex_less(d, (int)q, lastd, lasti)) continue;
            const bool less = lane < k && lex_less(d, (int)q, ld, li);
            const unsigned lm = __ballot_sync(0xffffffffu, less);
            const int pos = __ffs(lm) - 1;
            const float upd = __shfl_up_sync(0xffffffffu, ld, 1);
            const int upi = __shfl_up_sync(0xffffffffu, li, 1);
            if (lane < k) {
                if (lane == pos) { ld = d; li = (int)q; }
                else if (lane > pos) { ld = upd; li = upi; }
            }
        }
        md[warp][lane] = ld;
        mi[warp][lane] = li;
        __syncthreads();
        if (warp == 0) {
            float ed[8];
            int ei[8];
#pragma unroll
            for (int m = 0; m < 8; ++m) {
                ed[m] = lane < k ? md[m][lane] : kInf;
                ei[m] = lane < k ? mi[m][lane] : kNoIdx;
            }
            for (int c = 0; c < k; ++c) {
                float bd = kInf;
                int bi = kNoIdx;
#pragma unroll
                for (int m = 0; m < 8; ++m)
                    if (lex_less(ed[m], ei[m], bd, bi)) { bd = ed[m]; bi = ei[m]; }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    const float od = __shfl_xor_sync(0xffffffffu, bd, o);
                    const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
                    if (lex_less(od, oi, bd, bi)) { bd = od; bi = oi; }
                }
#pragma unroll
                for (int m = 0; m < 8; ++m)
                    if (ei[m] == bi) { ed[m] = kInf; ei[m] = kNoIdx; }
                if (lane == 0) { col_idx[p * k + c] = bi; dist2[p * k + c] = bd; }
            }
        }
        __syncthreads();
    }
}

// Exact rescan for long rows (D above the 32 x 32 features the batched form
// keeps in registers): work items (one failed row, one of cs =
// exact_splits of F column ranges) taken persistently, so that a few
// rows still spread over every SM.  The row's features are staged in shared
// memory; each of the 8 warps streams a share of the range, computing every
// distance with exact_d2 (the same per-lane order and butterfly) and keeping
// a register top-k (lane i holds entry i); the 8 lists are merged into the
// (row, range) partial list at ((f cs + range) k), as the batched form does.
__global__ void __launch_bounds__(256)
knn_fallback_wide_kernel(const float* __restrict__ X, int64_t N, int D, int k, int ctas,
                         const int32_t* __restrict__ fb_list, const long long* count_ptr,
                         long long cap, float* __restrict__ part_d, int32_t* __restrict__ part_i) {
    extern __shared__ float xs[];   // D floats: the row's features
    __shared__ float md[8][32];
    __shared__ int mi[8][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long count = *(const volatile long long*)count_ptr;
    const int col_splits = exact_splits(count, 1, ctas, N, cap, k);
    for (long long item = blockIdx.x; item < count * col_splits; item += gridDim.x) {
        const long long f = item / col_splits;
        const int cs = (int)(item % col_splits);
        const int64_t p = fb_list[f];
        const int64_t q0 = (int64_t)cs * N / col_splits, q1 = (int64_t)(cs + 1) * N / col_splits;
        __syncthreads();   // the previous item is done with xs and md / mi
        for (int j = threadIdx.x; j < D; j += blockDim.x) xs[j] = X[p * D + j];
        __syncthreads();
        float ld = kInf;
        int li = kNoIdx;
        for (int64_t q = q0 + warp; q < q1; q += 8) {
            if (q == p) continue;
            const float d = exact_d2(xs, X + q * D, D, lane);
            const float lastd = __shfl_sync(0xffffffffu, ld, k - 1);
            const int lasti = __shfl_sync(0xffffffffu, li, k - 1);
            if (!lex_less(d, (int)q, lastd, lasti)) continue;
            const bool less = lane < k && lex_less(d, (int)q, ld, li);
            const int pos = __ffs(__ballot_sync(0xffffffffu, less)) - 1;
            const float upd = __shfl_up_sync(0xffffffffu, ld, 1);
            const int upi = __shfl_up_sync(0xffffffffu, li, 1);
            if (lane < k) {
                if (lane == pos) { ld = d; li = (int)q; }
                else if (lane > pos) { ld = upd; li = upi; }
            }
        }
        md[warp][lane] = lane < k ? ld : kInf;
        mi[warp][lane] = lane < k ? li : kNoIdx;
        __syncthreads();
        if (warp == 0) {
            float ed[8];
            int ei[8];
#pragma unroll
            for (int m = 0; m < 8; ++m) { ed[m] = md[m][lane]; ei[m] = mi[m][lane]; }
            for (int c = 0; c < k; ++c) {
                float bd = kInf;
                int bi = kNoIdx;
#pragma unroll
                for (int m = 0; m < 8; ++m)
                    if (lex_less(ed[m], ei[m], bd, bi)) { bd = ed[m]; bi = ei[m]; }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    const float od = __shfl_xor_sync(0xffffffffu, bd, o);
                    const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
                    if (lex_less(od, oi, bd, bi)) { bd = od; bi = oi; }
                }
#pragma unroll
                for (int m = 0; m < 8; ++m)
                    if (ei[m] == bi) { ed[m] = kInf; ei[m] = kNoIdx; }
                if (lane == 0) {
                    part_d[(f * col_splits + cs) * k + c] = bd;
                    part_i[(f * col_splits + cs) * k + c] = bi;
                }
            }
        }
    }
}

// Batched exact rescan of the rows that failed the certificate.  Work items
// (R failed rows, one of cs = exact_splits of F column ranges) are
// taken persistently, so the grid does not depend on the count F.  The R
// rows' features are cached in registers, lane-strided like exact_d2; each
// of the block's 8 warps streams a share of the column range once for all R
// rows, computing every distance with exact_d2's arithmetic (same per-lane
// fmaf order, same butterfly), and keeps a register top-k per row (lane i
// holds entry i).  The 8 warp lists are merged in shared memory into one
// list per (row, column range), written to part_d / part_i at
// ((f cs + range) k).
template <int R, int DPL>
__global__ void __launch_bounds__(256)
knn_fallback_batch_kernel(const float* __restrict__ X, int64_t N, int D, int k, int ctas,
                          const int32_t* __restrict__ fb_list, const long long* count_ptr,
                          long long cap, float* __restrict__ part_d,
                          int32_t* __restrict__ part_i) {
    __shared__ float md[8][R][32];
    __shared__ int mi[8][R][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long count = *(const volatile long long*)count_ptr;
    const long long nbatch = (count + R - 1) / R;
    const int col_splits = exact_splits(count, R, ctas, N, cap, k);
    for (long long item = blockIdx.x; item < nbatch * col_splits; item += gridDim.x) {
        const long long b = item / col_splits;
        const int cs = (int)(item % col_splits);
        const int64_t q0 = (int64_t)cs * N / col_splits, q1 = (int64_t)(cs + 1) * N / col_splits;
        int64_t prow[R];
        float xr[R][DPL];
        float ld[R], lastd[R];
        int li[R], lasti[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const long long f = b * R + r;
            prow[r] = (f < count) ? (int64_t)fb_list[f] : -1;
#pragma unroll
            for (int t = 0; t < DPL; ++t) {
                const int j = lane + 32 * t;
                xr[r][t] = (prow[r] >= 0 && j < D) ? X[prow[r] * D + j] : 0.f;
            }
            ld[r] = kInf; li[r] = kNoIdx; lastd[r] = kInf; lasti[r] = kNoIdx;
        }
        // the next column's features are loaded while this one is summed
        float xq[DPL];
#pragma unroll
        for (int t = 0; t < DPL; ++t) {
            const int j = lane + 32 * t;
            xq[t] = (q0 + warp < q1 && j < D) ? X[(q0 + warp) * D + j] : 0.f;
        }
        for (int64_t q = q0 + warp; q < q1; q += 8) {
            float xn[DPL];
#pragma unroll
            for (int t = 0; t < DPL; ++t) {
                const int j = lane + 32 * t;
                xn[t] = (q + 8 < q1 && j < D) ? X[(q + 8) * D + j] : 0.f;
            }
            // every row's lane sums, then their butterflies side by side (the
            // R chains overlap), then the insertions; each sum in exact_d2's order
            float part[R];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                part[r] = 0.f;
#pragma unroll
                for (int t = 0; t < DPL; ++t) {
                    if (lane + 32 * t < D) {
                        const float df = xr[r][t] - xq[t];
                        part[r] = fmaf(df, df, part[r]);
                    }
                }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
#pragma unroll
                for (int r = 0; r < R; ++r) part[r] += __shfl_xor_sync(0xffffffffu, part[r], o);
#pragma unroll
            for (int r = 0; r < R; ++r) {
                if (prow[r] < 0 || q == prow[r]) continue;
                if (!lex_less(part[r], (int)q, lastd[r], lasti[r])) continue;
                const bool less = lane < k && lex_less(part[r], (int)q, ld[r], li[r]);
                const int pos = __ffs(__ballot_sync(0xffffffffu, less)) - 1;
                const float upd = __shfl_up_sync(0xffffffffu, ld[r], 1);
                const int upi = __shfl_up_sync(0xffffffffu, li[r], 1);
                if (lane < k) {
                    if (lane == pos) { ld[r] = part[r]; li[r] = (int)q; }
                    else if (lane > pos) { ld[r] = upd; li[r] = upi; }
                }
                lastd[r] = __shfl_sync(0xffffffffu, ld[r], k - 1);
                lasti[r] = __shfl_sync(0xffffffffu, li[r], k - 1);
            }
#pragma unroll
            for (int t = 0; t < DPL; ++t) xq[t] = xn[t];
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
            md[warp][r][lane] = lane < k ? ld[r] : kInf;
            mi[warp][r][lane] = lane < k ? li[r] : kNoIdx;
        }
        __syncthreads();
        for (int r = warp; r < R; r += 8) {
            const long long f = b * R + r;
            if (f >= count) continue;
            float ed[8];
            int ei[8];
#pragma unroll
            for (int m = 0; m < 8; ++m) { ed[m] = md[m][r][lane]; ei[m] = mi[m][r][lane]; }
            for (int c = 0; c < k; ++c) {
                float bd = kInf;
                int bi = kNoIdx;
#pragma unroll
                for (int m = 0; m < 8; ++m)
                    if (lex_less(ed[m], ei[m], bd, bi)) { bd = ed[m]; bi = ei[m]; }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    const float od = __shfl_xor_sync(0xffffffffu, bd, o);
                    const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
                    if (lex_less(od, oi, bd, bi)) { bd = od; bi = oi; }
                }
#pragma unroll
                for (int m = 0; m < 8; ++m)
                    if (ei[m] == bi) { ed[m] = kInf; ei[m] = kNoIdx; }
                if (lane == 0) {
                    part_d[(f * col_splits + cs) * k + c] = bd;
                    part_i[(f * col_splits + cs) * k + c] = bi;
                }
            }
        }
        __syncthreads();
    }
}

// Merge the partial lists of every failed row (cs = exact_splits of F
// of k entries at ((f cs) k)) into its k nearest: chunks of 7 entries per
// lane beside the running k best (lane i holds entry i), k rounds of a warp
// minimum per chunk.
__global__ void __launch_bounds__(256)
knn_fallback_merge_kernel(int64_t N, int together, int ctas, int k,
                          const int32_t* __restrict__ fb_list, const long long* count_ptr,
                          long long cap, const float* __restrict__ part_d,
                          const int32_t* __restrict__ part_i, int32_t* __restrict__ col_idx,
                          float* __restrict__ dist2) {
    const int lane = threadIdx.x & 31;
    const long long count = *(const volatile long long*)count_ptr;
    const int col_splits = exact_splits(count, together, ctas, N, cap, k);
    const int total = col_splits * k;
    const int64_t nw = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t f = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); f < count;
         f += nw) {
        const int64_t p = fb_list[f];
        const float* pd = part_d + f * total;
        const int32_t* pi = part_i + f * total;
        float bestd = kInf;   // lane i < k: the i-th best so far
        int besti = kNoIdx;
        for (int e0 = 0; e0 < total; e0 += 7 * 32) {
            float ed[8];
            int ei[8];
            ed[7] = bestd;
            ei[7] = besti;
#pragma unroll
            for (int m = 0; m < 7; ++m) {
                const int e = e0 + lane + 32 * m;
                ed[m] = e < total ? pd[e] : kInf;
                ei[m] = e < total ? pi[e] : kNoIdx;
            }
            for (int c = 0; c < k; ++c) {
                float bd = kInf;
                int bi = kNoIdx;
#pragma unroll
                for (int m = 0; m < 8; ++m)
                    if (lex_less(ed[m], ei[m], bd, bi)) { bd = ed[m]; bi = ei[m]; }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    const float od = __shfl_xor_sync(0xffffffffu, bd, o);
                    const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
                    if (lex_less(od, oi, bd, bi)) { bd = od; bi = oi; }
                }
                // the winner is unique (distinct indices): remove it where it sits
#pragma unroll
                for (int m = 0; m < 8; ++m)
                    if (ei[m] == bi && ed[m] == bd) { ed[m] = kInf; ei[m] = kNoIdx; }
                if (lane == c) { bestd = bd; besti = bi; }
            }
        }
        if (lane < k) { col_idx[p * k + lane] = besti; dist2[p * k + lane] = bestd; }
    }
}

int choose_kc(int k) { return (k + 4 <= 16) ? 16 : 32; }

struct KnnPlan {
    int64_t Np;
    int Dp, kc, splits, row_blocks, n_tiles;
    bool bf16;
    bool aug;    // tensor-core tiles with the norms folded into one more K slice
    // tensor-core sweep: CTAs, entries of a row list, and whether its work is
    // cut only between row blocks (no lists beyond one per row)
    int units, stride, aligned;
    // two-term stage (bfloat16 and N >= kTwoTermMinRows): row capacity (a
    // multiple of 128) and CTAs
    bool two_term;
    int64_t fcap;
    int sunits;
    // points sorted by region, tiles out of reach left out (knn_group.cu)
    bool grouped;
};

// Sweeps shorter than this are not worth the sort's launches (0.15 to 0.2 ms).
// Tiles per CTA times K slices and their fixed part: 490 at 19937 x 256 (0.46 ms
// grouped, 0.47 not), 1060 at 30000 x 64 (0.47 and 0.85), 14800 at 70000 x 784
// with 10 clusters (1.70 and 5.69; with one cluster, where nothing can be left
// out, 6.21 and 5.65).
constexpr int64_t kGroupMinWork = 500;
// Tiles around a row block's own columns that the first pass takes: 4, and 8
// from 2000 column tiles on, where regions are longer (4 against 8: 0.39 and
// 0.45 ms at 42099 x 64, 4.93 and 5.23 at 200000 x 128, 88.7 and 85.5 at 1e6 x
// 128).
int group_window(int n_tiles) { return n_tiles < 2000 ? 4 : 8; }

// Rows the two-term tensor-core stage takes at most (fewer at large D, see
// make_plan); the open rows beyond it go to the float32 stage.
constexpr int64_t kSplitRowCap = 65536;
// Below this many points the open rows go straight to the float32 stage (its
// tiles over N points are cheap there, and the two-term stage's four launches
// would cost more than they save: the batched form runs many such graphs).
constexpr int64_t kTwoTermMinRows = 100000;
constexpr int kTcCols = 256;   // columns of a tensor-core tile

size_t plan_bytes(const KnnPlan& pl, int64_t N, int D);

// The plan, within `budget` bytes of workspace: with too little for row lists
// of 64 entries and one list more per CTA, lists of 32 and whole row blocks
// per CTA (slower, more rows left open; the same graph).
KnnPlan make_plan(const slk_ctx* ctx, int64_t N, int D, int k, int precision, size_t budget) {
    KnnPlan pl{};
    pl.bf16 = (precision == SLK_KNN_BF16_RERANK);
    pl.kc = choose_kc(k);
    // the tensor-core tiles read 256-row column tiles: keep them inside the matrix
    pl.Np = (int64_t)align_up((size_t)N, pl.bf16 ? 256 : 128);
    pl.Dp = (int)align_up((size_t)D, pl.bf16 ? 64 : BK);
    pl.row_blocks = (int)(pl.Np / BM);
    const int sms = ctx->num_sms > 0 ? ctx->num_sms : 148;
    if (pl.bf16) {
        // where the tiles' epilogue outweighs their MMAs (small D), fold the
        // norms into the MMAs: the epilogue then reads no norms
        pl.aug = pl.Dp <= 256;
        pl.n_tiles = (int)(pl.Np / kTcCols);
        const int64_t tiles = (int64_t)pl.row_blocks * pl.n_tiles;
        pl.units = (int)std::min<int64_t>(sms, tiles);
        // two-term query rows: at most 65536, and operands (h and l) of at most 64 MiB
        const int64_t by_mem = std::max<int64_t>(128, ((int64_t)1 << 24) / pl.Dp / 128 * 128);
        pl.fcap = std::min<int64_t>(std::min<int64_t>((int64_t)align_up((size_t)N, 128), kSplitRowCap),
                                    by_mem);
        pl.sunits = (int)std::min<int64_t>(sms, 4 * (pl.fcap / 128));
        pl.two_term = N >= kTwoTermMinRows;
        pl.stride = kSweepStride;
        pl.aligned = 0;
        // the tile table must stay a small part of the workspace
        pl.grouped = tiles / pl.units * (2 + pl.Dp / 64) >= kGroupMinWork && pl.n_tiles < 65536 &&
                     pl.n_tiles > 16 && pl.n_tiles <= 32 * (kSweepStride * 8 + 2 * pl.Dp);
        if (pl.grouped && plan_bytes(pl, N, D) > budget) pl.grouped = false;
        if (plan_bytes(pl, N, D) > budget) {
            pl.stride = 32;
            pl.aligned = 1;
        }
        return pl;
    }
    pl.n_tiles = (int)(pl.Np / BN);
    const int max_splits = (32 * MAXE) / pl.kc;
    const int cap = 2 * sms;  // resident CTAs
    // smallest split count giving >= 2 waves, then the one with the best wave fill
    int best = 1;
    double best_eff = -1.0;
    for (int s = 1; s <= max_splits && s <= pl.n_tiles; ++s) {
        const int64_t total = (int64_t)pl.row_blocks * s;
        const int64_t waves = (total + cap - 1) / cap;
        double eff = (double)total / (double)(waves * cap);
        if (total < 2 * cap && s < max_splits && s < pl.n_tiles) eff *= 0.5;  // too few CTAs
        if (eff > best_eff + 1e-9) { best_eff = eff; best = s; }
        if (total >= 8 * cap) break;
    }
    pl.splits = best;
    return pl;
}

// Row lists of the sweeps (rows of 128-row slots).
size_t sweep_rows(const KnnPlan& pl) {
    return (size_t)pl.Np + (pl.aligned ? 0 : (size_t)pl.units * 128);
}
// Floats of one of the two halves of the candidate buffer (distances, indices).
size_t cand_floats(const KnnPlan& pl) {
    return pl.bf16 ? sweep_rows(pl) * pl.stride : (size_t)pl.splits * pl.Np * pl.kc;
}

// The scratch of a graph, in the order of knn_graph_launch.
struct KnnBufs {
    double* colsum;
    void* xt;
    float *norms, *rho, *cand_d;
    int32_t *cand_i, *fb;
    float *norms32, *mu;
    int32_t* fb2;
    __nv_bfloat16* xl16;
    float *norms_s, *rho_s;
    __nv_bfloat16 *qh, *ql;
    float* qnorm;
    uint2* scand;
    __nv_bfloat16* aug;
    GroupBufs grp;
};
KnnBufs carve_knn(WsCarver& wc, const KnnPlan& pl, int64_t N, int D) {
    KnnBufs b{};
    b.colsum = wc.take<double>(D);
    b.xt = wc.take<unsigned char>((pl.bf16 ? 2 : 4) * (size_t)pl.Np * pl.Dp);
    b.norms = wc.take<float>(pl.Np);
    b.rho = wc.take<float>(pl.Np);
    // one block: float32 lists in two halves, the sweep's lists as pairs
    b.cand_d = wc.take<float>(2 * cand_floats(pl));
    b.cand_i = reinterpret_cast<int32_t*>(b.cand_d + cand_floats(pl));
    b.fb = wc.take<int32_t>(N);
    b.norms32 = wc.take<float>(pl.Np);
    b.mu = wc.take<float>(D);
    b.fb2 = wc.take<int32_t>(N);
    if (pl.bf16 && pl.two_term) {
        b.xl16 = wc.take<__nv_bfloat16>((size_t)pl.Np * pl.Dp);
        b.norms_s = wc.take<float>(pl.Np);
        b.rho_s = wc.take<float>(pl.Np);
        b.qh = wc.take<__nv_bfloat16>((size_t)pl.fcap * pl.Dp);
        b.ql = wc.take<__nv_bfloat16>((size_t)pl.fcap * pl.Dp);
        b.qnorm = wc.take<float>(pl.fcap);
        b.scand = wc.take<uint2>(((size_t)pl.fcap + (size_t)pl.sunits * 128) * kSweepStride);
    }
    if (pl.aug) b.aug = wc.take<__nv_bfloat16>(32 * (size_t)pl.Np);
    if (pl.grouped) group_carve(wc, b.grp, N, pl.Np, pl.Dp, pl.n_tiles);
    return b;
}
size_t plan_bytes(const KnnPlan& pl, int64_t N, int D) {
    WsCarver wc(nullptr);
    carve_knn(wc, pl, N, D);
    return wc.off + 4096;
}

}  // namespace

size_t knn_ws_bytes(const slk_ctx* ctx, int64_t N, int D, int k, int precision) {
    return plan_bytes(make_plan(ctx, N, D, k, precision, SIZE_MAX), N, D);
}
size_t knn_ws_min_bytes(const slk_ctx* ctx, int64_t N, int D, int k, int precision) {
    return plan_bytes(make_plan(ctx, N, D, k, precision, 0), N, D);
}

namespace {

// Column sums, mu and the prepared rows on the context's stream; 16-byte
// loads where the row layout and the summation bound allow them.
slk_status launch_prep(slk_ctx* ctx, const float* X, int64_t N, int D, int Dp, int64_t Np,
                       double* colsum, float* mu, float* xt32, __nv_bfloat16* xt16,
                       float* norms, float* rho, float* norms32, __nv_bfloat16* aug, const GroupBufs* grp,
                       DevState* st, bool tiles = false) {
    cudaStream_t s = ctx->stream;
    const bool v4 = D % 4 == 0 && Dp >= 128 && (reinterpret_cast<uintptr_t>(X) & 15) == 0 &&
                    (reinterpret_cast<uintptr_t>(mu) & 15) == 0;
    int gy = (int)((N + 511) / 512);   // 64 rows per thread
    if (gy > 8192) gy = 8192;
    if (gy < 1) gy = 1;
    const int groups = v4 ? D / 4 : D;
    const dim3 cgrid((unsigned)((groups + 31) / 32), (unsigned)gy);
    if (v4) col_sum_kernel<4><<<cgrid, dim3(32, 8), 0, s>>>(X, N, D, colsum);
    else col_sum_kernel<1><<<cgrid, dim3(32, 8), 0, s>>>(X, N, D, colsum);
    mu_kernel<<<(D + 255) / 256, 256, 0, s>>>(colsum, N, D, mu);
    SLK_LAUNCH_CHECK(ctx, "col_sum_kernel");
    const int32_t* perm = nullptr;
    if (grp) {
        const slk_status r = group_order_launch(ctx, *grp, X, N, D, Dp, mu);
        if (r != SLK_OK) return r;
        perm = grp->perm;
    }
    int64_t pg = (Np + 7) / 8;
    if (pg > (int64_t)ctx->num_sms * 64) pg = (int64_t)ctx->num_sms * 64;
    const Operand to = xt16 ? Operand::bf16 : tiles ? Operand::f32_tiles : Operand::f32_rows;
    if (v4)
        prep_rows_kernel<4><<<(unsigned)pg, 256, 0, s>>>(X, N, D, Dp, Np, mu, to, xt32, xt16,
                                                         norms, rho, norms32, aug, perm, st);
    else
        prep_rows_kernel<1><<<(unsigned)pg, 256, 0, s>>>(X, N, D, Dp, Np, mu, to, xt32, xt16,
                                                         norms, rho, norms32, aug, perm, st);
    SLK_LAUNCH_CHECK(ctx, "prep_rows_kernel");
    return SLK_OK;
}

}  // namespace

slk_status knn_prep_fp32_launch(slk_ctx* ctx, const float* X, int64_t N, int D, int Dp, int64_t Np,
                                double* colsum, float* mu, float* xt, float* norms, float* rho,
                                DevState* st) {
    cudaStream_t s = ctx->stream;
    SLK_CUDA_TRY(ctx, cudaMemsetAsync(colsum, 0, sizeof(double) * D, s));
    SLK_CUDA_TRY(ctx, cudaMemsetAsync(&st->knn_max_norm_bits, 0, 2 * sizeof(unsigned int), s));
    SLK_COUNT_LAUNCH(ctx, 2);
    return launch_prep(ctx, X, N, D, Dp, Np, colsum, mu, xt, nullptr, norms, rho, nullptr, nullptr,
                       nullptr, st);
}

slk_status knn_graph_launch(slk_ctx* ctx, const float* X, int64_t N, int D, int k,
                            int precision, int64_t* row_ptr, int32_t* col_idx, float* dist2,
                            void* ws, size_t ws_bytes, DevState* st) {
    const KnnPlan pl = make_plan(ctx, N, D, k, precision, ws_bytes);
    ctx->knn_last_bf16 = pl.bf16;
    ctx->knn_last_two_term = pl.bf16 && pl.two_term;
    WsCarver wc(ws);
    const KnnBufs kb = carve_knn(wc, pl, N, D);
    double* colsum = kb.colsum;
    void* xt = kb.xt;
    float *norms = kb.norms, *rho = kb.rho, *cand_d = kb.cand_d, *norms32 = kb.norms32, *mu = kb.mu;
    int32_t *cand_i = kb.cand_i, *fb = kb.fb, *fb2 = kb.fb2;
    __nv_bfloat16* aug = kb.aug;
    cudaStream_t s = ctx->stream;

    SLK_CUDA_TRY(ctx, cudaMemsetAsync(colsum, 0, sizeof(double) * D, s));
    SLK_CUDA_TRY(ctx, cudaMemsetAsync(&st->fallback_count, 0, sizeof(long long), s));
    SLK_CUDA_TRY(ctx, cudaMemsetAsync(&st->knn_max_norm_bits, 0, 3 * sizeof(unsigned int), s));
    SLK_CUDA_TRY(ctx, cudaMemsetAsync(&st->knn_max_norm32_bits, 0, sizeof(unsigned int), s));
    SLK_CUDA_TRY(ctx, cudaMemsetAsync(&st->fallback2_count, 0, sizeof(long long), s));
    SLK_CUDA_TRY(ctx, cudaMemsetAsync(&st->knn_max_norm_s_bits, 0, 4 * sizeof(unsigned int), s));
    SLK_CUDA_TRY(ctx, cudaMemsetAsync(&st->fallback3_count, 0, sizeof(long long), s));
    SLK_CUDA_TRY(ctx, cudaMemsetAsync(&st->knn_sweep, 0, sizeof(unsigned long long), s));
    {
        PhaseScope ps(ctx, SLK_PHASE_KNN_PREP);
        SLK_COUNT_LAUNCH(ctx, 3);
        const slk_status r = launch_prep(ctx, X, N, D, pl.Dp, pl.Np, colsum, mu,
                                         pl.bf16 ? nullptr : (float*)xt,
                                         pl.bf16 ? (__nv_bfloat16*)xt : nullptr, norms, rho,
                                         pl.bf16 ? norms32 : nullptr, pl.aug ? aug : nullptr,
                                         pl.grouped ? &kb.grp : nullptr, st, !pl.bf16);
        if (r != SLK_OK) return r;
    }
    // rounding unit of a tile's dot-product accumulation: 2^-23 on the tensor
    // cores (products exact, each accumulator add off by at most one ulp,
    // truncating; an assumption), 2^-24 for float32
    const double u_acc = pl.bf16 ? 1.1920928955078125e-07 : 5.9604644775390625e-08;
    // folded norms: 6 more products a dot, and the aug terms' magnitudes
    // (about (n_p + n_q) / 2) join the products' sum: 2 |p| |q| + n_p +
    // n_q = (|p| + |q|)^2, so the bound keeps its form with a 1.01 factor
    const double g_dot = (double)(pl.Dp + (pl.aug ? 6 : 0)) * u_acc;
    const double gam = (pl.aug ? 1.01 : 1.0) * g_dot / (1.0 - g_dot);
    SweepWork work{};
    work.per = work.n_tiles = pl.n_tiles;
    work.row_blocks = pl.row_blocks;
    work.units = pl.units;
    work.aligned = pl.aligned;
    const SweepLists lists{reinterpret_cast<uint2*>(cand_d), pl.stride};
    {
        PhaseScope ps(ctx, SLK_PHASE_KNN_CAND);
        SLK_COUNT_LAUNCH(ctx, 1);
        if (pl.bf16) {
            SweepOperands op{};
            op.a_hi = op.b_hi = (const __nv_bfloat16*)xt;
            op.aug = aug;
            op.row_norms = op.col_norms = norms;
            op.rho = rho;
            op.a_rows = op.b_rows = pl.Np;
            op.N = N;
            op.D = D;
            op.Dp = pl.Dp;
            slk_status r;
            if (pl.grouped) {
                // the tiles around each block, then those that can still matter
                SweepWork first = work;
                first.per = group_window(pl.n_tiles);
                first.aligned = 1;
                r = knn_sweep_launch(ctx, op, first, k, gam, lists, false, kb.grp.thr, kb.grp.kth, st);
                if (r != SLK_OK) return r;
                r = group_tiles_launch(ctx, kb.grp, (const __nv_bfloat16*)xt, N, pl.Np, pl.Dp, first);
                if (r != SLK_OK) return r;
                SLK_COUNT_LAUNCH(ctx, 1);
                work.tiles = kb.grp.tiles;
                work.start = kb.grp.start;
                work.max_cnt = kb.grp.max_cnt;
            }
            r = knn_sweep_launch(ctx, op, work, k, gam, lists, pl.grouped, nullptr,
                                 pl.grouped ? kb.grp.kth : nullptr, st);
            if (r != SLK_OK) return r;
        } else {
#define SLK_CAND(KC_)                                                                         \
    {                                                                                         \
        auto kern = knn_cand_fp32_kernel<KC_>;                                                \
        const int smem = (int)sizeof(CandSmem<KC_>);                                          \
        SLK_CUDA_TRY(ctx, cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem)); \
        kern<<<dim3((unsigned)pl.row_blocks, (unsigned)pl.splits), KT, smem, s>>>(            \
            (const float*)xt, norms, N, pl.Dp, pl.n_tiles, pl.Np, cand_d, cand_i);            \
    }
            if (pl.kc == 16) SLK_CAND(16) else SLK_CAND(32)
#undef SLK_CAND
            SLK_LAUNCH_CHECK(ctx, "knn_cand_fp32_kernel");
        }
    }
    SelectArgs sel{};
    sel.X = X;
    sel.N = N;
    sel.D = D;
    sel.Dp = pl.Dp;
    sel.k = k;
    sel.row_ptr = row_ptr;
    sel.col_idx = col_idx;
    sel.dist2 = dist2;
    sel.st = st;
    {
        PhaseScope ps(ctx, SLK_PHASE_KNN_RERANK);
        SLK_COUNT_LAUNCH(ctx, 1);
        int64_t grid = (N + 7) / 8;
        if (grid > (int64_t)ctx->num_sms * 16) grid = (int64_t)ctx->num_sms * 16;
        if (pl.bf16) {
            sel.w = work;
            sel.lists = lists;
            sel.perm = pl.grouped ? kb.grp.perm : nullptr;
            sel.norms = norms;
            sel.rho = rho;
            sel.gam = gam;
            sel.fb_list = fb;
            sel.fb_count = (unsigned long long*)&st->fallback_count;
            knn_select_kernel<false><<<(unsigned)grid, 256, 0, s>>>(sel);
            SLK_LAUNCH_CHECK(ctx, "knn_select_kernel");
        } else {
            // entries per lane: the splits' lists, KC each, over 32 lanes
            const int per_lane = (pl.splits * pl.kc + 31) / 32;
#define SLK_RERANK(KC_, E_)                                                                   \
    knn_rerank_kernel<KC_, 0, E_><<<(unsigned)grid, 256, 0, s>>>(                             \
        X, N, D, pl.Dp, k, pl.splits, pl.Np, cand_d, cand_i, norms, rho, gam, row_ptr, col_idx, \
        dist2, fb, st)
#define SLK_RERANK_E(KC_)                                                                     \
    if (per_lane <= 4) SLK_RERANK(KC_, 4);                                                    \
    else if (per_lane <= 8) SLK_RERANK(KC_, 8);                                               \
    else SLK_RERANK(KC_, 16);
            if (pl.kc == 16) { SLK_RERANK_E(16) }
            else { SLK_RERANK_E(32) }
#undef SLK_RERANK_E
#undef SLK_RERANK
            SLK_LAUNCH_CHECK(ctx, "knn_rerank_kernel");
        }
    }
    {
        PhaseScope ps(ctx, SLK_PHASE_KNN_FALLBACK);
        // rows still open after this stage: the exact scan reads them from
        // (list, count); with bfloat16 candidates a float32 stage comes first
        const int32_t* exact_list = fb;
        const long long* exact_count = &st->fallback_count;
        if (pl.bf16) {
            // the float32 stage's input and its failures (for the exact scan)
            const int32_t* f32_in = fb;
            int32_t* fb3 = pl.two_term ? fb : fb2;   // the list that is not its input
            const long long* f32_cnt = &st->fallback_count;
            if (pl.two_term) {
                f32_in = fb2;
                f32_cnt = &st->fallback2_count;
                // (a) two-term bfloat16 tiles of the open rows on the tensor cores
                // (h . h + h . l + l . h of s = h + l, about 16 significant bits
                // of v), the rerank under their certificate; its failures, and
                // open rows beyond the stage's capacity, go on to (b)
                const bool v4 = D % 4 == 0 && pl.Dp >= 128 && (reinterpret_cast<uintptr_t>(X) & 15) == 0 &&
                                (reinterpret_cast<uintptr_t>(mu) & 15) == 0;
                int64_t pg = (pl.Np + 7) / 8;
                if (pg > (int64_t)ctx->num_sms * 64) pg = (int64_t)ctx->num_sms * 64;
                SLK_COUNT_LAUNCH(ctx, 4);
                // the operand back in the points' order where the sweep had sorted it
                __nv_bfloat16* xh = pl.grouped ? (__nv_bfloat16*)xt : nullptr;
                if (v4)
                    prep_split_kernel<4><<<(unsigned)pg, 256, 0, s>>>(X, N, D, pl.Dp, pl.Np, mu,
                                                                      &st->fallback_count, xh, kb.xl16,
                                                                      kb.norms_s, kb.rho_s, st);
                else
                    prep_split_kernel<1><<<(unsigned)pg, 256, 0, s>>>(X, N, D, pl.Dp, pl.Np, mu,
                                                                      &st->fallback_count, xh, kb.xl16,
                                                                      kb.norms_s, kb.rho_s, st);
                SLK_LAUNCH_CHECK(ctx, "prep_split_kernel");
                int64_t gg = (pl.fcap + 7) / 8;
                if (gg > (int64_t)ctx->num_sms * 16) gg = (int64_t)ctx->num_sms * 16;
                gather_split_kernel<<<(unsigned)gg, 256, 0, s>>>((const __nv_bfloat16*)xt, kb.xl16, kb.norms_s,
                                                                pl.Dp, fb, &st->fallback_count, pl.fcap,
                                                                kb.qh, kb.ql, kb.qnorm);
                SLK_LAUNCH_CHECK(ctx, "gather_split_kernel");
                // dot products of 3 Dp bfloat16 products (2^-23 accumulator
                // unit, as above), |h|, |l| within 1.004 |s| and 0.0040 |s|,
                // plus the dropped l . l term (at most 1.016 2^-16 |s_p| |s_q|)
                const double g3 = 3.0 * (double)pl.Dp * 1.1920928955078125e-07;
                const double gam_s = 1.02 * g3 / (1.0 - g3) + 1.02 * 1.52587890625e-05;
                SweepOperands op{};
                op.a_hi = kb.qh;
                op.a_lo = kb.ql;
                op.b_hi = (const __nv_bfloat16*)xt;
                op.b_lo = kb.xl16;
                op.row_norms = kb.qnorm;
                op.col_norms = kb.norms_s;
                op.rho = kb.rho_s;
                op.ids = fb;
                op.rows_dev = &st->fallback_count;
                op.a_rows = pl.fcap;
                op.b_rows = pl.Np;
                op.N = N;
                op.D = D;
                op.Dp = pl.Dp;
                SweepWork swork{};
                swork.per = swork.n_tiles = pl.n_tiles;
                swork.row_blocks = (int)(pl.fcap / 128);
                swork.units = pl.sunits;
                swork.aligned = 0;
                const SweepLists slists{kb.scand, kSweepStride};
                slk_status r = knn_sweep_launch(ctx, op, swork, k, gam_s, slists, false, nullptr, nullptr, st);
                if (r != SLK_OK) return r;
                sel.w = swork;
                sel.lists = slists;
                sel.perm = nullptr;
                sel.norms = kb.norms_s;
                sel.rho = kb.rho_s;
                sel.gam = gam_s;
                sel.fb_list = fb2;
                sel.fb_count = (unsigned long long*)&st->fallback2_count;
                sel.fb_in = fb;
                sel.count_in = &st->fallback_count;
                sel.cap = pl.fcap;
                knn_select_kernel<true><<<(unsigned)(ctx->num_sms * 4), 256, 0, s>>>(sel);
                SLK_LAUNCH_CHECK(ctx, "knn_select_kernel (two-term stage)");
            }
            // (b) float32 distance tiles of the rows still open against every
            // point, then the rerank under the float32 certificate; its
            // failures go on float32 lists of at least 2k candidates (the gap
            // between the k-th and the last decides the certificate)
            const int kcq = (2 * k <= 16) ? 16 : 32;
            // column splits chosen on the device from the count (query_splits)
            const long long qcap = (long long)cand_floats(pl);
            const int n_tiles = (int)((N + BN - 1) / BN);
            SLK_COUNT_LAUNCH(ctx, 2);
            const unsigned qgrid = (unsigned)(ctx->num_sms * 2);
#define SLK_QCAND(KC_)                                                                        \
    {                                                                                         \
        auto kern = knn_cand_query_kernel<KC_>;                                               \
        const int smem = (int)sizeof(CandSmem<KC_>);                                          \
        SLK_CUDA_TRY(ctx, cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem)); \
        kern<<<qgrid, KT, smem, s>>>(X, N, D, pl.Dp, mu, norms32, f32_in, f32_cnt, qcap,      \
                                     n_tiles, cand_d, cand_i);                                \
    }
            if (kcq == 16) SLK_QCAND(16) else SLK_QCAND(32)
#undef SLK_QCAND
            SLK_LAUNCH_CHECK(ctx, "knn_cand_query_kernel");
            const unsigned rgrid = (unsigned)(ctx->num_sms * 4);   // grid-stride over the open rows
            const double g32 = (double)pl.Dp * 5.9604644775390625e-08;
            const double gam32 = g32 / (1.0 - g32);
            if (kcq == 16)
                knn_rerank_kernel<16, 1><<<rgrid, 256, 0, s>>>(
                    X, N, D, pl.Dp, k, 0, qcap, cand_d, cand_i, norms32, nullptr, gam32, row_ptr,
                    col_idx, dist2, fb3, st, f32_in, f32_cnt, &st->fallback3_count);
            else
                knn_rerank_kernel<32, 1><<<rgrid, 256, 0, s>>>(
                    X, N, D, pl.Dp, k, 0, qcap, cand_d, cand_i, norms32, nullptr, gam32, row_ptr,
                    col_idx, dist2, fb3, st, f32_in, f32_cnt, &st->fallback3_count);
            SLK_LAUNCH_CHECK(ctx, "knn_rerank_kernel (float32 stage)");
            exact_list = fb3;
            exact_count = &st->fallback3_count;
        }
        // the batched rescan's partial lists reuse the candidate buffer
        // (its lists are read by now): cs column ranges of k entries for each
        // of the F open rows, cs chosen on the device from F
        const long long cap = (long long)cand_floats(pl);
        const int dpl = (D + 31) / 32;
        if (dpl <= 32) {
            SLK_COUNT_LAUNCH(ctx, 2);
            const unsigned grid = (unsigned)(ctx->num_sms * 2);
#define SLK_FB(R_, DPL_)                                                                     \
    knn_fallback_batch_kernel<R_, DPL_><<<grid, 256, 0, s>>>(X, N, D, k, (int)grid, exact_list, \
                                                             exact_count, cap, cand_d, cand_i)
            if (dpl <= 4) SLK_FB(16, 4);
            else if (dpl <= 8) SLK_FB(8, 8);
            else if (dpl <= 16) SLK_FB(4, 16);
            else SLK_FB(2, 32);
#undef SLK_FB
            SLK_LAUNCH_CHECK(ctx, "knn_fallback_batch_kernel");
            knn_fallback_merge_kernel<<<(unsigned)(ctx->num_sms * 2), 256, 0, s>>>(
                N, exact_rows(D), (int)grid, k, exact_list, exact_count, cap, cand_d, cand_i, col_idx,
                dist2);
            SLK_LAUNCH_CHECK(ctx, "knn_fallback_merge_kernel");
        } else if ((size_t)D * sizeof(float) <= kWideSmemMax) {
            // long rows: staged in shared memory, (row, column range) items
            SLK_COUNT_LAUNCH(ctx, 2);
            const int smem = (int)((size_t)D * sizeof(float));
            SLK_CUDA_TRY(ctx, cudaFuncSetAttribute(knn_fallback_wide_kernel,
                                                   cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
            const int grid = ctx->num_sms * 4;
            knn_fallback_wide_kernel<<<(unsigned)grid, 256, smem, s>>>(
                X, N, D, k, grid, exact_list, exact_count, cap, cand_d, cand_i);
            SLK_LAUNCH_CHECK(ctx, "knn_fallback_wide_kernel");
            knn_fallback_merge_kernel<<<(unsigned)(ctx->num_sms * 2), 256, 0, s>>>(
                N, 1, grid, k, exact_list, exact_count, cap, cand_d, cand_i, col_idx, dist2);
            SLK_LAUNCH_CHECK(ctx, "knn_fallback_merge_kernel");
        } else {
        SLK_COUNT_LAUNCH(ctx, 1);
        knn_fallback_kernel<<<(unsigned)(ctx->num_sms * 2), 256, 0, s>>>(X, N, D, k, exact_list,
                                                                         exact_count, col_idx, dist2);
        SLK_LAUNCH_CHECK(ctx, "knn_fallback_kernel");
        }
    }
    return SLK_OK;
}
