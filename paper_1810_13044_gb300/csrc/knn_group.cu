// Which column tiles a row block of the kNN sweep can leave out.
//
// The points are sorted by their nearest of 128 pivots (rows of the bfloat16
// operand, drawn from a sample by squared distance to the pivots before them)
// and inside a region by their second nearest, so that a 128-row block mostly
// lies in one part of one region.  For two
// pivots c_i, c_j let
//   f_ij(x) = (||x - c_j||^2 - ||x - c_i||^2) / (2 ||c_i - c_j||)
//           = ((|c_j|^2 - |c_i|^2) / 2 - x . (c_j - c_i)) / ||c_i - c_j||,
// the signed distance of x from the border between them, positive on c_i's
// side.  It is linear with unit slope, so ||x - y|| >= f_ij(x) + f_ji(y) for any
// x and y.  With i the pivot of row block b, j that of column block t:
//   every x in b, y in t:  ||x - y|| >= f_ij(x) + lo_t(i),  lo_t(i) = min_y f_ji(y).
// A first sweep over the 8 tiles around each block's own columns leaves every
// row with a threshold T below which a column's squared operand distance must
// lie to matter (knn_cert.cuh), so tile t can be left out for block b when
//   min_x (f_ij(x) - sqrt(T_x)) + lo_t(i) >= 0
// for both column blocks of the tile; f is lowered by the rounding of its dot
// products.  The second sweep runs over the remaining tiles and the rows'
// lists go on from the first one's, so the graph does not depend on the
// pivots.
// Candidates of the graph (both sweeps and the passes between them), and the
// preparation with the sort, in ms, against one sweep over every tile:
//   70000 x 784, 10 clusters, k = 5       1.18 + 0.52    5.50 + 0.19
//   60001 x 50, 30 clusters, k = 8        0.44 + 0.21    2.26 + 0.05
//   200000 x 128, 100 manifolds, k = 10   5.59 + 0.40   17.64 + 0.17
//   1e6 x 128, 100 manifolds, k = 10      86.7 + 1.24   309.3 + 0.70
//   70000 x 784, one cluster, k = 5       5.69 + 0.52    5.47 + 0.18
//   1e6 x 128, one cluster, k = 10       300.2 + 1.91   291.0 + 1.35
#include <cuda_bf16.h>
#include <math.h>
#include <stdint.h>

#include "knn_group.cuh"

namespace {

constexpr int kDraw = 32;        // pivots drawn per round
constexpr int kRounds = kPivots / kDraw;

// ------------------------------------------------------------------- pivots

__device__ __forceinline__ int64_t sample_row(int s, int S, int64_t N) {
    return (int64_t)s * N / S;
}

// Every step-th feature of the sampled points (any of them do for the draw).
__global__ void group_sample_kernel(const float* __restrict__ X, int64_t N, int D, int S, int dims, int step,
                                    float* __restrict__ xs, float* __restrict__ mind2) {
    const int s = blockIdx.x;
    const float* x = X + sample_row(s, S, N) * D;
    for (int j = threadIdx.x; j < dims; j += blockDim.x) xs[s * kGrpDims + j] = x[(int64_t)j * step];
    if (threadIdx.x == 0) mind2[s] = __int_as_float(0x7f800000);
}

// One round: distances to the last kDraw pivots, then (last block) kDraw new
// ones at equal steps of the running sum of mind2, i.e. drawn in proportion to
// it.  Round 0 only draws, at equal steps of the sample.
__global__ void __launch_bounds__(256)
group_draw_kernel(const float* __restrict__ xs, int S, int dims, int round, float* __restrict__ mind2,
                  int32_t* __restrict__ pick, unsigned* __restrict__ done) {
    __shared__ float pre[kGrpSample];
    __shared__ float wt[8];
    __shared__ int last;
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    if (round > 0) {
        for (int s = blockIdx.x * 8 + w; s < S; s += gridDim.x * 8) {
            float x[kGrpDims / 32];
#pragma unroll
            for (int j = 0; j < kGrpDims / 32; ++j)
                x[j] = lane + 32 * j < dims ? xs[(int64_t)s * kGrpDims + lane + 32 * j] : 0.f;
            float best = mind2[s];
#pragma unroll 4
            for (int c = 0; c < kDraw; ++c) {
                const float* y = xs + (int64_t)pick[(round - 1) * kDraw + c] * kGrpDims;
                float d = 0.f;
#pragma unroll
                for (int j = 0; j < kGrpDims / 32; ++j) {
                    const float df = lane + 32 * j < dims ? x[j] - y[lane + 32 * j] : 0.f;
                    d = fmaf(df, df, d);
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
                best = fminf(best, d);
            }
            if (lane == 0) mind2[s] = best;
        }
        __threadfence();
        __syncthreads();
    }
    if (t == 0) last = atomicAdd(done, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    if (t == 0) *done = 0u;
    if (round == 0) {
        if (t < kDraw) pick[t] = (int)((int64_t)t * S / kDraw);
        return;
    }
    // running sums: thread t holds samples 16 t .. 16 t + 15
    constexpr int PER = kGrpSample / 256;
    float v[PER], run = 0.f;
#pragma unroll
    for (int i = 0; i < PER; ++i) v[i] = t * PER + i < S ? fminf(__ldcg(mind2 + t * PER + i), 1e30f) : 0.f;
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        run += v[i];
        v[i] = run;
    }
    float incl = run;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const float y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) wt[w] = incl;
    __syncthreads();
    float off = incl - run, total = 0.f;
    for (int i = 0; i < 8; ++i) {
        if (i < w) off += wt[i];
        total += wt[i];
    }
#pragma unroll
    for (int i = 0; i < PER; ++i) pre[t * PER + i] = v[i] + off;
    __syncthreads();
    if (t < kDraw) {
        const float r = ((float)t + 0.5f) / kDraw * total;
        int lo = 0, hi = S - 1;   // first sample whose running sum reaches r
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (pre[mid] >= r) hi = mid; else lo = mid + 1;
        }
        pick[round * kDraw + t] = lo;
    }
}

// Pivot j as the bfloat16 operand row of its point, and its squared norm.
__global__ void __launch_bounds__(128)
group_pivot_kernel(const float* __restrict__ X, int64_t N, int D, int Dp, int S, const float* __restrict__ mu,
                   const int32_t* __restrict__ pick, __nv_bfloat16* __restrict__ pv, float* __restrict__ pn2) {
    __shared__ float part[4];
    const int j = blockIdx.x, t = threadIdx.x;
    const float* x = X + sample_row(pick[j], S, N) * D;
    float n2 = 0.f;
    for (int d = t; d < Dp; d += 128) {
        const __nv_bfloat16 b = __float2bfloat16_rn(d < D ? x[d] - mu[d] : 0.f);
        pv[(int64_t)j * Dp + d] = b;
        const float v = __bfloat162float(b);
        n2 = fmaf(v, v, n2);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) n2 += __shfl_xor_sync(0xffffffffu, n2, o);
    if ((t & 31) == 0) part[t >> 5] = n2;
    __syncthreads();
    if (t == 0) pn2[j] = part[0] + part[1] + part[2] + part[3];
}

__global__ void __launch_bounds__(256)
group_pdist_kernel(const __nv_bfloat16* __restrict__ pv, int Dp, float* __restrict__ pdist) {
    const int i = blockIdx.x, lane = threadIdx.x & 31;
    const __nv_bfloat162* a = reinterpret_cast<const __nv_bfloat162*>(pv + (int64_t)i * Dp);
    for (int j = threadIdx.x >> 5; j < kPivots; j += 8) {
        const __nv_bfloat162* b = reinterpret_cast<const __nv_bfloat162*>(pv + (int64_t)j * Dp);
        float d = 0.f;
        for (int e = lane; e < Dp / 2; e += 32) {
            const float2 u = __bfloat1622float2(a[e]), v = __bfloat1622float2(b[e]);
            const float x = u.x - v.x, y = u.y - v.y;
            d = fmaf(x, x, d);
            d = fmaf(y, y, d);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
        if (lane == 0) pdist[i * kPivots + j] = sqrtf(d);
    }
}

// Order of the pivots: each followed by the nearest one left, so that a block
// that holds the end of one region and the start of the next rarely joins two
// far apart.
__global__ void __launch_bounds__(256)
group_chain_kernel(const float* __restrict__ pdist, int32_t* __restrict__ chain) {
    extern __shared__ float sd[];   // [kPivots][kPivots]
    for (int i = threadIdx.x; i < kPivots * kPivots; i += 256) sd[i] = pdist[i];
    __syncthreads();
    const int lane = threadIdx.x;
    if (lane >= 32) return;
    bool used[kPivots / 32] = {};
    int cur = 0;
    if (lane == 0) used[0] = true;
    for (int n = 0; n < kPivots; ++n) {
        if (lane == 0) chain[n] = cur;
        unsigned best = 0xffffffffu;
        int at = 0;
#pragma unroll
        for (int q = 0; q < kPivots / 32; ++q) {
            const unsigned v = used[q] ? 0xffffffffu : __float_as_uint(sd[cur * kPivots + q * 32 + lane]);
            if (v < best) { best = v; at = q * 32 + lane; }
        }
        const unsigned m = __reduce_min_sync(0xffffffffu, best);
        const unsigned who = __ballot_sync(0xffffffffu, best == m);
        cur = __shfl_sync(0xffffffffu, at, __ffs(who) - 1);
#pragma unroll
        for (int q = 0; q < kPivots / 32; ++q)
            if (cur == q * 32 + lane) used[q] = true;
    }
}

// ------------------------------------------------- products with the pivots

constexpr int GK = 64;             // features per slice
constexpr int GS = GK + 8;         // shared-memory row stride (bf16): conflict-free ldmatrix

__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], const __nv_bfloat16* p) {
    const uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a));
}
__device__ __forceinline__ void mma16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, "
        "{%8, %9}, {%0, %1, %2, %3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

struct DotArgs {
    const float* X;               // first pass: features, mu
    const float* mu;
    const __nv_bfloat16* xt;      // bounds: the sorted operand
    int64_t N;
    int D, Dp, vec;
    const __nv_bfloat16* pv;
    const float* pn2;
    const float* pdist;
    const int32_t* chain;
    int32_t* lab;
    int32_t* lab2;
    // bounds
    const int32_t* perm;
    const float* thr;
    float* sl;
    float* lo_t;
    int32_t* rep;
    int64_t n_blocks;
};

// 128 rows against the 128 pivots (places of the chain): 8 warps of 16 rows,
// bf16 products on mma.sync (128 columns: one fragment tile per warp; a small
// part of the graph's time, bound by reading the rows).  BOUNDS false: the
// nearest pivot of each row.  BOUNDS true: the block's slack and depth.
template <bool BOUNDS>
__global__ void __launch_bounds__(256)
group_dots_kernel(const DotArgs a) {
    __shared__ __align__(16) __nv_bfloat16 As[128][GS], Bs[kPivots][GS];
    __shared__ float s_n2[kPivots], s_gi[128], s_x2[128];
    __shared__ float s_lo[8][kPivots], s_sl[8][kPivots];
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    const int64_t row0 = (int64_t)blockIdx.x * 128;
    if (t < kPivots) s_n2[t] = a.pn2[a.chain[t]];
    float acc[16][4];
#pragma unroll
    for (int n = 0; n < 16; ++n)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[n][q] = 0.f;
    float x2 = 0.f;   // bounds: part of the squared norm of row t / 2
    for (int k0 = 0; k0 < a.Dp; k0 += GK) {
        // 8 lanes x 16 bytes per row of the slice
        for (int i = t; i < kPivots * 8; i += 256) {
            const int r = i >> 3, c = (i & 7) * 8;
            *reinterpret_cast<uint4*>(&Bs[r][c]) =
                __ldg(reinterpret_cast<const uint4*>(a.pv + (int64_t)a.chain[r] * a.Dp + k0 + c));
        }
        for (int i = t; i < 128 * 8; i += 256) {
            const int r = i >> 3, c = (i & 7) * 8;
            uint4 v = make_uint4(0u, 0u, 0u, 0u);
            if (row0 + r < a.N) {
                if (BOUNDS) {
                    v = __ldg(reinterpret_cast<const uint4*>(a.xt + (row0 + r) * a.Dp + k0 + c));
                } else {
                    float f[8];
                    const float* x = a.X + (row0 + r) * a.D;
                    if (a.vec && k0 + c + 8 <= a.D) {
                        const float4 p = __ldg(reinterpret_cast<const float4*>(x + k0 + c));
                        const float4 q = __ldg(reinterpret_cast<const float4*>(x + k0 + c + 4));
                        f[0] = p.x; f[1] = p.y; f[2] = p.z; f[3] = p.w;
                        f[4] = q.x; f[5] = q.y; f[6] = q.z; f[7] = q.w;
#pragma unroll
                        for (int e = 0; e < 8; ++e) f[e] -= __ldg(a.mu + k0 + c + e);
                    } else {
#pragma unroll
                        for (int e = 0; e < 8; ++e)
                            f[e] = k0 + c + e < a.D ? x[k0 + c + e] - __ldg(a.mu + k0 + c + e) : 0.f;
                    }
                    __nv_bfloat162 b[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) b[e] = __floats2bfloat162_rn(f[2 * e], f[2 * e + 1]);
                    v = *reinterpret_cast<const uint4*>(b);
                }
            }
            *reinterpret_cast<uint4*>(&As[r][c]) = v;
        }
        __syncthreads();
        if (BOUNDS) {
            const __nv_bfloat162* x = reinterpret_cast<const __nv_bfloat162*>(&As[t >> 1][(t & 1) * 32]);
#pragma unroll
            for (int e = 0; e < 16; ++e) {
                const float2 v = __bfloat1622float2(x[e]);
                x2 = fmaf(v.x, v.x, x2);
                x2 = fmaf(v.y, v.y, x2);
            }
        }
#pragma unroll
        for (int kk = 0; kk < GK; kk += 16) {
            uint32_t af[4];
            ldsm4(af, &As[16 * w + (lane & 15)][kk + (lane >> 4) * 8]);
#pragma unroll
            for (int n = 0; n < 16; n += 2) {
                uint32_t bf[4];   // two 8-column tiles: rows of Bs are columns of B
                ldsm4(bf, &Bs[8 * n + (lane & 7) + ((lane >> 4) << 3)][kk + ((lane >> 3) & 1) * 8]);
                mma16816(acc[n], af, bf[0], bf[1]);
                mma16816(acc[n + 1], af, bf[2], bf[3]);
            }
        }
        __syncthreads();
    }
    // acc[n][q]: row 16 w + lane / 4 + 8 (q / 2), column 8 n + 2 (lane % 4) + q % 2
    const int ra = 16 * w + (lane >> 2), rb = ra + 8, c0 = 2 * (lane & 3);
    if (!BOUNDS) {
        // nearest (ia, ib) and second nearest (ja, jb) pivot of the two rows
        const float inf = __int_as_float(0x7f800000);
        float ba = inf, bb = inf, ca = inf, cb = inf;
        int ia = 0, ib = 0, ja = 0, jb = 0;
        auto take = [](float v, int c, float& b1, int& i1, float& b2, int& i2) {
            if (v < b1) { b2 = b1; i2 = i1; b1 = v; i1 = c; }
            else if (v < b2) { b2 = v; i2 = c; }
        };
#pragma unroll
        for (int n = 0; n < 16; ++n) {
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const int c = 8 * n + c0 + q;
                take(0.5f * s_n2[c] - acc[n][q], c, ba, ia, ca, ja);
                take(0.5f * s_n2[c] - acc[n][q + 2], c, bb, ib, cb, jb);
            }
        }
#pragma unroll
        for (int o = 1; o < 4; o <<= 1) {
            const float oa = __shfl_xor_sync(0xffffffffu, ba, o), ob = __shfl_xor_sync(0xffffffffu, bb, o);
            const float pa = __shfl_xor_sync(0xffffffffu, ca, o), pb = __shfl_xor_sync(0xffffffffu, cb, o);
            const int xa = __shfl_xor_sync(0xffffffffu, ia, o), xb = __shfl_xor_sync(0xffffffffu, ib, o);
            const int ya = __shfl_xor_sync(0xffffffffu, ja, o), yb = __shfl_xor_sync(0xffffffffu, jb, o);
            take(oa, xa, ba, ia, ca, ja);
            take(pa, ya, ba, ia, ca, ja);
            take(ob, xb, bb, ib, cb, jb);
            take(pb, yb, bb, ib, cb, jb);
        }
        if ((lane & 3) == 0) {
            if (row0 + ra < a.N) { a.lab[row0 + ra] = ia; a.lab2[row0 + ra] = ja; }
            if (row0 + rb < a.N) { a.lab[row0 + rb] = ib; a.lab2[row0 + rb] = jb; }
        }
        return;
    }
    const float inf = __int_as_float(0x7f800000);
    // the block's pivot: that of its middle row
    const int64_t mid = row0 + 64 < a.N ? row0 + 64 : a.N - 1;
    const int i = a.lab[a.perm[mid]];
    if (threadIdx.x == 0) a.rep[blockIdx.x] = i;
    const float xh = x2 + __shfl_xor_sync(0xffffffffu, x2, 1);
    if ((t & 1) == 0) s_x2[t >> 1] = xh;
#pragma unroll
    for (int n = 0; n < 16; ++n)
#pragma unroll
        for (int q = 0; q < 2; ++q)
            if (8 * n + c0 + q == i) {
                s_gi[ra] = acc[n][q];
                s_gi[rb] = acc[n][q + 2];
            }
    __syncthreads();
    const float ga = s_gi[ra], gb = s_gi[rb];
    const float na = sqrtf(s_x2[ra]) * 1.001f, nb = sqrtf(s_x2[rb]) * 1.001f;
    const bool la = row0 + ra < a.N, lb = row0 + rb < a.N;
    // a row whose list gave up (-inf) is left open whatever the tiles
    const float Ta = la ? a.thr[row0 + ra] : -inf, Tb = lb ? a.thr[row0 + rb] : -inf;
    const float sa = Ta > 0.f ? sqrtf(Ta) * 1.00001f : 0.f, sb = Tb > 0.f ? sqrtf(Tb) * 1.00001f : 0.f;
    // rounding of the dot products and norms, relative to the norms' products
    const float eps = (float)(a.Dp + 32) * 2.4e-7f;
    const float ni = s_n2[i], nri = sqrtf(ni);
#pragma unroll
    for (int n = 0; n < 16; ++n) {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int c = 8 * n + c0 + q;
            const float nj = s_n2[c], nrm = fmaxf(nri, sqrtf(nj));
            const float dist = a.pdist[a.chain[i] * kPivots + a.chain[c]];
            const bool border = c != i && dist > 1e-3f * nrm && dist > 1e-18f;
            const float inv = 1.f / dist;
            auto depth = [&](float g, float gi, float nx) {
                const float f = (0.5f * (nj - ni) - (g - gi)) * inv;
                return f - 2e-5f * fabsf(f) - eps * (nx + nrm) * nrm * inv;
            };
            float fa = la ? depth(acc[n][q], ga, na) : inf, fb = lb ? depth(acc[n][q + 2], gb, nb) : inf;
            if (!border) { fa = la ? -inf : inf; fb = lb ? -inf : inf; }
            float lo = fminf(fa, fb);
            float sl = fminf(Ta > -inf ? fa - sa : inf, Tb > -inf ? fb - sb : inf);
#pragma unroll
            for (int o = 4; o < 32; o <<= 1) {
                lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
                sl = fminf(sl, __shfl_xor_sync(0xffffffffu, sl, o));
            }
            if (lane < 4) {
                s_lo[w][c] = lo;
                s_sl[w][c] = sl;
            }
        }
    }
    __syncthreads();
    if (t < kPivots) {
        float lo = s_lo[0][t], sl = s_sl[0][t];
#pragma unroll
        for (int q = 1; q < 8; ++q) {
            lo = fminf(lo, s_lo[q][t]);
            sl = fminf(sl, s_sl[q][t]);
        }
        a.sl[(int64_t)blockIdx.x * kPivots + t] = sl;
        a.lo_t[(int64_t)t * a.n_blocks + blockIdx.x] = lo;
    }
}

// -------------------------------------------------------------------- tiles

// One block per row block: the tiles it must sweep beside the first pass's
// window.  FILL false counts them, FILL true lists them from start[rb].
template <bool FILL>
__global__ void __launch_bounds__(256)
group_tiles_kernel(const float* __restrict__ sl, const float* __restrict__ lo_t,
                   const int32_t* __restrict__ rep, SweepWork first, int32_t* __restrict__ cnt,
                   const int64_t* __restrict__ start, uint16_t* __restrict__ tiles) {
    __shared__ float s_sl[kPivots];
    __shared__ int s_n, s_w[8];
    const int t = threadIdx.x, lane = t & 31, w = t >> 5, rb = blockIdx.x;
    const int64_t nb = first.row_blocks;
    if (t < kPivots) s_sl[t] = sl[(int64_t)rb * kPivots + t];
    if (t == 0) s_n = 0;
    __syncthreads();
    const int i = rep[rb];
    const float* lo = lo_t + (int64_t)i * nb;
    const int w0 = sweep_tile0(first, rb), w1 = w0 + first.per;
    uint16_t* out = FILL ? tiles + start[rb] : nullptr;
    // FILL: the region's own tiles first (their columns lower the thresholds
    // most), then the others
    for (int pass = 0; pass < (FILL ? 2 : 1); ++pass) {
        for (int b0 = 0; b0 < first.n_tiles; b0 += 256) {
            const int tile = b0 + t;
            bool keep = false;
            if (tile < first.n_tiles && (tile < w0 || tile >= w1)) {
                const int g0 = 2 * tile, g1 = g0 + 1;   // its two column blocks
                const int r0 = rep[g0], r1 = g1 < nb ? rep[g1] : r0;
                keep = !(s_sl[r0] + lo[g0] >= 0.f);
                if (g1 < nb && !keep) keep = !(s_sl[r1] + lo[g1] >= 0.f);
                if (FILL) keep = keep && (r0 == i || r1 == i) == (pass == 0);
            }
            const unsigned m = __ballot_sync(0xffffffffu, keep);
            if (lane == 0) s_w[w] = __popc(m);
            __syncthreads();
            int at = s_n, all = 0;
            for (int q = 0; q < 8; ++q) {
                if (q < w) at += s_w[q];
                all += s_w[q];
            }
            if (FILL && keep) out[at + __popc(m & ((1u << lane) - 1u))] = (uint16_t)tile;
            __syncthreads();
            if (t == 0) s_n += all;
            __syncthreads();
        }
    }
    if (!FILL && t == 0) cnt[rb] = s_n;
}

// start[] from cnt[] and the largest count (one block).
__global__ void __launch_bounds__(1024)
group_scan_kernel(const int32_t* __restrict__ cnt, int n, int64_t* __restrict__ start,
                  int32_t* __restrict__ max_cnt) {
    __shared__ int64_t wt[32];
    __shared__ int s_max;
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    const int per = (n + 1023) / 1024;
    if (t == 0) s_max = 0;
    __syncthreads();
    int64_t run = 0;
    int mx = 0;
    for (int i = t * per; i < n && i < (t + 1) * per; ++i) {
        run += cnt[i];
        mx = max(mx, cnt[i]);
    }
    atomicMax(&s_max, mx);
    int64_t incl = run;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int64_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) wt[w] = incl;
    __syncthreads();
    int64_t off = incl - run;
    for (int i = 0; i < w; ++i) off += wt[i];
    for (int i = t * per; i < n && i < (t + 1) * per; ++i) {
        start[i] = off;
        off += cnt[i];
    }
    if (t == 1023) start[n] = off;
    if (t == 0) *max_cnt = s_max;
}

// dst[i] = src[perm[i]]; and first[i] = perm[second[i]] (in place of second).
__global__ void group_gather_kernel(const int32_t* __restrict__ src, const int32_t* __restrict__ perm,
                                    int64_t N, int32_t* __restrict__ dst) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x)
        dst[i] = src[perm[i]];
}
__global__ void group_compose_kernel(const int32_t* __restrict__ perm, int64_t N, int32_t* __restrict__ second) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x)
        second[i] = perm[second[i]];
}

// enough to see clusters of a thousandth of the points
int sample_size(int64_t N) { return (int)(N < kGrpSample ? N : N < 200000 ? kGrpSample / 2 : kGrpSample); }

}  // namespace

size_t group_carve(WsCarver& wc, GroupBufs& b, int64_t N, int64_t Np, int Dp, int n_tiles) {
    const size_t blocks = (size_t)(Np / 128), sort = (size_t)((N + 1023) / 1024);
    b.xs = wc.take<float>((size_t)kGrpSample * kGrpDims);
    b.mind2 = wc.take<float>(kGrpSample);
    b.pick = wc.take<int32_t>(kPivots);
    b.done = wc.take<unsigned>(1);
    b.pv = wc.take<__nv_bfloat16>((size_t)kPivots * Dp);
    b.pn2 = wc.take<float>(kPivots);
    b.pdist = wc.take<float>(kPivots * kPivots);
    b.chain = wc.take<int32_t>(kPivots);
    b.lab = wc.take<int32_t>(N);
    b.lab2 = wc.take<int32_t>(N);
    b.perm2 = wc.take<int32_t>(N);
    b.counts = wc.take<int32_t>(sort * kPivots);
    b.base = wc.take<int64_t>(sort * kPivots);
    b.off = wc.take<int64_t>(kPivots + 1);
    b.perm = wc.take<int32_t>(N);
    b.thr = wc.take<float>(Np);
    b.kth = wc.take<float>(Np);
    b.sl = wc.take<float>(blocks * kPivots);
    b.lo_t = wc.take<float>(blocks * kPivots);
    b.rep = wc.take<int32_t>(blocks);
    b.cnt = wc.take<int32_t>(blocks);
    b.start = wc.take<int64_t>(blocks + 1);
    b.max_cnt = wc.take<int32_t>(1);
    b.tiles = wc.take<uint16_t>(blocks * (size_t)n_tiles);
    return wc.off;
}

slk_status group_order_launch(slk_ctx* ctx, const GroupBufs& b, const float* X, int64_t N, int D, int Dp,
                              const float* mu) {
    cudaStream_t s = ctx->stream;
    const int S = sample_size(N);
    const int step = (D + kGrpDims - 1) / kGrpDims, dims = D / step;
    SLK_COUNT_LAUNCH(ctx, 5 + kRounds);
    SLK_CUDA_TRY(ctx, cudaMemsetAsync(b.done, 0, sizeof(unsigned), s));
    group_sample_kernel<<<S, 128, 0, s>>>(X, N, D, S, dims, step, b.xs, b.mind2);
    for (int r = 0; r < kRounds; ++r)
        group_draw_kernel<<<r ? (unsigned)((S + 7) / 8) : 1u, 256, 0, s>>>(b.xs, S, dims, r, b.mind2, b.pick,
                                                                             b.done);
    group_pivot_kernel<<<kPivots, 128, 0, s>>>(X, N, D, Dp, S, mu, b.pick, b.pv, b.pn2);
    group_pdist_kernel<<<kPivots, 256, 0, s>>>(b.pv, Dp, b.pdist);
    const int chain_smem = (int)sizeof(float) * kPivots * kPivots;
    SLK_CUDA_TRY(ctx, cudaFuncSetAttribute(group_chain_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           chain_smem));
    group_chain_kernel<<<1, 256, chain_smem, s>>>(b.pdist, b.chain);
    DotArgs a{};
    a.X = X;
    a.mu = mu;
    a.N = N;
    a.D = D;
    a.Dp = Dp;
    a.vec = D % 4 == 0 && (reinterpret_cast<uintptr_t>(X) & 15) == 0;
    a.pv = b.pv;
    a.pn2 = b.pn2;
    a.chain = b.chain;
    a.lab = b.lab;
    a.lab2 = b.lab2;
    group_dots_kernel<false><<<(unsigned)((N + 127) / 128), 256, 0, s>>>(a);
    SLK_LAUNCH_CHECK(ctx, "group_dots_kernel");
    // by second nearest, then (stable) by nearest pivot
    slk_status r = label_sort_launch(ctx, b.lab2, N, kPivots, b.counts, b.base, b.off, b.perm2);
    if (r != SLK_OK) return r;
    SLK_COUNT_LAUNCH(ctx, 2);
    const unsigned gg = (unsigned)((N + 255) / 256 < ctx->num_sms * 16 ? (N + 255) / 256 : ctx->num_sms * 16);
    group_gather_kernel<<<gg, 256, 0, s>>>(b.lab, b.perm2, N, b.lab2);
    r = label_sort_launch(ctx, b.lab2, N, kPivots, b.counts, b.base, b.off, b.perm);
    if (r != SLK_OK) return r;
    group_compose_kernel<<<gg, 256, 0, s>>>(b.perm2, N, b.perm);
    SLK_LAUNCH_CHECK(ctx, "group_compose_kernel");
    return SLK_OK;
}

slk_status group_tiles_launch(slk_ctx* ctx, const GroupBufs& b, const __nv_bfloat16* xt, int64_t N,
                              int64_t Np, int Dp, const SweepWork& first) {
    cudaStream_t s = ctx->stream;
    DotArgs a{};
    a.xt = xt;
    a.N = N;
    a.Dp = Dp;
    a.pv = b.pv;
    a.pn2 = b.pn2;
    a.pdist = b.pdist;
    a.chain = b.chain;
    a.lab = b.lab;
    a.perm = b.perm;
    a.thr = b.thr;
    a.sl = b.sl;
    a.lo_t = b.lo_t;
    a.rep = b.rep;
    a.n_blocks = Np / 128;
    SLK_COUNT_LAUNCH(ctx, 4);
    const unsigned nb = (unsigned)(Np / 128);
    group_dots_kernel<true><<<nb, 256, 0, s>>>(a);
    group_tiles_kernel<false><<<nb, 256, 0, s>>>(b.sl, b.lo_t, b.rep, first, b.cnt, b.start, b.tiles);
    group_scan_kernel<<<1, 1024, 0, s>>>(b.cnt, (int)nb, b.start, b.max_cnt);
    group_tiles_kernel<true><<<nb, 256, 0, s>>>(b.sl, b.lo_t, b.rep, first, b.cnt, b.start, b.tiles);
    SLK_LAUNCH_CHECK(ctx, "group_tiles_kernel");
    return SLK_OK;
}
