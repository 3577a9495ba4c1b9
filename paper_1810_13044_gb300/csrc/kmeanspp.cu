// K-means++ seeding on the GPU (the initial seeds of Section 4.2, which
// cites Arthur & Vassilvitskii 2007 for them), with the random draws made
// by the caller: seed 0 is the point `first`; seed i is the first point p
// whose running sum D(x_0)^2 + ... + D(x_p)^2 exceeds u_i * sum_q D(x_q)^2,
// D(x)^2 the squared distance to the closest seed chosen so far (the last
// point if no running sum does; point floor(u_i N) if every D^2 is 0).
//
// One launch per seed (kpp_step_kernel):
//   update  the distance to the new seed c, min into closest[p].  The float64
//           distance (exact float64 differences) is what bounds a plain pass
//           -- GB300 runs float64 at 1/64 of the float32 rate: 1.31 ms for
//           1e6 x 128, against 0.08 ms for reading X -- so a point gets one
//           only if it can lower closest[p]:
//             triangle inequality: with s the closest seed so far,
//               d(c, s) >= 2 d(p, s) gives d(p, c) >= d(p, s); neither X nor
//               float64 is touched (8 bytes a point);
//             float32 distance: its lower bound reaches closest[p].
//           Both bounds are inflated by the rounding of their float32 sums,
//           so closest[] holds the same bits as a pass over every point.
//   select  the last block to finish: prefix sums over 256-point tiles (each
//           tile's sum is kept, and recomputed only when one of its points
//           changed), the tile that holds u_i * total, the point inside it,
//           then the float32 bounds d(c, s)^2 of the chosen point c against
//           every earlier seed s for the next update.
// 99 seeds of 1e6 x 128 (100 clusters): 11.1 ms; two launches a seed with a
// float64 pass over every point and a one-block selection took 174.7 ms.
#include <math.h>
#include <stdint.h>

#include "slk_internal.cuh"

namespace {

constexpr int kTile = 256;           // points per tile = threads per block
// Seeds whose mutual distances are bounded: the last block computes them alone,
// at most 4096 rows a seed.  Against a float64 pass a seed, in ms: 20000 x 128,
// L = 1000: 130.7, now 29.9; 5000 x 784, L = 3000: 416, 349; 20000 x 32, L = 6000:
// 779, 482.
constexpr int kMaxBoundSeeds = 4096;
constexpr float kTiny = 1e-30f, kHuge = 1e38f;   // float32 sums outside are not trusted

struct KppArgs {
    const float* X;
    int64_t N;
    int D;
    int n_tiles;
    const double* u;        // [L - 1]
    int32_t* seeds;
    double* closest;        // [N] D(x)^2
    float* closest_up;      // [N] the same rounded up
    int32_t* own;           // [N] position of the closest seed (the first of equals)
    double* tile_sum;       // [n_tiles]
    float* dcc;             // [L] lower bound of ||new seed - seed j||^2 / 4 (0: none)
    unsigned* done;         // blocks finished
    float shrink;           // 1 - relative error of a float32 squared distance (0: bounds off)
};

// Squared distances of U points (rows xs[u]) to c by the G lanes of a
// subgroup, lane sub of it: the float32 screening sums, in any order.
template <bool VEC4, int G, int U>
__device__ __forceinline__ void screen(const float* (&xs)[U], const float* __restrict__ c, int D,
                                       int sub, float (&out)[U]) {
#pragma unroll
    for (int q = 0; q < U; ++q) out[q] = 0.f;
    if (VEC4) {
        const float4* c4 = reinterpret_cast<const float4*>(c);
        for (int j = sub; j < (D >> 2); j += G) {
            const float4 b = __ldg(c4 + j);
#pragma unroll
            for (int q = 0; q < U; ++q) {
                const float4 a = __ldg(reinterpret_cast<const float4*>(xs[q]) + j);
                const float d0 = a.x - b.x, d1 = a.y - b.y, d2 = a.z - b.z, d3 = a.w - b.w;
                out[q] = fmaf(d0, d0, out[q]);
                out[q] = fmaf(d1, d1, out[q]);
                out[q] = fmaf(d2, d2, out[q]);
                out[q] = fmaf(d3, d3, out[q]);
            }
        }
    } else {
        for (int j = sub; j < D; j += G) {
            const float b = __ldg(c + j);
#pragma unroll
            for (int q = 0; q < U; ++q) {
                const float d = __ldg(xs[q] + j) - b;
                out[q] = fmaf(d, d, out[q]);
            }
        }
    }
#pragma unroll
    for (int q = 0; q < U; ++q)
#pragma unroll
        for (int o = G / 2; o > 0; o >>= 1) out[q] += __shfl_xor_sync(0xffffffffu, out[q], o);
}

// The float64 distance by the same lanes.  With G lanes >= the row's words
// the lanes of a 32-lane butterfly beyond them would add zeros, so the bits
// do not depend on G.
template <bool VEC4, int G>
__device__ __forceinline__ double exact64(const float* __restrict__ x, const float* __restrict__ c,
                                          int D, int sub) {
    double acc = 0.0;
    if (VEC4) {
        const float4* x4 = reinterpret_cast<const float4*>(x);
        const float4* c4 = reinterpret_cast<const float4*>(c);
        for (int j = sub; j < (D >> 2); j += G) {
            const float4 a = __ldg(x4 + j), b = __ldg(c4 + j);
            const double d0 = (double)a.x - (double)b.x, d1 = (double)a.y - (double)b.y;
            const double d2 = (double)a.z - (double)b.z, d3 = (double)a.w - (double)b.w;
            acc = fma(d0, d0, acc);
            acc = fma(d1, d1, acc);
            acc = fma(d2, d2, acc);
            acc = fma(d3, d3, acc);
        }
    } else {
        for (int j = sub; j < D; j += G) {
            const double d = (double)__ldg(x + j) - (double)__ldg(c + j);
            acc = fma(d, d, acc);
        }
    }
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    return acc;
}

// Inclusive prefix sums of one value per thread over the block (256 threads).
__device__ __forceinline__ double block_scan(double v, double* warp_tot) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const double y = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += y;
    }
    if (lane == 31) warp_tot[w] = v;
    __syncthreads();
    double off = 0.0;
    for (int i = 0; i < w; ++i) off += warp_tot[i];
    __syncthreads();
    return off + v;
}

// Seed i from closest[] (one block; every other block's writes are visible).
__device__ void kpp_select(const KppArgs& a, int i) {
    __shared__ double wt[8];
    __shared__ double s_off, s_total;
    __shared__ int s_pos, s_last;
    const int t = threadIdx.x;
    const int per = (a.n_tiles + kTile - 1) / kTile;   // tiles of one thread's strip
    const int64_t q0 = (int64_t)t * per;
    const int b = (int)min((int64_t)a.n_tiles, q0), e = (int)min((int64_t)a.n_tiles, q0 + per);
    double strip = 0.0;
    for (int j = b; j < e; ++j) strip += __ldcg(a.tile_sum + j);
    const double incl = block_scan(strip, wt);
    double excl = __shfl_up_sync(0xffffffffu, incl, 1);
    if ((t & 31) == 0) {
        excl = 0.0;
        for (int w = 0; w < (t >> 5); ++w) excl += wt[w];
    }
    if (t == kTile - 1) s_total = incl;
    if (t == 0) { s_pos = kTile; s_last = 0; }
    __syncthreads();
    const double total = s_total, r_u = a.u[i - 1], r = r_u * total;
    if (!(total > 0.0)) {
        const int64_t pick = (int64_t)(r_u * (double)a.N);
        if (t == 0) a.seeds[i] = (int32_t)(pick < a.N - 1 ? pick : a.N - 1);
        return;
    }
    // only strips that hold something: each lane of the scan adds in an order of
    // its own, so a prefix may round up across empty strips (those past n_tiles
    // among them), or the last one that counts may round below r
    if (strip > 0.0) {
        if (incl > r) atomicMin(&s_pos, t);
        atomicMax(&s_last, t);
    }
    __syncthreads();
    const int owner = s_pos < kTile ? s_pos : r < total ? s_last : kTile;
    if (owner >= kTile) {   // no running sum exceeds r
        if (t == 0) a.seeds[i] = (int32_t)(a.N - 1);
        return;
    }
    __syncthreads();
    if (t == owner) {
        // the strip's first tile whose end exceeds r; rounding can leave none
        // (the strip's sum was added in another order): its last non-empty one
        double run = excl, off = excl;
        int tile = -1, last = b;
        for (int j = b; j < e && tile < 0; ++j) {
            const double s = __ldcg(a.tile_sum + j);
            if (s > 0.0) {
                last = j;
                off = run;
                if (run + s > r) tile = j;
            }
            run += s;
        }
        s_off = off;
        s_pos = tile >= 0 ? tile : last;
    }
    __syncthreads();
    const int64_t p = (int64_t)s_pos * kTile + t;
    const double off = s_off;
    __syncthreads();
    if (t == 0) { s_pos = kTile; s_last = 0; }
    const double v = p < a.N ? __ldcg(a.closest + p) : 0.0;
    const double run = block_scan(v, wt);   // its barriers order s_pos / s_last too
    if (v > 0.0) {
        if (off + run > r) atomicMin(&s_pos, t);
        atomicMax(&s_last, t);
    }
    __syncthreads();
    const int at = s_pos < kTile ? s_pos : s_last;
    if (t == at) a.seeds[i] = (int32_t)p;
}

template <bool VEC4, int G>
__global__ void __launch_bounds__(kTile)
kpp_step_kernel(const KppArgs a, int i) {
    constexpr int U = 4;              // points a subgroup screens at a time
    constexpr int S = 32 / G;         // subgroups of a warp
    __shared__ uint8_t s_list[kTile / 32][32], s_ex[kTile / 32][32];
    __shared__ double s_w[kTile / 32];
    __shared__ int s_lastblk;
    const int t = threadIdx.x, lane = t & 31, w = t >> 5, sub = lane % G, grp = lane / G;
    const float* c = a.X + (int64_t)a.seeds[i - 1] * a.D;
    const unsigned below = (1u << lane) - 1u;
    for (int tile = blockIdx.x; tile < a.n_tiles; tile += gridDim.x) {
        const int64_t p0 = (int64_t)tile * kTile + w * 32, p = p0 + lane;
        const bool in = p < a.N;
        const float cup = (in && i > 1) ? a.closest_up[p] : __int_as_float(0x7f800000);
        // the triangle inequality
        bool need = in;
        if (in && i > 1) need = !(a.dcc[a.own[p]] >= cup);
        unsigned m = __ballot_sync(0xffffffffu, need);
        int n = __popc(m);
        bool changed = false;
        if (n > 0) {
            uint8_t* list = s_list[w];
            uint8_t* ex = s_ex[w];
            if (need) list[__popc(m & below)] = (uint8_t)lane;
            __syncwarp();
            int ne = 0;               // points left for the float64 distance
            if (i > 1 && a.shrink > 0.f) {
                for (int k0 = 0; k0 < n; k0 += S * U) {
                    const float* xs[U];
                    int at[U];
#pragma unroll
                    for (int q = 0; q < U; ++q) {
                        const int k = k0 + q * S + grp;
                        at[q] = list[k < n ? k : n - 1];
                        xs[q] = a.X + (p0 + at[q]) * a.D;
                    }
                    float d[U];
                    screen<VEC4, G, U>(xs, c, a.D, sub, d);
#pragma unroll
                    for (int q = 0; q < U; ++q) {
                        const int k = k0 + q * S + grp;
                        const float cu = __shfl_sync(0xffffffffu, cup, at[q]);
                        const bool sure = d[q] > kTiny && d[q] < kHuge && d[q] * a.shrink >= cu;
                        const bool want = sub == 0 && k < n && !sure;
                        const unsigned em = __ballot_sync(0xffffffffu, want);
                        if (want) ex[ne + __popc(em & below)] = (uint8_t)at[q];
                        ne += __popc(em);
                    }
                }
                __syncwarp();
            } else {
                ex = list;
                ne = n;
            }
            for (int k0 = 0; k0 < ne; k0 += S) {
                const int k = k0 + grp;
                const int at = ex[k < ne ? k : ne - 1];
                const double d = exact64<VEC4, G>(a.X + (p0 + at) * a.D, c, a.D, sub);
                if (sub == 0 && k < ne) {
                    const int64_t q = p0 + at;
                    // (a distance takes the place of a NaN, inf - inf to an earlier seed)
                    if (i == 1 || d < a.closest[q] || isnan(a.closest[q])) {
                        a.closest[q] = d;
                        a.closest_up[q] = __double2float_ru(d);
                        a.own[q] = i - 1;
                        changed = true;
                    }
                }
            }
        }
        // the tile's sum (fixed order), only when one of its points moved
        if (__syncthreads_or(changed)) {
            double v = in ? a.closest[p] : 0.0;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if (lane == 0) s_w[w] = v;
            __syncthreads();
            if (t == 0) {
                double s = 0.0;
#pragma unroll
                for (int k = 0; k < kTile / 32; ++k) s += s_w[k];
                a.tile_sum[tile] = s;
            }
            __syncthreads();
        }
    }
    __threadfence();
    __syncthreads();
    if (t == 0) s_lastblk = atomicAdd(a.done, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!s_lastblk) return;
    __threadfence();
    if (t == 0) *a.done = 0u;
    kpp_select(a, i);
    __syncthreads();
    // bounds ||seed i - seed j||^2 / 4 for the next update (a quarter, so that
    // it compares with D(x)^2)
    const float* x = a.X + (int64_t)a.seeds[i] * a.D;
    for (int j0 = w * U; j0 < i; j0 += (kTile / 32) * U) {
        const float* xs[U];
        float d[U];
#pragma unroll
        for (int q = 0; q < U; ++q) xs[q] = a.X + (int64_t)a.seeds[j0 + q < i ? j0 + q : i - 1] * a.D;
        if (j0 < kMaxBoundSeeds) screen<VEC4, 32, U>(xs, x, a.D, lane, d);
#pragma unroll
        for (int q = 0; q < U; ++q)
            if (lane == 0 && j0 + q < i)
                a.dcc[j0 + q] = (j0 < kMaxBoundSeeds && d[q] > kTiny && d[q] < kHuge)
                                    ? 0.25f * d[q] * a.shrink : 0.f;
    }
}

__global__ void kpp_first_kernel(int32_t first, int32_t* seeds) { seeds[0] = first; }

}  // namespace

size_t kmeanspp_ws_bytes(int64_t N, int L) {
    const size_t tiles = (size_t)((N + kTile - 1) / kTile);
    return align_up(sizeof(double) * (size_t)N, 256) + align_up(sizeof(double) * (size_t)L, 256) +
           2 * align_up(sizeof(float) * (size_t)N, 256) + align_up(sizeof(double) * tiles, 256) +
           align_up(sizeof(float) * (size_t)L, 256) + 512;
}

slk_status kmeanspp_launch(slk_ctx* ctx, const float* X, int64_t N, int D, int L, int32_t first,
                           const double* u_host, int32_t* seeds, void* ws) {
    WsCarver wc(ws);
    KppArgs a{};
    a.X = X;
    a.N = N;
    a.D = D;
    a.n_tiles = (int)((N + kTile - 1) / kTile);
    a.closest = wc.take<double>((size_t)N);
    double* u = wc.take<double>((size_t)(L > 1 ? L - 1 : 1));
    a.u = u;
    a.seeds = seeds;
    a.closest_up = wc.take<float>((size_t)N);
    a.own = wc.take<int32_t>((size_t)N);
    a.tile_sum = wc.take<double>((size_t)a.n_tiles);
    a.dcc = wc.take<float>((size_t)L);
    a.done = wc.take<unsigned>(1);
    // a float32 squared distance of D terms: at most D/32 + 8 roundings of its
    // sums and 2 of each difference, taken twice over; rows so long that this
    // says nothing are not screened
    const double rel = ((double)D / 32.0 + 32.0) * 1.1920928955078125e-07;
    if (L > 1) {
        SLK_CUDA_TRY(ctx, cudaMemcpyAsync(u, u_host, sizeof(double) * (size_t)(L - 1),
                                          cudaMemcpyHostToDevice, ctx->stream));
        SLK_CUDA_TRY(ctx, cudaMemsetAsync(a.done, 0, sizeof(unsigned), ctx->stream));
    }
    SLK_COUNT_LAUNCH(ctx, L);
    kpp_first_kernel<<<1, 1, 0, ctx->stream>>>(first, seeds);
    SLK_LAUNCH_CHECK(ctx, "kpp_first_kernel");
    const bool vec4 = (D % 4 == 0) && ((reinterpret_cast<uintptr_t>(X) & 15) == 0);
    // lanes per point: the smallest power of two that covers a row's words
    const int words = vec4 ? D / 4 : D;
    int g = 1;
    while (g < words && g < 32) g *= 2;
    // with G < 32 the lanes' words are one each: the float32 sums pass through
    // at most 4 + 5 roundings, within rel
    a.shrink = rel < 0.5 ? (float)(1.0 - rel) : 0.f;
    int64_t grid = a.n_tiles;
    if (grid > (int64_t)ctx->num_sms * 8) grid = (int64_t)ctx->num_sms * 8;
    for (int i = 1; i < L; ++i) {
#define SLK_KPP(V_, G_) kpp_step_kernel<V_, G_><<<(unsigned)grid, kTile, 0, ctx->stream>>>(a, i)
        if (vec4) {
            if (g <= 4) SLK_KPP(true, 4);
            else if (g == 8) SLK_KPP(true, 8);
            else if (g == 16) SLK_KPP(true, 16);
            else SLK_KPP(true, 32);
        } else {
            if (g <= 4) SLK_KPP(false, 4);
            else if (g == 8) SLK_KPP(false, 8);
            else if (g == 16) SLK_KPP(false, 16);
            else SLK_KPP(false, 32);
        }
#undef SLK_KPP
        SLK_LAUNCH_CHECK(ctx, "kpp_step_kernel");
    }
    return SLK_OK;
}
