// Unary term, kNN-edge weights and the discrete energy.
//
// Unary, Eq. (general-second) with the Gaussian kernel of Section 4.2:
//   a_{p,l} = exp(-||x_p - m_l||^2 / (2 sigma^2)),  z_p^0 = softmax(a_p) (Algorithm 1),
// m_l = x_{modes[l]} (SLK-BO) or a row of the mode vectors M (SLK-MS).
// Energy, Eq. (1) at one-hot z:
//   E = -sum_p k(x_p, m_{l_p}) + (lambda/2) sum_p sum_{e in row p} w_e ||z_p - z_q||^2.
#include <math.h>
#include <stdint.h>

#include "slk_internal.cuh"

namespace {

constexpr int kUPG = 128;      // points per point group (4 per lane)
constexpr int kUDC = 32;       // feature chunk staged in shared memory (float32 partial sums)
constexpr int kUThreads = 256;
constexpr int kUS = kUDC + 4;  // row stride of a staged point: 16-byte rows, eight of them on all 32 banks

// Row stride of the staged mode values: 4 G rounded up to 4 x odd, so that
// 16-byte rows stay aligned and the staging stores are at most 4-way
// bank-conflicted.
__host__ __device__ inline int unary_mode_stride(int G) { return 4 * (G | 1); }

// 4-byte asynchronous global -> shared copy; n = 0 fills the word with zero
// (the source is then not read).
__device__ __forceinline__ void cp_async4(float* dst, const float* src, int n) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ void cp_async16(float* dst, const float* src, int n) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait0() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait1() { asm volatile("cp.async.wait_group 1;" ::: "memory"); }

// Thread tile: 4 points (lane + 32 i) x 4 labels.  A warp covers one point
// group of 128 and one label group of 4; a block holds PG point groups and G
// label groups (G PG warps), and loops over passes of 4 G labels.  Features
// go in chunks of 32: X staged [point][36] (16-byte copies where the rows
// allow, a thread reads four features of a point at once), the pass's mode
// values [feature][S] (S = 4 x odd: one 16-byte broadcast per label group),
// two buffers filled by asynchronous copies so that the next chunk (of this
// pass or the next) loads while this one is summed.  Each pair's squared
// differences over a chunk are summed in float32 in feature order; the chunk
// sums are added as an unevaluated pair of floats (2Sum: about as accurate as a
// float64 sum and off the slow float64 pipe).  Vector modes (SLK-MS) come as M
// (float32) or as a float64 state split into M + Mlo (LO): (x - m_hi) - m_lo
// keeps the difference accurate to float32 relative to itself, not to |m|.
//
// The sums take N L D differences and products; what it spent beyond them were
// the copies of four bytes and the rows of A and Z0, written and read by one
// lane per row.  So a pass's values of A go through the freed buffer and out as
// they lie in memory; with one pass the softmax is formed there too, a thread per
// row, with several the rows come back and are spread over groups of 8, 16 or 32
// lanes, the fewest idle.  (With a power of two of lanes per row throughout, rows of
// 9, 20 or 33 labels left half of them idle: 10 to 25 % slower than a lane per row
// at 100000 x 9 and 20000 x 50.)  Three blocks per SM (two where the second half
// of the modes takes registers); blocks of one point group, two only where a
// block has one label group; a single buffer where there is only one step.
// Kernel alone, with the lane per row and now: 10^6 x 128, L = 100: 3.15 and
// 2.16 ms (float32 units 0.64); L = 5: 0.291 and 0.197; 70000 x 784, L = 10: 0.17
// and 0.11; 100000 x 9, L = 20: 0.031 and 0.024.
template <bool LO, bool V4>
__global__ void __launch_bounds__(kUThreads, LO ? 2 : 3)
unary_kernel(const float* __restrict__ X, int64_t N, int D, const int32_t* __restrict__ modes,
             const float* __restrict__ M, const float* __restrict__ Mlo, int L, int G, int PG,
             const float* __restrict__ sigma_dev, float* __restrict__ A, float* __restrict__ Z0) {
    constexpr int PPL = kUPG / 32;   // points per lane
    extern __shared__ __align__(16) float sm[];
    const int S = unary_mode_stride(G), npts = PG * kUPG;
    const int nthr = blockDim.x;
    const int xbuf = npts * kUS, mbuf = kUDC * S;
    float* xs = sm;                                    // 2 x [npts][kUS]
    const int nch = (D + kUDC - 1) / kUDC;
    const int nsteps = ((L + 4 * G - 1) / (4 * G)) * nch;   // (pass, chunk) pairs
    const int bufs = nsteps > 1 ? 2 : 1;
    float* mh = xs + bufs * xbuf;                      // 2 x [kUDC][S]
    float* mlo = mh + bufs * mbuf;                     // 2 x [kUDC][S] (LO only)
    __shared__ int mrow[SLK_MAX_L];
    __shared__ float zsum[2 * kUPG];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int g = warp % G, pg = warp / G;
    const int64_t p0 = (int64_t)blockIdx.x * npts;
    const int rows = (int)min((int64_t)npts, N - p0);
    // nl labels from l0 of the block's first n rows, as they lie in memory
    auto each = [&](int n, int nl, auto&& f) {
        const int dr = nthr / nl, dl = nthr - dr * nl;
        int r = t / nl, l = t - r * nl;
#pragma unroll 4
        while (r < n) {
            f(r, l);
            r += dr;
            l += dl;
            if (l >= nl) {
                l -= nl;
                ++r;
            }
        }
    };
    const bool kept = L <= 4 * G;   // one pass: the softmax needs no way back from A
    if (M == nullptr)
        for (int l = t; l < L; l += nthr) mrow[l] = modes[l];
    __syncthreads();
    const float sg = *sigma_dev;
    const float inv2s2 = 1.0f / (2.0f * sg * sg);
    // Step s: pass s / nch (labels l0 = 4 G (s / nch) ..), chunk s % nch, buffer s & 1.
    auto stage = [&](int s) {
        const int d0 = (s % nch) * kUDC, l0 = (s / nch) * 4 * G, b = s & 1;
        const int dc = min(kUDC, D - d0);
        float* xb = xs + b * xbuf;
        if (V4) {
            for (int i = t; i < npts * (kUDC / 4); i += nthr) {
                const int r = i / (kUDC / 4), c = 4 * (i % (kUDC / 4));
                const int64_t p = p0 + r;
                const bool ok = p < N && c < dc;
                cp_async16(xb + r * kUS + c, ok ? X + p * D + d0 + c : X, ok ? 16 : 0);
            }
        } else {
            for (int i = t; i < npts * kUDC; i += nthr) {
                const int r = i / kUDC, c = i % kUDC;
                const int64_t p = p0 + r;
                const bool ok = p < N && c < dc;
                cp_async4(xb + r * kUS + c, ok ? X + p * D + d0 + c : X, ok ? 4 : 0);
            }
        }
        float* hb = mh + b * mbuf;
        float* lb = mlo + b * mbuf;
        for (int i = t; i < 4 * G * kUDC; i += nthr) {
            const int r = i / kUDC, c = i % kUDC;   // label l0 + r, feature d0 + c
            const int l = l0 + r;
            const bool ok = l < L && c < dc;
            const float* src = !ok ? X : M ? M + (int64_t)l * D + d0 + c
                                          : X + (int64_t)mrow[l] * D + d0 + c;
            cp_async4(hb + c * S + r, src, ok ? 4 : 0);
            if (LO) cp_async4(lb + c * S + r, ok ? Mlo + (int64_t)l * D + d0 + c : Mlo, ok ? 4 : 0);
        }
        cp_async_commit();
    };
    stage(0);
    float hi[PPL][4], lo[PPL][4];   // chunk sums added as an unevaluated float pair (2Sum)
    for (int s = 0; s < nsteps; ++s) {
        const int k = s % nch, l0 = (s / nch) * 4 * G, b = s & 1;
        const int dc = min(kUDC, D - k * kUDC);
        if (k == 0) {
#pragma unroll
            for (int i = 0; i < PPL; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    hi[i][j] = 0.f;
                    lo[i][j] = 0.f;
                }
        }
        if (s + 1 < nsteps) stage(s + 1);
        else cp_async_commit();          // an empty group keeps the wait count uniform
        cp_async_wait1();                // this thread's copies of step s have landed
        __syncthreads();                 // ... and every thread's
        const float* xrow = xs + b * xbuf + (pg * kUPG + lane) * kUS;
        const float* hb = mh + b * mbuf + 4 * g;
        const float* lb = mlo + b * mbuf + 4 * g;
        float part[PPL][4];
#pragma unroll
        for (int i = 0; i < PPL; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) part[i][j] = 0.f;
        // (zeros past the last feature add nothing)
        for (int c = 0; c < dc; c += 4) {
            float4 x4[PPL];
#pragma unroll
            for (int i = 0; i < PPL; ++i)
                x4[i] = *reinterpret_cast<const float4*>(xrow + 32 * i * kUS + c);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const float4 h4 = *reinterpret_cast<const float4*>(hb + (c + u) * S);
                const float m[4] = {h4.x, h4.y, h4.z, h4.w};
                float ml[4] = {0.f, 0.f, 0.f, 0.f};
                if (LO) {
                    const float4 l4 = *reinterpret_cast<const float4*>(lb + (c + u) * S);
                    ml[0] = l4.x; ml[1] = l4.y; ml[2] = l4.z; ml[3] = l4.w;
                }
#pragma unroll
                for (int i = 0; i < PPL; ++i) {
                    const float x = u == 0 ? x4[i].x : u == 1 ? x4[i].y : u == 2 ? x4[i].z : x4[i].w;
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        float df = x - m[j];
                        if (LO) df -= ml[j];
                        part[i][j] = fmaf(df, df, part[i][j]);
                    }
                }
            }
        }
#pragma unroll
        for (int i = 0; i < PPL; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                // 2Sum (Knuth): s + e == hi + part exactly
                const float sum = __fadd_rn(hi[i][j], part[i][j]);
                const float bb = __fsub_rn(sum, hi[i][j]);
                const float e = __fadd_rn(__fsub_rn(hi[i][j], __fsub_rn(sum, bb)),
                                          __fsub_rn(part[i][j], bb));
                lo[i][j] = __fadd_rn(lo[i][j], e);
                hi[i][j] = sum;
            }
        __syncthreads();                 // buffer b is read
        if (k == nch - 1) {
            float* out = xs + b * xbuf;
#pragma unroll
            for (int i = 0; i < PPL; ++i) {
                float a[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) a[j] = expf(-__fadd_rn(hi[i][j], lo[i][j]) * inv2s2);
                *reinterpret_cast<float4*>(out + (pg * kUPG + lane + 32 * i) * kUS + 4 * g) =
                    make_float4(a[0], a[1], a[2], a[3]);
            }
            __syncthreads();
            auto put_a = [&](int r, int l) { A[(p0 + r) * L + l0 + l] = out[r * kUS + l]; };
            const bool one = nsteps == 1;   // the only step has a single buffer
            if (one) {
                each(rows, L, put_a);
                __syncthreads();
            }
            if (kept && Z0) {   // a thread per row: exp (beside A where there is room) and the sum
                float* z = one ? out : xs + (b ^ 1) * xbuf;
                for (int r = t; r < rows; r += nthr) {
                    const float* ar = out + r * kUS;
                    float m = -INFINITY, sum = 0.f;
#pragma unroll 2
                    for (int l = 0; l < L; l += 4) {
                        const float4 v = *reinterpret_cast<const float4*>(ar + l);
                        m = fmaxf(m, v.x);
                        if (l + 1 < L) m = fmaxf(m, v.y);
                        if (l + 2 < L) m = fmaxf(m, v.z);
                        if (l + 3 < L) m = fmaxf(m, v.w);
                    }
#pragma unroll 2
                    for (int l = 0; l < L; l += 4) {
                        float4 v = *reinterpret_cast<const float4*>(ar + l);
                        v = make_float4(expf(v.x - m), expf(v.y - m), expf(v.z - m), expf(v.w - m));
                        sum += v.x;
                        if (l + 1 < L) sum += v.y;
                        if (l + 2 < L) sum += v.z;
                        if (l + 3 < L) sum += v.w;
                        *reinterpret_cast<float4*>(z + r * kUS + l) = v;
                    }
                    zsum[r] = sum;
                }
            }
            if (!one) each(rows, min(4 * G, L - l0), put_a);
            __syncthreads();             // buffer b is free for step s + 2
        }
    }
    if (Z0 == nullptr) return;
    if (kept) {
        const float* z = nsteps == 1 ? xs : xs + (nsteps & 1) * xbuf;
        each(rows, L, [&](int r, int l) { Z0[(p0 + r) * L + l] = z[r * kUS + l] / zsum[r]; });
        return;
    }
    // several passes: the block's rows of A (written, last barrier) come back, as
    // many as fit
    const int Ls = L | 1, batch = min(npts, 2 * xbuf / Ls);
    int LR = 32;
    for (int q = 16; q >= 8; q >>= 1)
        if ((L + q - 1) / q * q < (L + LR - 1) / LR * LR) LR = q;
    const int gl = lane % LR, gr = t / LR, ng = nthr / LR;
    for (int r0 = 0; r0 < rows; r0 += batch) {
        const int nr = min(batch, rows - r0);
        each(nr, L, [&](int r, int l) { cp_async4(xs + r * Ls + l, A + (p0 + r0 + r) * L + l, 4); });
        cp_async_commit();
        cp_async_wait0();
        __syncthreads();
#pragma unroll 2
        for (int r = gr; r - gr < nr; r += ng) {   // (all lanes take part in the shuffles)
            float* ar = xs + min(r, nr - 1) * Ls;
            float m = -INFINITY;
            for (int l = gl; l < L; l += LR) m = fmaxf(m, ar[l]);
            for (int o = LR >> 1; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
            if (r < nr)
                for (int l = gl; l < L; l += LR) ar[l] = expf(ar[l] - m);
        }
        __syncthreads();
        for (int r = t; r < nr; r += nthr) {
            float s = 0.f;
#pragma unroll 8
            for (int l = 0; l < L; ++l) s += xs[r * Ls + l];
            zsum[r] = s;
        }
        __syncthreads();
        each(nr, L, [&](int r, int l) { Z0[(p0 + r0 + r) * L + l] = xs[r * Ls + l] / zsum[r]; });
        __syncthreads();
    }
}

__global__ void weights_kernel(const float* __restrict__ dist2, int64_t nnz, int heat,
                               const float* __restrict__ sigma_dev, float* __restrict__ w) {
    const float sg = heat ? *sigma_dev : 1.f;
    const float inv2s2 = 1.0f / (2.0f * sg * sg);
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < nnz;
         e += (int64_t)gridDim.x * blockDim.x)
        w[e] = heat ? expf(-dist2[e] * inv2s2) : 1.f;
}

__global__ void set_sigma_kernel(float sigma, DevState* st) { st->sigma = sigma; }

// One warp per point: squared distance to its mode (warp_sq_dist) and the
// cut edges of its row (weights summed as float pairs).  Lane i keeps the
// distance and cut of the warp's points i, i + 32, ... until it has to add
// them, so that the float64 kernel value exp(-d2 / (2 sigma^2)) is one
// warp-wide instruction sequence per 32 points rather than one single-lane
// sequence per point.  V4: 16-byte row loads (warp_sq_dist4).
template <bool V4>
__global__ void __launch_bounds__(256, 4)
energy_kernel(const float* __restrict__ X, int D, const int32_t* __restrict__ labels,
              const int64_t* __restrict__ row_ptr, const int32_t* __restrict__ col_idx,
              const float* __restrict__ w, int64_t N, const int32_t* __restrict__ modes,
              const float* __restrict__ M, const float* __restrict__ Mlo,
              const float* __restrict__ sigma_dev, float lambda, DevState* st) {
    __shared__ double red[8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const double sg = (double)*sigma_dev;
    const double inv2s2 = 1.0 / (2.0 * sg * sg);
    double acc = 0.0;  // per-lane partial of E
    const int64_t nwarps = (int64_t)gridDim.x * 8;
    double my_d2 = 0.0, my_cut = 0.0;
    bool mine = false;
    int slot = 0;   // lane that keeps the current point
    for (int64_t p = (int64_t)blockIdx.x * 8 + warp; p < N; p += nwarps) {
        const int lp = labels[p];
        const float* xp = X + p * D;
        const float* xm = M ? M + (int64_t)lp * D : X + (int64_t)modes[lp] * D;
        const float* xl = Mlo ? Mlo + (int64_t)lp * D : nullptr;
        const double d2 = V4 ? warp_sq_dist4(xp, xm, xl, D, lane) : warp_sq_dist(xp, xm, xl, D, lane);
        float ch = 0.f, cl = 0.f;
        for (int64_t e = row_ptr[p] + lane; e < row_ptr[p + 1]; e += 32) {
            const int q = col_idx[e];
            if (labels[q] != lp) fpair_add(ch, cl, w ? w[e] : 1.f, 0.f);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
            fpair_add(ch, cl, __shfl_xor_sync(0xffffffffu, ch, o), __shfl_xor_sync(0xffffffffu, cl, o));
        if (lane == slot) {
            my_d2 = d2;
            my_cut = (double)ch + (double)cl;
            mine = true;
        }
        if (++slot == 32) {
            // ||z_p - z_q||^2 = 2 for every cut edge
            if (mine) acc += -exp(-my_d2 * inv2s2) + 0.5 * (double)lambda * 2.0 * my_cut;
            mine = false;
            slot = 0;
        }
    }
    if (mine) acc += -exp(-my_d2 * inv2s2) + 0.5 * (double)lambda * 2.0 * my_cut;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) red[warp] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int i = 0; i < 8; ++i) s += red[i];
        atomicAdd(&st->energy, s);
    }
}

}  // namespace

slk_status unary_launch(slk_ctx* ctx, const float* X, int64_t N, int D, const int32_t* modes,
                        int L, const float* sigma_dev, float* A, float* Z0, const float* M,
                        const float* Mlo) {
    PhaseScope ps(ctx, SLK_PHASE_UNARY);
    SLK_COUNT_LAUNCH(ctx, 1);
    // label groups of 4: up to 8 warps per pass, the passes balanced
    const int gtot = (L + 3) / 4;
    const int passes = (gtot + 7) / 8;
    const int G = (gtot + passes - 1) / passes;
    const int PG = G == 1 ? 2 : 1;
    const int bufs = passes > 1 || D > kUDC ? 2 : 1;
    const size_t smem = bufs * sizeof(float) * ((size_t)PG * kUPG * kUS +
                                             (Mlo ? 2 : 1) * (size_t)kUDC * unary_mode_stride(G));
    // 16-byte copies need every row of X on a 16-byte boundary
    const bool v4 = (D & 3) == 0 && (reinterpret_cast<uintptr_t>(X) & 15) == 0;
    auto kern = Mlo ? (v4 ? unary_kernel<true, true> : unary_kernel<true, false>)
                    : (v4 ? unary_kernel<false, true> : unary_kernel<false, false>);
    SLK_CUDA_TRY(ctx, cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    const int64_t npts = (int64_t)PG * kUPG;
    const unsigned grid = (unsigned)((N + npts - 1) / npts);
    kern<<<grid, 32 * G * PG, smem, ctx->stream>>>(X, N, D, modes, M, Mlo, L, G, PG, sigma_dev, A, Z0);
    SLK_LAUNCH_CHECK(ctx, "unary_kernel");
    return SLK_OK;
}

slk_status weights_launch(slk_ctx* ctx, const float* dist2, int64_t nnz, int affinity,
                          const float* sigma_dev, float* w) {
    SLK_COUNT_LAUNCH(ctx, 1);
    int64_t grid = (nnz + 255) / 256;
    if (grid > (int64_t)ctx->num_sms * 16) grid = (int64_t)ctx->num_sms * 16;
    if (grid < 1) grid = 1;
    weights_kernel<<<(unsigned)grid, 256, 0, ctx->stream>>>(
        dist2, nnz, affinity == SLK_AFFINITY_HEAT ? 1 : 0, sigma_dev, w);
    SLK_LAUNCH_CHECK(ctx, "weights_kernel");
    return SLK_OK;
}

slk_status set_sigma_launch(slk_ctx* ctx, float sigma, DevState* st) {
    SLK_COUNT_LAUNCH(ctx, 1);
    set_sigma_kernel<<<1, 1, 0, ctx->stream>>>(sigma, st);
    SLK_LAUNCH_CHECK(ctx, "set_sigma_kernel");
    return SLK_OK;
}

slk_status energy_launch(slk_ctx* ctx, const float* X, int D, const int32_t* labels,
                         const int64_t* row_ptr, const int32_t* col_idx, const float* w,
                         int64_t N, int L, const int32_t* modes, const float* sigma_dev,
                         float lambda, DevState* st, const float* M, const float* Mlo) {
    (void)L;
    PhaseScope ps(ctx, SLK_PHASE_ENERGY);
    SLK_COUNT_LAUNCH(ctx, 1);
    SLK_CUDA_TRY(ctx, cudaMemsetAsync(&st->energy, 0, sizeof(double), ctx->stream));
    int64_t grid = (N + 7) / 8;   // one wave: 4 CTAs per SM (launch bounds)
    if (grid > (int64_t)ctx->num_sms * 4) grid = (int64_t)ctx->num_sms * 4;
    auto al16 = [](const float* q) { return (reinterpret_cast<uintptr_t>(q) & 15) == 0; };
    const bool v4 = D % 4 == 0 && al16(X) && (M == nullptr || al16(M)) && (Mlo == nullptr || al16(Mlo));
    if (v4)
        energy_kernel<true><<<(unsigned)grid, 256, 0, ctx->stream>>>(
            X, D, labels, row_ptr, col_idx, w, N, modes, M, Mlo, sigma_dev, lambda, st);
    else
        energy_kernel<false><<<(unsigned)grid, 256, 0, ctx->stream>>>(
            X, D, labels, row_ptr, col_idx, w, N, modes, M, Mlo, sigma_dev, lambda, st);
    SLK_LAUNCH_CHECK(ctx, "energy_kernel");
    return SLK_OK;
}
