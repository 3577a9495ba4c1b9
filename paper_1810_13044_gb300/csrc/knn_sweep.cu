// Candidates of the exact kNN graph on the tensor cores (tcgen05): for 128-row
// blocks of points against 256-column tiles,
//   dt(p, q) = ||xt_p||^2 + ||xt_q||^2 - 2 xt_p . xt_q
// in bfloat16 products with float32 accumulation; every row keeps the columns
// whose dt can still belong to one of its k nearest (knn_cert.cuh).
//
// One persistent CTA per SM:
//   warp 0      TMA producer: 64-wide K slices of the A (128 rows) and B
//               (256 rows) tiles, 128-byte swizzle, into a 3-stage ring;
//   warp 1      TMEM owner (512 columns = two 128 x 256 fp32 accumulators)
//               and MMA issuer (one thread, M = 128, N = 256, K = 16);
//   warps 2-5   epilogue, one row per thread (TMEM lanes 32 (w % 4) .. +31).
// Forms of the K loop:
//   PLAIN  the points' slices; the epilogue forms w = fl(||xt_q||^2 - 2 dot)
//          and compares it with the threshold less ||xt_p||^2 rounded up;
//   AUG    (Dp <= 256) one more slice of 16 columns folds the norms in:
//          [1, 1, 1, a_p] against [a_q, 1, 1, 1], a the three bfloat16 terms of
//          -||xt||^2 / 2, so the accumulator holds -dt / 2 and the epilogue
//          only compares (padding rows and columns carry -inf);
//   RES    (Dp <= 128) AUG with the row block's A slices and its folded-norm
//          slice resident in shared memory: the ring carries B slices only,
//          72 KiB per tile instead of 108;
//   SPLIT  two-term operands s = h + l of listed query rows: three passes over
//          the slices, h . h, h . l, l . h.
//
// The epilogue is what bounded these tiles when it kept each row's 32 or 64
// smallest dt as a sorted list: a merge (bitonic sort of 16 or 32 entries and a
// bitonic merge, unrolled) took 9 us per warp, and a row block needs 15 to 20
// of them however short its sweep.  Here a row has an unordered buffer of the
// columns below cert_thr(dk), dk an upper bound of its k-th smallest dt; appending
// is a predicated store.  When a buffer fills (a refresh), the warp lowers dk
// by counting the entries below trial values, and drops what the threshold has
// passed by: two short loops instead of the sort, and the threshold follows the
// k-th smallest, not the 32nd or 64th, so a block needs 5 to 12 of them.  A
// row that has more columns under its threshold than its list holds keeps the
// smallest ones and a bound on the rest.
// An insertion of every hit into the k smallest (min / max pairs, a branch per
// column) was slower: 0.71 ms against 0.37 at 19870 x 9, k = 5; with one warp
// per scheduler its chain of dependent instructions ran at 0.15 a cycle.
// Sweeps over every tile, the kernel with sorted lists and this one: 1.04 and
// 0.37 ms at 19870 x 9, 2.28 and 1.17 at 42099 x 64, 3.48 and 2.30 at 60001 x 50,
// 6.59 and 5.59 at 70000 x 784.  Points of one cluster, which leave no tile out,
// with k = 10: 19.6 and 15.7 ms at 200000 x 128, 87 and 79 at 500000 x 128, 126 and
// 126 at 500000 x 256, 293 and 291 at 1e6 x 128; with k = 24 hits are more (45
// instructions each) and the eight warps that took them for the sorted lists were
// quicker: 60.0 and 60.5 ms at 400000 x 128, 272 and 293 at 1e6 x 32.
//
// Every mbarrier wait is bounded in time; on a timeout the CTA raises an
// error bit, drains its own copies in flight, frees TMEM and returns.
#include <cstddef>
#include <type_traits>

#include "knn_cert.cuh"
#include "knn_sweep.cuh"
#include "tc_ptx.cuh"

namespace {

enum { PLAIN = 0, AUG = 1, RES = 2, SPLIT = 3 };

// Three operand stages and as many slots as fit beside them.  A stage's round
// trip (copy, MMAs, release) is longer than two stages' MMAs, so with two of them
// large sweeps waited for operands: 315 ms at 1e6 x 128 (now 291), 169 at 500000 x
// 256 (now 126).  More and smaller stages were slower: half slices of B's features
// (five, 64-byte rows) 367 ms at 1e6 x 128, half tiles of columns (five, N = 128)
// 459.  Slots fewer than 76 refresh the rows too often where clusters are dense:
// 1e6 x 128 manifolds 86.8 ms with 76, 91 with 72, 105 with 64 (87.6 with 80 and two
// stages); 104 slots lose 10 % at 19870 x 9, k = 5 (longer refreshes).
template <int FORM> struct Shape {
    static constexpr bool fold = FORM == AUG || FORM == RES;
    static constexpr int stages = 3;
    static constexpr int slots = FORM == RES ? 76 : 80;   // buffered candidates per row
};
constexpr int GRP = 8;               // columns appended between room checks
constexpr int RES_MAX_DP = 128;
constexpr int THREADS = 192;
constexpr int CHUNK = 32;            // columns per TMEM load

template <int FORM>
struct Smem {
    static constexpr int STAGES = Shape<FORM>::stages, SLOTS = Shape<FORM>::slots;
    uint8_t a[FORM == RES ? RES_MAX_DP / TC_BK : STAGES][A_BYTES];   // 1024-byte aligned
    uint8_t b[STAGES][B_BYTES];
    // candidates of each row (column = row of the block); a refresh reads them by
    // eights, up to four slots past the end (into what follows)
    float buf_d[SLOTS][TC_M];
    int buf_i[SLOTS][TC_M];
    uint8_t a_aug[FORM == RES ? AUG_A_BYTES : 16];   // 1024-byte aligned
    uint8_t b_aug[2][FORM == RES ? AUG_B_BYTES : 16];
    unsigned long long full[STAGES], empty[STAGES], tfull[2], tempty[2], afull, aempty;
    unsigned long long colbar[8];    // tile column handed from the producer to the epilogue
    int tcol[8];
    uint32_t tmem_base;
    int abort;
};
static_assert(offsetof(Smem<RES>, a_aug) % 1024 == 0 && Shape<RES>::stages == 3, "folded norms");
static_assert(sizeof(Smem<RES>) + 1024 <= 232448 && sizeof(Smem<AUG>) + 1024 <= 232448 &&
              sizeof(Smem<PLAIN>) + 1024 <= 232448, "shared memory");

// Place of a tile's folded norms (RES).  A slot is free again when the stage of
// a later tile's last slice is: with two slices a tile and three stages that
// stage's last MMAs were those of the tile in between, so two slots are enough;
// with one slice it takes as many as stages, the last in A's second slice, which
// such a form does not use.
template <int FORM>
__device__ __forceinline__ uint8_t* aug_slot(Smem<FORM>& s, int nkb0, uint32_t stage, uint32_t tile) {
    const uint32_t i = nkb0 == 1 ? stage : tile & 1u;
    return i == 2u ? s.a[1] : s.b_aug[i];
}

struct SweepArgs {
    SweepWork w;
    SweepLists out;
    const float* row_norms;
    const float* col_norms;
    const float* rho;
    const int32_t* ids;
    const long long* rows_dev;
    float* thr;                // per row, out (nullable)
    float* kth;                // resume: k-th smallest dt per row of the lists continued; else out
    int64_t n_rows;            // rows (points form)
    int D, Dp, k, resume;
    double gam;
    const DevState* st;
    unsigned* err_flag;
    unsigned long long* sweep;
};

// The pieces of this CTA: false when it has no more.
struct Pieces {
    int64_t g, ge;
    int rb;
    __device__ void begin(const SweepWork& w) {
        if (w.aligned && !w.tiles) {   // whole row blocks, dealt out in turn
            rb = blockIdx.x;
            return;
        }
        const int64_t total = sweep_total(w), chunk = sweep_chunk(w, total);
        g = (int64_t)blockIdx.x * chunk;
        ge = g + chunk < total ? g + chunk : total;
        rb = 0;
        if (!w.tiles) {
            rb = g < total ? (int)(g / w.per) : 0;
        } else if (g < ge) {
            int lo = 0, hi = w.row_blocks;   // last block with start <= g
            while (hi - lo > 1) {
                const int mid = (lo + hi) >> 1;
                if (w.start[mid] <= g) lo = mid; else hi = mid;
            }
            rb = lo;
        }
    }
    __device__ bool next(const SweepWork& w, int& block, int& i0, int& i1) {
        if (w.aligned && !w.tiles) {
            if (rb >= w.row_blocks) return false;
            block = rb;
            i0 = 0;
            i1 = w.per;
            rb += gridDim.x;
            return true;
        }
        while (g < ge) {
            int64_t s0, s1;
            sweep_block(w, rb, s0, s1);
            if (g >= s1) { ++rb; continue; }
            const int64_t e = ge < s1 ? ge : s1;
            block = rb;
            i0 = (int)(g - s0);
            i1 = (int)(e - s0);
            g = e;
            return true;
        }
        return false;
    }
};

__device__ __forceinline__ int tile_at(const SweepWork& w, int rb, int i) {
    return w.tiles ? __ldg(w.tiles + w.start[rb] + i) : sweep_tile0(w, rb) + i;
}

// A row's buffer, its threshold and what it is derived from.
struct RowState {
    int cnt;       // buffered entries
    float dk;      // k of the columns seen have dt <= dk
    float tcap;    // lowered when more columns lie under the threshold than the
                   // list holds: the row keeps its smallest ones and every other
                   // column has dt >= tcap (-inf: ties, the row is left open)
    float thr;
};

// Entries of a lane's buffer at or below (LE) or below three values.
template <bool LE>
__device__ __forceinline__ void count3(const float* d, int cnt, int top, float m1, float m2, float m3, int& c1,
                                       int& c2, int& c3) {
    c1 = c2 = c3 = 0;
    for (int e0 = 0; e0 < top; e0 += 8) {
        float v[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] = d[(e0 + e) * TC_M];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const float x = e0 + e < cnt ? v[e] : __int_as_float(0x7f800000);
            c1 += LE ? x <= m1 : x < m1;
            c2 += LE ? x <= m2 : x < m2;
            c3 += LE ? x <= m3 : x < m3;
        }
    }
}

// Refresh of the warp's 32 rows (lane = row): lower dk, drop what the threshold
// has passed by, and with more than `most` entries left keep at most `keep`
// (the smallest).  Loads are issued eight at a time; the searches count the
// entries below three trial values per pass.
__device__ __noinline__ RowState refresh(float* d, int* idx, RowState s, int k, int most, int keep, bool all,
                                         const CertConsts& cc, float sp, float rp) {
    const float inf = __int_as_float(0x7f800000);
    const int top = (__reduce_max_sync(0xffffffffu, s.cnt) + 7) & ~7;   // at most the buffer (a multiple of 8)
    float mn = inf, mx = -inf;
    for (int e0 = 0; e0 < top; e0 += 8) {
        float v[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] = d[(e0 + e) * TC_M];
#pragma unroll
        for (int e = 0; e < 8; ++e)
            if (e0 + e < s.cnt) {
                mn = fminf(mn, v[e]);
                mx = fmaxf(mx, v[e]);
            }
    }
    // an upper bound of the k-th smallest entry, within 2^-8 of its range (dk
    // says nothing while a capped row's bound is the lower one)
    const bool low = s.cnt >= k && (all || s.thr < s.tcap || s.tcap == inf);
    if (__any_sync(0xffffffffu, low)) {
        float lo = mn, hi = fminf(s.dk, mx);
#pragma unroll 1
        for (int it = 0; it < 4; ++it) {
            const float w = 0.25f * (hi - lo);
            const float m1 = lo + w, m2 = lo + 2.f * w, m3 = lo + 3.f * w;
            int c1, c2, c3;
            count3<true>(d, s.cnt, top, m1, m2, m3, c1, c2, c3);
            if (c1 >= k) hi = m1;
            else if (c2 >= k) { lo = m1; hi = m2; }
            else if (c3 >= k) { lo = m2; hi = m3; }
            else lo = m3;
        }
        if (low) s.dk = hi;
    }
    s.thr = fminf(s.tcap, cert_thr(cc, sp, rp, s.dk));
    int n, n2, n3;
    count3<false>(d, s.cnt, top, s.thr, s.thr, s.thr, n, n2, n3);
    if (__any_sync(0xffffffffu, n > most)) {
        // a threshold below which between k and `keep` entries stay
        float lo = mn, hi = fminf(s.thr, mx);
        int below = 0;
        const bool cut = n > most;
#pragma unroll 1
        for (int it = 0; it < 4 && __any_sync(0xffffffffu, cut && below < keep - 6); ++it) {
            const float w = 0.25f * (hi - lo);
            const float m1 = lo + w, m2 = lo + 2.f * w, m3 = lo + 3.f * w;
            int c1, c2, c3;
            count3<false>(d, s.cnt, top, m1, m2, m3, c1, c2, c3);
            if (c3 <= keep) { lo = m3; below = c3; }
            else if (c2 <= keep) { lo = m2; below = c2; hi = m3; }
            else if (c1 <= keep) { lo = m1; below = c1; hi = m2; }
            else hi = m1;
        }
        if (cut) s.thr = s.tcap = below >= k ? lo : -inf;
    }
    __syncwarp();
    n = 0;
    for (int e0 = 0; e0 < top; e0 += 8) {
        float v[8];
        int c[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            v[e] = d[(e0 + e) * TC_M];
            c[e] = idx[(e0 + e) * TC_M];
        }
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            if (e0 + e < s.cnt && v[e] < s.thr) {
                d[n * TC_M] = v[e];
                idx[n * TC_M] = c[e];
                ++n;
            }
        }
    }
    s.cnt = n;
    return s;
}
// A refresh cuts a list of more than FULL entries to at most KEEP, so that the
// buffer has room for some 20 more (with KEEP = 60 fewer rows stay open, but it
// fills again after about ten).
constexpr int FULL = 54, KEEP = 52;

template <int FORM>
__global__ void __launch_bounds__(THREADS, 1)
knn_sweep_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                 const __grid_constant__ CUtensorMap tmA2, const __grid_constant__ CUtensorMap tmB2,
                 const SweepArgs a_in) {
    constexpr bool FOLD = Shape<FORM>::fold;
    constexpr int STAGES = Shape<FORM>::stages, SLOTS = Shape<FORM>::slots;
    extern __shared__ uint8_t smem_raw[];
    using SMT = Smem<FORM>;
    SMT& s = *reinterpret_cast<SMT*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const float inf = __int_as_float(0x7f800000);
    SweepWork w = a_in.w;
    int64_t n_rows = a_in.n_rows;
    if constexpr (FORM == SPLIT) {
        // query rows counted on the device (every thread reads the same value)
        long long rows = *a_in.rows_dev;
        const long long cap = (long long)w.row_blocks * TC_M;
        if (rows > cap) rows = cap;
        if (rows < 0) rows = 0;
        n_rows = rows;
        w.row_blocks = (int)((rows + TC_M - 1) / TC_M);
    }
    const int nkb0 = a_in.Dp / TC_BK;             // K slices of one operand pass
    const int nkb = FORM == SPLIT ? 3 * nkb0 : (FORM == AUG ? nkb0 + 1 : nkb0);
    volatile int* abort = &s.abort;

    if (threadIdx.x == 0) {
        for (int i = 0; i < STAGES; ++i) {
            mbar_init(&s.full[i], 1);
            mbar_init(&s.empty[i], 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&s.tfull[i], 1);
            mbar_init(&s.tempty[i], 4);
        }
        mbar_init(&s.afull, 1);
        mbar_init(&s.aempty, 1);
        for (int i = 0; i < 8; ++i) mbar_init(&s.colbar[i], 1);
        s.abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         su32(&s.tmem_base)),
                     "r"(TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s.tmem_base;
    Pieces pc;
    pc.begin(w);
    int rb, i0, i1;

    if (warp == 0) {
        // ------------------------------------------------------------ producer
        if (lane == 0) {
            asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmA)) : "memory");
            asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmB)) : "memory");
            if constexpr (FORM != PLAIN) {
                asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmA2)) : "memory");
                asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmB2)) : "memory");
            }
            uint32_t iter = 0, aload = 0, tseq = 0;
            bool ok = true;
            while (ok && pc.next(w, rb, i0, i1)) {
                const int arow = rb * TC_M;
                if constexpr (FORM == RES) {
                    // the row block's A slices, once the MMA warp has released
                    // the previous block's
                    if (aload > 0 && !(ok = mbar_wait(&s.aempty, (aload - 1) & 1, abort))) break;
                    mbar_expect_tx(&s.afull, (uint32_t)nkb0 * A_BYTES + AUG_A_BYTES);
                    for (int kb = 0; kb < nkb0; ++kb) tma_load_2d(s.a[kb], &tmA, &s.afull, kb * TC_BK, arow);
                    tma_load_2d(s.a_aug, &tmA2, &s.afull, 0, arow);
                    ++aload;
                }
                // over all columns, the piece's tiles start where the other CTAs
                // are (the global count of tiles issued per CTA, modulo the piece)
                // and wrap around, so that CTAs that drift apart still read the
                // same B tiles from L2; what a row keeps does not depend on the
                // order.  Listed tiles come nearest first
                const int nt = i1 - i0;
                const int off = w.tiles ? 0
                                        : (int)((*(volatile unsigned long long*)a_in.sweep / (unsigned)gridDim.x) %
                                                (unsigned long long)nt);
                int t = tile_at(w, rb, i0 + off % nt);
                for (int i = 0; i < nt && ok; ++i) {
                    // the tile's column block for the epilogue (released by the arrival)
                    const uint32_t slot = tseq & 7u;
                    s.tcol[slot] = t;
                    mbar_arrive(&s.colbar[slot]);
                    ++tseq;
                    if ((tseq & 15u) == 0u) atomicAdd(a_in.sweep, 16ull);
                    const int bcol = t * TC_N;
                    t = tile_at(w, rb, i0 + (off + i + 1) % nt);   // the next one, ahead of its use
                    for (int kb = 0; kb < nkb; ++kb) {
                        const uint32_t st = iter % STAGES, use = iter / STAGES;
                        if (use > 0 && !(ok = mbar_wait(&s.empty[st], (use - 1) & 1, abort))) break;
                        if constexpr (FORM == RES) {
                            // the last slice with the tile's folded norms
                            const bool last = kb == nkb0 - 1;
                            mbar_expect_tx(&s.full[st], B_BYTES + (last ? AUG_B_BYTES : 0u));
                            tma_load_2d(s.b[st], &tmB, &s.full[st], kb * TC_BK, bcol);
                            if (last) tma_load_2d(aug_slot(s, nkb0, st, tseq - 1), &tmB2, &s.full[st], 16, bcol);
                        } else if (FORM == AUG && kb == nkb0) {
                            // the folded norms: 16 columns of A (x = 0) and B (x = 16)
                            mbar_expect_tx(&s.full[st], AUG_A_BYTES + AUG_B_BYTES);
                            tma_load_2d(s.a[st], &tmA2, &s.full[st], 0, arow);
                            tma_load_2d(s.b[st], &tmB2, &s.full[st], 16, bcol);
                        } else {
                            const CUtensorMap* ma = &tmA;
                            const CUtensorMap* mb = &tmB;
                            int kx = kb;
                            if constexpr (FORM == SPLIT) {
                                // passes h . h, h . l, l . h
                                const int part = kb / nkb0;
                                kx = kb - part * nkb0;
                                if (part == 2) ma = &tmA2;
                                if (part == 1) mb = &tmB2;
                            }
                            mbar_expect_tx(&s.full[st], A_BYTES + B_BYTES);
                            tma_load_2d(s.a[st], ma, &s.full[st], kx * TC_BK, arow);
                            tma_load_2d(s.b[st], mb, &s.full[st], kx * TC_BK, bcol);
                        }
                        ++iter;
                    }
                }
            }
            // drain: every issued load must have landed before the CTA leaves
            if (!ok || *abort) {
                const uint32_t first = iter > STAGES ? iter - STAGES : 0;
                for (uint32_t i = first; i < iter; ++i) {
                    const unsigned long long t0 = globaltimer_ns();
                    while (!mbar_test(&s.full[i % STAGES], (i / STAGES) & 1) &&
                           globaltimer_ns() - t0 < kWaitNs) {
                    }
                }
                if (aload > 0) {
                    const unsigned long long t0 = globaltimer_ns();
                    while (!mbar_test(&s.afull, (aload - 1) & 1) && globaltimer_ns() - t0 < kWaitNs) {
                    }
                }
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer
        if (lane == 0) {
            uint32_t iter = 0, tcount = 0, aload = 0;
            bool ok = true;
            while (ok && pc.next(w, rb, i0, i1)) {
                if constexpr (FORM == RES) {
                    // release the previous block once its MMAs complete, then
                    // wait for the new one
                    if (aload > 0) umma_commit(&s.aempty);
                    if (!(ok = mbar_wait(&s.afull, aload & 1, abort))) break;
                    tc_fence_after();
                    ++aload;
                }
                for (int i = i0; i < i1 && ok; ++i) {
                    const uint32_t acc = tcount & 1, use = tcount >> 1;
                    if (use > 0 && !(ok = mbar_wait(&s.tempty[acc], (use - 1) & 1, abort))) break;
                    tc_fence_after();
                    const uint32_t d_tmem = tmem + acc * TC_N;
                    for (int kb = 0; kb < nkb; ++kb) {
                        const uint32_t st = iter % STAGES;
                        if (!(ok = mbar_wait(&s.full[st], (iter / STAGES) & 1, abort))) break;
                        tc_fence_after();
                        if (FORM == AUG && kb == nkb0) {
                            // folded norms: one K = 16 step in 32-byte swizzle rows
                            umma(d_tmem, sw32_desc(su32(s.a[st])), sw32_desc(su32(s.b[st])), 1u);
                        } else {
                            const uint64_t da = sw128_desc(su32(s.a[FORM == RES ? kb : st]));
                            const uint64_t db = sw128_desc(su32(s.b[st]));
#pragma unroll
                            for (int k = 0; k < TC_BK / 16; ++k)   // 32-byte steps inside the swizzle row
                                umma(d_tmem, da + (uint64_t)(2 * k), db + (uint64_t)(2 * k),
                                     (kb | k) != 0 ? 1u : 0u);
                            if (FORM == RES && kb == nkb0 - 1)
                                umma(d_tmem, sw32_desc(su32(s.a_aug)),
                                     sw32_desc(su32(aug_slot(s, nkb0, st, tcount))), 1u);
                        }
                        umma_commit(&s.empty[st]);
                        ++iter;
                    }
                    if (!ok) break;
                    umma_commit(&s.tfull[acc]);
                    ++tcount;
                }
            }
            if (!ok || *abort) {
                // let the MMAs already issued finish before TMEM is released
                if (iter > 0) {
                    const uint32_t i = iter - 1;
                    const unsigned long long t0 = globaltimer_ns();
                    while (!mbar_test(&s.empty[i % STAGES], (i / STAGES) & 1) &&
                           globaltimer_ns() - t0 < kWaitNs) {
                    }
                }
            }
        }
    } else {
        // ------------------------------------------------------------ epilogue
        const int sub = warp & 3;
        const int r = sub * 32 + lane;
        const DevState* st = a_in.st;
        const CertConsts cc =
            FORM == SPLIT ? cert_make(a_in.gam, a_in.Dp, a_in.D, st->knn_max_norm_s_bits,
                                      st->knn_max_rho_s_bits, st->knn_max_kappa_s_bits)
                          : cert_make(a_in.gam, a_in.Dp, a_in.D, st->knn_max_norm_bits,
                                      st->knn_max_rho_bits, st->knn_max_kappa_bits);
        float* bd = &s.buf_d[0][r];
        int* bi = &s.buf_i[0][r];
        uint32_t tcount = 0;
        bool ok = true;
        const int stride = a_in.out.stride;
        while (ok && pc.next(w, rb, i0, i1)) {
            const int64_t row = (int64_t)rb * TC_M + r;
            const bool live = row < n_rows;
            const float np_ = live ? a_in.row_norms[row] : inf;
            const int self = FORM == SPLIT ? (live ? a_in.ids[row] : -1) : (int)row;
            const float sp = live ? sqrtf(np_) * cc.sn_infl : 0.f;
            const float rp = live ? a_in.rho[self] * 1.000001f : 0.f;
            RowState rs{0, inf, inf, inf};
            if (a_in.resume && live) {
                if (i0 == 0) {
                    const uint2* src = a_in.out.cand + row * stride;
                    const int n = sweep_count(src[0].x);
                    if (n < 0) rs.tcap = -inf;
                    else if (sweep_capped(src[0].x)) rs.tcap = __uint_as_float(src[1 + n].x);
                    for (int e = 0; e < n; ++e) {
                        const uint2 v = src[1 + e];
                        bd[e * TC_M] = __uint_as_float(v.x);
                        bi[e * TC_M] = (int)v.y;
                    }
                    rs.cnt = n < 0 ? 0 : n;
                }
                rs.dk = a_in.kth[row];   // from the earlier sweep
            }
            rs.thr = fminf(rs.tcap, cert_thr(cc, sp, rp, rs.dk));
            for (int i = i0; i < i1; ++i) {
                const uint32_t acc = tcount & 1, use = tcount >> 1;
                const uint32_t slot = tcount & 7u;
                ok = mbar_wait(&s.colbar[slot], (tcount >> 3) & 1u, abort);
                if (!__all_sync(0xffffffffu, ok)) { ok = false; break; }
                const int col0 = s.tcol[slot] * TC_N;
                ok = mbar_wait(&s.tfull[acc], use & 1, abort);
                if (!__all_sync(0xffffffffu, ok)) { ok = false; break; }
                tc_fence_after();
                const uint32_t tbase = tmem + ((uint32_t)(sub * 32) << 16) + acc * TC_N;
                const float* ncol_g = a_in.col_norms + col0;
                // one chunk of 32 columns against the row's threshold.  FOLD: the
                // accumulator holds -dt / 2, a column passes when it exceeds -thr / 2
                // (both scalings exact); otherwise w = fl(||xt_q||^2 - 2 dot) < thr -
                // ||xt_p||^2 rounded up whenever dt < thr, compared negated alike
                const bool own = FORM == SPLIT || (unsigned)((rb * TC_M) - col0) < (unsigned)TC_N;
                auto process = [&](const uint32_t (&rv)[CHUNK], int ch) {
                    float v[CHUNK];
                    if constexpr (FOLD) {
#pragma unroll
                        for (int j = 0; j < CHUNK; ++j) v[j] = __uint_as_float(rv[j]);
                    } else {
                        // column norms by uniform 16-byte loads (L1 hits after the
                        // first warp; padding columns hold +inf)
                        const float4* n4 = reinterpret_cast<const float4*>(ncol_g + ch * CHUNK);
#pragma unroll
                        for (int q = 0; q < CHUNK / 4; ++q) {
                            const float4 c4 = __ldg(n4 + q);
                            v[4 * q + 0] = fmaf(2.f, __uint_as_float(rv[4 * q + 0]), -c4.x);
                            v[4 * q + 1] = fmaf(2.f, __uint_as_float(rv[4 * q + 1]), -c4.y);
                            v[4 * q + 2] = fmaf(2.f, __uint_as_float(rv[4 * q + 2]), -c4.z);
                            v[4 * q + 3] = fmaf(2.f, __uint_as_float(rv[4 * q + 3]), -c4.w);
                        }
                    }
                    const int cb = col0 + ch * CHUNK;
                    if (own) {   // a row is not its own neighbour
#pragma unroll
                        for (int j = 0; j < CHUNK; ++j)
                            if (cb + j == self) v[j] = -inf;
                    }
                    float lim = FOLD ? -0.5f * rs.thr : -__fsub_ru(rs.thr, np_);
                    // votes narrow down to the groups of 8 columns in which some
                    // row has a hit (to groups of 4: 12 % slower)
                    float mg[CHUNK / GRP];
#pragma unroll
                    for (int q = 0; q < CHUNK / GRP; ++q) {
                        const float* t = v + GRP * q;
                        mg[q] = fmax3(fmax3(t[0], t[1], t[2]), fmax3(t[3], t[4], t[5]), fmaxf(t[6], t[7]));
                    }
                    const float mx = fmaxf(fmax3(mg[0], mg[1], mg[2]), mg[3]);
                    if (!__any_sync(0xffffffffu, mx > lim)) return;
#pragma unroll
                    for (int q = 0; q < CHUNK / GRP; ++q) {
                        if (!__any_sync(0xffffffffu, mg[q] > lim)) continue;
                        if (__any_sync(0xffffffffu, rs.cnt > SLOTS - GRP)) {
                            rs = refresh(bd, bi, rs, a_in.k, FULL, KEEP, false, cc, sp, rp);
                            lim = FOLD ? -0.5f * rs.thr : -__fsub_ru(rs.thr, np_);
                        }
#pragma unroll
                        for (int j = GRP * q; j < GRP * q + GRP; ++j) {
                            if (v[j] > lim) {
                                bd[rs.cnt * TC_M] = FOLD ? -2.f * v[j] : __fsub_rn(np_, v[j]);
                                bi[rs.cnt * TC_M] = cb + j;
                                ++rs.cnt;
                            }
                        }
                    }
                };
                auto release = [&]() {   // this warp's last TMEM read of the tile is done
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&s.tempty[acc]);
                };
                // the load of the next chunk is in flight while one is filtered
                uint32_t ra[CHUNK], rb2[CHUNK];
                tmem_ld32_issue(tbase, ra);
#pragma unroll 1
                for (int ch = 0; ch < TC_N / CHUNK; ch += 2) {
                    tmem_wait_regs(ra);
                    tmem_ld32_issue(tbase + (ch + 1) * CHUNK, rb2);
                    process(ra, ch);
                    tmem_wait_regs(rb2);
                    if (ch + 2 < TC_N / CHUNK) tmem_ld32_issue(tbase + (ch + 2) * CHUNK, ra);
                    else release();
                    process(rb2, ch + 1);
                }
                ++tcount;
            }
            if (!ok) break;
            // the piece's list
            const int64_t o = i0 == 0 ? row : (int64_t)(a_in.w.row_blocks + blockIdx.x) * TC_M + r;
            const int room = stride - 2;   // beside the header and a capped list's bound
            rs = refresh(bd, bi, rs, a_in.k, room, room, true, cc, sp, rp);
            const int n = rs.cnt;
            const bool fits = live && rs.tcap > -inf, capped = rs.tcap < cert_thr(cc, sp, rp, rs.dk);
            if (!a_in.resume && a_in.thr != nullptr) {
                a_in.thr[row] = rs.thr;
                a_in.kth[row] = rs.dk;
            }
            uint2* dst = a_in.out.cand + o * stride;
            dst[0] = make_uint2(fits ? sweep_header(n, capped) : kSweepOpen, __float_as_uint(rs.dk));
            if (fits) {
                for (int e = 0; e < n; ++e)
                    dst[1 + e] = make_uint2(__float_as_uint(bd[e * TC_M]), (unsigned)bi[e * TC_M]);
                if (capped) dst[1 + n] = make_uint2(__float_as_uint(rs.tcap), 0u);
            }
        }
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                     "r"(TMEM_COLS)
                     : "memory");
    }
    if (threadIdx.x == 0 && s.abort) atomicOr(a_in.err_flag, 2u);
}

CUresult encode_2d(EncodeTiledFn enc, CUtensorMap* m, const void* p, int64_t cols, int64_t rows,
                   int box_cols, int box_rows, CUtensorMapSwizzle sw) {
    const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)cols * 2};
    const cuuint32_t box[2] = {(cuuint32_t)box_cols, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(p), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, sw, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
}

template <int FORM>
slk_status launch_form(slk_ctx* ctx, const CUtensorMap (&m)[4], const SweepArgs& a) {
    auto kern = knn_sweep_kernel<FORM>;
    const size_t smem = sizeof(Smem<FORM>) + 1024;
    SLK_CUDA_TRY(ctx, cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    kern<<<(unsigned)a.w.units, THREADS, smem, ctx->stream>>>(m[0], m[1], m[2], m[3], a);
    SLK_LAUNCH_CHECK(ctx, "knn_sweep_kernel");
    return SLK_OK;
}

}  // namespace

slk_status knn_sweep_launch(slk_ctx* ctx, const SweepOperands& op, const SweepWork& w, int k,
                            double gam, const SweepLists& out, bool resume, float* thr, float* kth,
                            DevState* st) {
    const bool split = op.a_lo != nullptr;
    if (op.Dp % TC_BK != 0 || op.a_rows % TC_M != 0 || op.b_rows % TC_N != 0 || op.a_rows <= 0 ||
        out.stride < 2 || out.stride > kSweepStride || w.units < 1 || w.per < 1 || w.per > w.n_tiles)
        return set_err(ctx, SLK_ERR_INVALID_ARG, "bad sweep shape %lld / %lld x %d", (long long)op.a_rows,
                       (long long)op.b_rows, op.Dp);
    const void* ptrs[5] = {op.a_hi, op.a_lo, op.b_hi, op.b_lo, op.aug};
    for (const void* q : ptrs)
        if ((reinterpret_cast<uintptr_t>(q) & 15) != 0)
            return set_err(ctx, SLK_ERR_INVALID_ARG, "bf16 operand not 16-byte aligned");
    EncodeTiledFn enc = encode_fn();
    if (!enc) return set_err(ctx, SLK_ERR_CUDA, "cuTensorMapEncodeTiled is not available");
    CUtensorMap m[4];   // A, B, A2, B2
    CUresult rc[4];
    rc[0] = encode_2d(enc, &m[0], op.a_hi, op.Dp, op.a_rows, TC_BK, TC_M, CU_TENSOR_MAP_SWIZZLE_128B);
    rc[1] = encode_2d(enc, &m[1], op.b_hi, op.Dp, op.b_rows, TC_BK, TC_N, CU_TENSOR_MAP_SWIZZLE_128B);
    m[2] = m[0];
    m[3] = m[1];
    rc[2] = rc[3] = CUDA_SUCCESS;
    if (split) {
        rc[2] = encode_2d(enc, &m[2], op.a_lo, op.Dp, op.a_rows, TC_BK, TC_M, CU_TENSOR_MAP_SWIZZLE_128B);
        rc[3] = encode_2d(enc, &m[3], op.b_lo, op.Dp, op.b_rows, TC_BK, TC_N, CU_TENSOR_MAP_SWIZZLE_128B);
    } else if (op.aug) {
        rc[2] = encode_2d(enc, &m[2], op.aug, 32, op.a_rows, 16, TC_M, CU_TENSOR_MAP_SWIZZLE_32B);
        rc[3] = encode_2d(enc, &m[3], op.aug, 32, op.b_rows, 16, TC_N, CU_TENSOR_MAP_SWIZZLE_32B);
    }
    for (CUresult q : rc)
        if (q != CUDA_SUCCESS) return set_err(ctx, SLK_ERR_CUDA, "tensor map encoding failed (%d)", (int)q);
    SweepArgs a{};
    a.w = w;
    a.out = out;
    a.row_norms = op.row_norms;
    a.col_norms = op.col_norms;
    a.rho = op.rho;
    a.ids = op.ids;
    a.rows_dev = op.rows_dev;
    a.thr = thr;
    a.kth = kth;
    a.n_rows = op.N;
    a.D = op.D;
    a.Dp = op.Dp;
    a.k = k;
    a.resume = resume ? 1 : 0;
    a.gam = gam;
    a.st = st;
    a.err_flag = &st->knn_error;
    a.sweep = &st->knn_sweep;
    if (split) return launch_form<SPLIT>(ctx, m, a);
    if (!op.aug) return launch_form<PLAIN>(ctx, m, a);
    // a resident A block pays a pipeline drain per row block: only for sweeps
    // of some length
    if (op.Dp <= RES_MAX_DP && w.per >= 32) return launch_form<RES>(ctx, m, a);
    return launch_form<AUG>(ctx, m, a);
}
