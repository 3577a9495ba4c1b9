// Interface of the tensor-core candidate sweep (knn_sweep.cu).
#pragma once

#include <cuda_bf16.h>

#include "slk_internal.cuh"

constexpr int kSweepStride = 64;   // entries of a row list at most (a header, then candidates)
constexpr int kSweepMaxSeg = 16;   // lists a row block is cut into at most

constexpr unsigned kSweepOpen = 0xffffffffu;   // header of a row list that gave up

// Work of one sweep: for every 128-row block a sequence of 256-column tiles.
// The blocks' sequences laid end to end are cut into equal chunks, one per
// CTA, so a block's tiles may be shared by consecutive CTAs; each then writes
// a list of its own (slot rb for the block's first piece, slot row_cap / 128 + u
// for the piece that CTA u continues).
struct SweepWork {
    const uint16_t* tiles;    // column tiles of all blocks, or NULL: `per` tiles from tile0(rb)
    const int64_t* start;     // [blocks + 1] first tile of a block (with tiles)
    const int32_t* max_cnt;   // most tiles of a block (with tiles)
    int per, n_tiles;
    int aligned;              // whole row blocks per CTA (dealt out in turn, without tiles)
    int row_blocks;
    int units;                // CTAs
};

#ifdef __CUDACC__
namespace {

__device__ __forceinline__ unsigned sweep_header(int n, bool capped) {
    return (unsigned)n | (capped ? 0x100u : 0u);
}
__device__ __forceinline__ int sweep_count(unsigned h) { return h == kSweepOpen ? -1 : (int)(h & 0xffu); }
__device__ __forceinline__ bool sweep_capped(unsigned h) { return h != kSweepOpen && (h & 0x100u) != 0u; }

// Tiles per CTA: an equal share, but no row block in more than kSweepMaxSeg pieces.
__device__ __forceinline__ int64_t sweep_chunk(const SweepWork& w, int64_t total) {
    int64_t c = (total + w.units - 1) / w.units;
    const int64_t mc = w.tiles ? (int64_t)*w.max_cnt : (int64_t)w.per;
    const int64_t lo = (mc + kSweepMaxSeg - 2) / (kSweepMaxSeg - 1);
    if (c < lo) c = lo;
    if (w.aligned && !w.tiles) c = (c + w.per - 1) / w.per * w.per;
    return c < 1 ? 1 : c;
}
__device__ __forceinline__ int64_t sweep_total(const SweepWork& w) {
    return w.tiles ? w.start[w.row_blocks] : (int64_t)w.row_blocks * w.per;
}
__device__ __forceinline__ void sweep_block(const SweepWork& w, int rb, int64_t& s0, int64_t& s1) {
    if (w.tiles) {
        s0 = w.start[rb];
        s1 = w.start[rb + 1];
    } else {
        s0 = (int64_t)rb * w.per;
        s1 = s0 + w.per;
    }
}
// First column tile of a window of `per` tiles around the block's own columns.
__device__ __forceinline__ int sweep_tile0(const SweepWork& w, int rb) {
    int t = rb / 2 - w.per / 2;
    if (t > w.n_tiles - w.per) t = w.n_tiles - w.per;
    return t < 0 ? 0 : t;
}

}  // namespace
#endif

// Row lists: entry 0 of a row is (header, k-th smallest dt of the piece), then
// n (dt, column) pairs in no order: every column below the row's threshold.
// Where more lie under it than the list holds, the list is capped: the columns
// it leaves out have dt >= the bound in entry n + 1.  kSweepOpen: ties at the
// k-th place, nothing is listed.
struct SweepLists {
    uint2* cand;      // [slots * 128][stride]
    int stride;       // 2 .. kSweepStride
};

// Operands of a sweep.  Points: rows = columns = the Np points of xt (aug: the
// folded norms, or NULL).  Split: rows are the query rows qh + ql (two bfloat16
// terms; *rows_dev of them, ids[i] their points), columns xh + xl.
struct SweepOperands {
    const __nv_bfloat16* a_hi;
    const __nv_bfloat16* a_lo;    // split only
    const __nv_bfloat16* b_hi;
    const __nv_bfloat16* b_lo;    // split only
    const __nv_bfloat16* aug;     // points only
    const float* row_norms;       // +inf beyond the rows
    const float* col_norms;       // +inf beyond the columns
    const float* rho;             // by point
    const int32_t* ids;           // split: point of row i (the list the rows came from)
    const long long* rows_dev;    // split
    int64_t a_rows, b_rows;       // padded: multiples of 128 and 256
    int64_t N;                    // points
    int D, Dp;
};

// resume: the rows' lists (of an earlier sweep over other tiles) go on, from the
// k-th smallest dt in kth.  Otherwise thr and kth (nullable, by row) receive
// each row's threshold and k-th smallest dt; the work is then cut only between
// row blocks (aligned).
slk_status knn_sweep_launch(slk_ctx* ctx, const SweepOperands& op, const SweepWork& w, int k,
                            double gam, const SweepLists& out, bool resume, float* thr, float* kth,
                            DevState* st);
