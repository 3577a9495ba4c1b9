// Grouping of the points for the tensor-core sweep (knn_group.cu).
#pragma once

#include "knn_sweep.cuh"

constexpr int kPivots = 128;          // pivots at most
constexpr int kGrpSample = 4096;      // points the pivots are drawn from at most
constexpr int kGrpDims = 128;         // features the draw looks at

struct GroupBufs {
    float* xs;            // [sample][kGrpDims] sampled features
    float* mind2;         // [sample] squared distance to the nearest pivot so far
    int32_t* pick;        // [kPivots] sample position of each pivot
    unsigned* done;       // blocks finished
    __nv_bfloat16* pv;    // [kPivots][Dp] pivots (rows of the bfloat16 operand)
    float* pn2;           // [kPivots] squared norms
    float* pdist;         // [kPivots][kPivots] distances
    int32_t* chain;       // [kPivots] pivot at each place of the order
    int32_t* lab;         // [N] place of the nearest pivot
    int32_t* lab2;        // [N] of the second nearest, then lab in the order by lab2
    int32_t* perm2;       // [N] the points by lab2
    int32_t* counts;      // counting sort: [blocks][kPivots]
    int64_t* base;
    int64_t* off;         // [kPivots + 1]
    int32_t* perm;        // [N] point at each place of the sorted order
    float* thr;           // [Np] threshold of each row after the first pass
    float* kth;           // [Np] its k-th smallest dt
    float* sl;            // [Np / 128][kPivots] slack of a row block toward each pivot
    float* lo_t;          // [kPivots][Np / 128] depth of a column block behind each pivot's border
    int32_t* rep;         // [Np / 128] representative pivot (place) of a block
    int32_t* cnt;         // [row blocks] tiles of the second pass
    int64_t* start;       // [row blocks + 1]
    int32_t* max_cnt;
    uint16_t* tiles;      // [row blocks * n_tiles]
};

size_t group_carve(WsCarver& wc, GroupBufs& b, int64_t N, int64_t Np, int Dp, int n_tiles);
// Pivots, the nearest one of each point and the sorted order (perm).
slk_status group_order_launch(slk_ctx* ctx, const GroupBufs& b, const float* X, int64_t N, int D, int Dp,
                              const float* mu);
// The second pass's tiles from the first one's thresholds: those outside the
// window of `first` that may hold a column nearer than a row's threshold.
slk_status group_tiles_launch(slk_ctx* ctx, const GroupBufs& b, const __nv_bfloat16* xt, int64_t N,
                              int64_t Np, int Dp, const SweepWork& first);
// Stable counting sort (init_modes.cu): perm lists the points by label, off the
// first place of every label; counts and base hold ceil(N / 1024) rows of L.
slk_status label_sort_launch(slk_ctx* ctx, const int32_t* lab, int64_t N, int L, int32_t* counts,
                             int64_t* base, int64_t* off, int32_t* perm);
