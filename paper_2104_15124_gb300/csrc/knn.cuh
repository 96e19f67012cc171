// Declarations shared by the kNN search kernels (knn.cu, knn_warp.cu).
#pragma once
#include "vb_internal.cuh"

namespace vb {

constexpr int TILE = 64;            // points per query tile and per candidate tile

// The same for a query held in registers (q[0..MP)) and a 16-byte aligned candidate row.
template <int MP>
__device__ __forceinline__ double canon_d2_q64(const double* q, const double* __restrict__ c, int m)
{
    double cv[MP];
#pragma unroll
    for (int r2 = 0; r2 < MP / 2; ++r2) {
        const double2 v = *(const double2*)(c + 2 * r2);
        cv[2 * r2] = v.x;
        cv[2 * r2 + 1] = v.y;
    }
    double acc = 0.0;
#pragma unroll
    for (int r = 0; r < MP; ++r) {
        if (r < m) {
            const double dl = __dsub_rn(q[r], cv[r]);
            const double sq = __dmul_rn(dl, dl);
            acc = r == 0 ? sq : __dadd_rn(acc, sq);
        }
    }
    return acc;
}

struct TileArgs {
    const float* xs;
    const double* xs64;   // FP64 copies of xs (exact), for the FP64 rescoring
    const float* tlo;
    const float* thi;
    const float* slo;     // boxes of super-tiles (64 consecutive tiles; FP32 search)
    const float* shi;
    const uint32_t* perm;
    int64_t n;
    int64_t ntiles;
    int m, k, L, prune, nseed;
    float lb_factor;     // 1 - 4 (m + 2) 2^-24, applied rounding down
    float band;          // 1 + 4 (m + 2) 2^-24: FP32 distances closer than this may swap in FP64
    double cert_factor;  // 1 - 2 (m + 2) 2^-24
    int32_t* nbr;
    double* nbr_d2;
    int* fb_list;
    int* fb_count;
    int* work;           // next query tile (persistent grid)
    const int* tile_list;   // optional list of query tiles to process (else all tiles)
    const int* tile_count;  // its length (device)
    const float* r2;        // radius search: per sorted point, squared radius bound
    float r2_scale;         // radius search: factor on r2 for this pass
    int count_retries;      // radius search: count the tiles this pass hands on (last pass only)
    int cap;                // radius search: candidates kept per query
    int* fail_flag;         // radius search: per query tile, set once it joins fail_list
    int* fail_list;
    int* fail_count;
    int* reach;             // warp search: groups counted, tiles a query summed over them
    Clouds cl;              // batched build: queries only take candidates from their own cloud
    DevReport* rep;
    // pipelined 16-bit search
    const unsigned char* blk;   // tile blocks (operand image + norms), tcp_blk_bytes(kp) each
    int kp;                     // K: m padded to 16
    int stages;                 // ring slots of staged tile blocks
    uint32_t* lbw;              // per CTA scratch: ntiles box bounds
    uint64_t* tlist;            // per CTA scratch: ntiles (bound, tile) keys in bound order
    uint4* lbs;                 // per CTA scratch: ntiles bounds of the four 32-query groups
    const float* trad;          // per tile: radius of its ball about the box centre (pipelined search)
    uint64_t* hdump;            // pipelined search: heaps handed to its row finish ([L][128] per query tile)
    float* dbg_d2;              // diagnostic: kept 16-bit distances per row ([n][L], original order)
    int32_t* dbg_idx;           // their original indices
};

template <int MP>
__device__ __forceinline__ float point_box_lb(const float* q, const float* lo, const float* hi)
{
    float acc = 0.f;
#pragma unroll
    for (int r = 0; r < MP; ++r) {
        float g = fmaxf(fmaxf(lo[r] - q[r], q[r] - hi[r]), 0.f);
        acc = fmaf(g, g, acc);
    }
    return acc;
}

// The warp search (knn_warp.cu) of every query tile; VB_ERR_UNSUPPORTED when it does not take the request.
bool warp_search_takes(int mp, const vb_knn_params* p);
vb_status launch_warp_search(const TileArgs& a, int mp, cudaStream_t s);

}  // namespace vb
