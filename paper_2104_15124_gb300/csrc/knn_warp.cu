// Exact kNN for m <= 8: one warp per query pair (steps a2-a5 of the build).
//
// The tiled searches of knn.cu give each query one thread and a shared-memory heap: a warp then
// waits for its slowest lane at every insertion, and a cloud of n points offers only n threads.
// Here a warp owns a group of consecutive points of the spatial order (all in one 64-point tile)
// and takes them two at a time, its 32 lanes sharing every step:
//   threshold  a bound on the query's k-th distance is known before its scan starts.  The
//              first query of a group gets it from the k-th smallest distance in its own and the
//              neighbouring tiles; every later query q from its predecessor p, whose k-th distance
//              R is exact by then: R(q) <= R(p) + |p - q| is proven (the k nearest of p, with q
//              itself exchanged for p, lie that close), and 1.3 R(p)^2 is tried first, since
//              consecutive points have nearly the same radius.  A scan that finds fewer than k
//              candidates under its threshold is repeated at a larger one (a few per cent of the
//              queries).  With a radius guess (learned or given) the guess bounds the threshold too.
//   scan       the lanes test the boxes of 32 candidate tiles at once, then two candidates per lane of
//              every tile that passes; a candidate under the threshold goes to its lane's
//              own list in shared memory (a list shared by ballot and popcount took 4.1 against 3.6 ms on
//              the torus), with the candidates dealt to the lanes by a hash of the tile; a lane whose list
//              runs out has the lists cut at a tighter threshold, or the query scanned again with
//              another dealing.  The group's tiles come from one list, built once per group from
//              super-tile and tile boxes.  No heap, no barrier.
//   selection  the lists (about 1.4 k entries in all) are sorted by a register bitonic network on 32-bit
//              keys (FP32 distance cut to 24 bits, list slot in the low 8).
//   rescoring  the first ranks get their canonical FP64 distance, one candidate per lane, and are
//              put in exact (d2, index) order by odd-even transposition, which nearly always finds
//              them in order already; the certificate is the one of the tiled search: the
//              k-th FP64 distance lies below the smallest FP64 distance that a candidate left out can
//              have (the next key's bucket edge, or the threshold, less the FP32 error band).
// A query that cannot be settled (ties across the list's end, overflow) sends its 64-point tile to
// the tiled search with full keys; so does a large cloud in which queries reach most tiles (WS_REACH below).
//
// Bound: instruction issue and the latency of dependent steps (about 1,800 warp instructions per
// query, 24 warps per SM; the FP64 rescoring keeps the FP64 pipe 30 % busy).  Measured against the
// tiled FP32 search, identical lists: 1M torus points (m = 4, k = 64) 6.51 -> 3.11 ms, 50k sphere
// points 0.51 -> 0.17 ms, 2,000 circle points 0.150 -> 0.012 ms, 20,011 Gaussian points in R^8
// (k = 48) 3.97 -> 1.23 ms (there every tile overflowed the compact keys' visit table and was
// searched twice); the staged BF16 search with a learned radius took 7.08 ms on the torus.
#include "knn.cuh"

#include <algorithm>

namespace vb {

constexpr int WS_WARPS = 4;      // warps per CTA; groups of 16 points then fill it from one 64-point tile
constexpr int WS_LIST = 256;     // candidate tiles a group's list holds (beyond it the boxes are rescanned per pair)
constexpr int WS_MAX_G = 16;     // points per group at most

// Where a query reaches most of a large cloud, every pair of queries loads the whole cloud from L2, and the
// tiled search, which loads it once for 64 queries, is the faster one (100k Gaussian points in R^8, k = 48:
// 1,680 tiles a query, 20 against 12 ms; 300k points of Student's t, 2 degrees, in R^4, 47 against 40 ms; at about
// 750 they are level, in 2 to 8 dimensions).  So the groups of the first WS_SAMPLE blocks, which lie all over
// the cloud, count the tiles a query that their first three queries take, and once the mean of WS_REACH_MIN
// groups is above WS_REACH, the groups that have not finished leave their tiles to it (13.8 and 45 ms with what
// was begun; clouds that stay pay 0.8 % for the counting).
constexpr int WS_REACH = 750, WS_REACH_MIN = 256, WS_SAMPLE = 256;

// Every lane keeps its own list of the candidates it found: ROWS entries, entry r of lane l at
// [r][l].  About 1.4 k / 32 are used; a lane about to run out has the whole list cut (ws_tighten).
// NS: sorted ranks kept for the rescoring (k <= 32 KB).  SB: bits of a list slot (r * 32 + l) in a key.
template <int KB> struct WsCfg {
    static constexpr int ROWS = KB == 1 ? 8 : KB == 2 ? 12 : 16;
    static constexpr int NS = 64 * KB;
    static constexpr int SB = KB == 1 ? 8 : 9;
    static constexpr int SEEDS = KB <= 2 ? 3 : 4;   // tiles searched for the first query's threshold
    static constexpr size_t BYTES = 2 * ROWS * 32 * sizeof(uint2) + WS_LIST * 4 + NS * 4;   // per warp
};

// Keys order by distance: a non-negative FP32 number cut to its top 31 - (SB - 1) bits, list slot below.
template <int SB> __device__ __forceinline__ uint32_t ws_key(uint32_t dbits, uint32_t slot)
{
    return ((dbits << 1) & ~((1u << SB) - 1u)) | slot;
}
template <int SB> __device__ __forceinline__ float ws_lo(uint32_t key)
{
    return __uint_as_float((key & ~((1u << SB) - 1u)) >> 1);
}

// Sorts keys[0 .. cnt) (cnt <= 32 R) in place; the first ns ranks are written back.
template <int R>
__device__ __forceinline__ void ws_sort_keys(uint32_t* keys, int cnt, int ns, int lane)
{
    uint32_t key[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int e = r * 32 + lane;
        key[r] = e < cnt ? keys[e] : ~0u;
    }
    warp_sort<R>(key, lane);
    __syncwarp();
#pragma unroll
    for (int r = 0; r < R; ++r)
        if (lane * R + r < ns) keys[lane * R + r] = key[r];
}
__device__ __noinline__ void ws_sort_keys256(uint32_t* keys, int cnt, int ns, int lane)
{
    ws_sort_keys<8>(keys, cnt, ns, lane);
}

// Cuts the lanes' lists (`rows` entries in this lane, at least k in all) to the candidates that can
// still be among the k nearest: bisects the FP32 distance T with k or slightly more entries at or
// below it; the threshold that every candidate then has to meet is T times the FP32 error band, and the
// entries above it are dropped.  Returns the entries left in this lane and the threshold.
struct WsCut {
    int rows;
    float thr;
};
template <int ROWS>
__device__ __noinline__ WsCut ws_tighten(uint2* lst, int rows, int k, float band, int lane)
{
    uint32_t d[ROWS];
    uint32_t mx = 0;
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
        d[r] = r < rows ? lst[r * 32 + lane].x : 0xffffffffu;
        if (r < rows) mx = max(mx, d[r]);
    }
    k = min(k + 2, (int)__reduce_add_sync(0xffffffffu, rows));   // so that the k-th clears the threshold
    uint32_t hi = __reduce_max_sync(0xffffffffu, mx), lo = hi > (4u << 23) ? hi - (4u << 23) : 0u;
    bool low_checked = lo == 0;
    while (lo < hi) {
        const uint32_t mid = low_checked ? lo + (hi - lo) / 2 : lo;
        int c = 0;
#pragma unroll
        for (int r = 0; r < ROWS; ++r) c += d[r] <= mid;
        c = __reduce_add_sync(0xffffffffu, c);
        if (!low_checked) {
            low_checked = true;
            if (c >= k) { hi = lo; lo = 0; }
        } else if (c >= k) {
            hi = mid;
            if (c <= k + 6) break;
        } else {
            lo = mid + 1;
        }
    }
    WsCut c;
    c.rows = 0;
    c.thr = __fmul_ru(__uint_as_float(hi), band);
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
        if (d[r] <= __float_as_uint(c.thr)) {   // all that the threshold admits, so that it bounds what is dropped
            lst[c.rows * 32 + lane] = make_uint2(d[r], lst[r * 32 + lane].y);
            ++c.rows;
        }
    }
    return c;
}

// Ranks 0 .. 32 NB - 1, rank r * 32 + lane in register r, put in (d2, index) order.  Non-negative
// doubles order like their bits; empty ranks carry ~0.
template <int NB>
__device__ __forceinline__ void ws_exact_order(unsigned long long (&d)[NB], uint32_t (&o)[NB], int lane)
{
    for (;;) {
        bool bad = false;
#pragma unroll
        for (int r = 0; r < NB; ++r) {
            unsigned long long pd = __shfl_up_sync(0xffffffffu, d[r], 1);
            uint32_t po = __shfl_up_sync(0xffffffffu, o[r], 1);
            if (r > 0) {
                const unsigned long long ld = __shfl_sync(0xffffffffu, d[r > 0 ? r - 1 : 0], 31);
                const uint32_t lo = __shfl_sync(0xffffffffu, o[r > 0 ? r - 1 : 0], 31);
                if (lane == 0) { pd = ld; po = lo; }
            }
            if (r > 0 || lane > 0) bad |= d[r] < pd || (d[r] == pd && o[r] < po);
        }
        if (!__any_sync(0xffffffffu, bad)) return;
#pragma unroll
        for (int r = 0; r < NB; ++r) {   // pairs (0, 1), (2, 3), ...
            const unsigned long long pd = __shfl_xor_sync(0xffffffffu, d[r], 1);
            const uint32_t po = __shfl_xor_sync(0xffffffffu, o[r], 1);
            const bool less = pd < d[r] || (pd == d[r] && po < o[r]);
            const bool more = pd > d[r] || (pd == d[r] && po > o[r]);
            if ((lane & 1) ? more : less) { d[r] = pd; o[r] = po; }
        }
        unsigned long long pd[NB];   // pairs (1, 2), (3, 4), ..., across the registers at lanes 31 and 0
        uint32_t po[NB];
        const int src = ((lane & 1) ? lane + 1 : lane - 1) & 31;
#pragma unroll
        for (int r = 0; r < NB; ++r) {
            pd[r] = __shfl_sync(0xffffffffu, d[r], src);
            po[r] = __shfl_sync(0xffffffffu, o[r], src);
            const unsigned long long nd = __shfl_sync(0xffffffffu, d[r + 1 < NB ? r + 1 : r], 0);
            const uint32_t no = __shfl_sync(0xffffffffu, o[r + 1 < NB ? r + 1 : r], 0);
            const unsigned long long ld = __shfl_sync(0xffffffffu, d[r > 0 ? r - 1 : r], 31);
            const uint32_t lo = __shfl_sync(0xffffffffu, o[r > 0 ? r - 1 : r], 31);
            if (lane == 31) { pd[r] = nd; po[r] = no; }
            if (lane == 0) { pd[r] = ld; po[r] = lo; }
        }
#pragma unroll
        for (int r = 0; r < NB; ++r) {
            const bool has = !(lane == 0 && r == 0) && !(lane == 31 && r == NB - 1);
            const bool less = pd[r] < d[r] || (pd[r] == d[r] && po[r] < o[r]);
            const bool more = pd[r] > d[r] || (pd[r] == d[r] && po[r] > o[r]);
            if (has && ((lane & 1) ? less : more)) { d[r] = pd[r]; o[r] = po[r]; }
        }
    }
}

// FP32 squared distance to a candidate row, coordinates two by two; at most m + 2 roundings deep,
// the error the bands assume.
template <int MP, int MR>
__device__ __forceinline__ float ws_dist(const float2 (&nq)[MP / 2], const float4 (&v)[MP / 4])
{
    float2 d = __fadd2_rn(make_float2(v[0].x, v[0].y), nq[0]);
    float2 s = __fmul2_rn(d, d);
    if constexpr (MR > 2) {
        d = __fadd2_rn(make_float2(v[0].z, v[0].w), nq[1]);
        s = __ffma2_rn(d, d, s);
#pragma unroll
        for (int j = 1; j < MP / 4; ++j) {
            d = __fadd2_rn(make_float2(v[j].x, v[j].y), nq[2 * j]);
            s = __ffma2_rn(d, d, s);
            d = __fadd2_rn(make_float2(v[j].z, v[j].w), nq[2 * j + 1]);
            s = __ffma2_rn(d, d, s);
        }
    }
    return s.x + s.y;
}

// The canonical sum as its definition has it: squares rounded, then added (out of line, so that the
// fused form below is a branch and not a predicated copy of both).
__device__ __noinline__ double ws_square_sum(double acc, double d1, double d2, double d3)
{
    acc = __dadd_rn(acc, __dmul_rn(d1, d1));
    acc = __dadd_rn(acc, __dmul_rn(d2, d2));   // an absent coordinate adds zero
    return __dadd_rn(acc, __dmul_rn(d3, d3));
}

// Canonical FP64 squared distance of sorted points pu and pos (one pair per lane).
template <int MP, int MR>
__device__ __forceinline__ double ws_canon(const TileArgs& a, int pu, uint32_t pos)
{
    const double* q64 = a.xs64 + (int64_t)pu * MP;
    const double* c64 = a.xs64 + (int64_t)pos * MP;
    double acc;
    if constexpr (MP == 4) {
        double dl[4];
        unsigned low = 0;
#pragma unroll
        for (int j = 0; j < (MR + 1) / 2; ++j) {
            const double2 qv = *(const double2*)(q64 + 2 * j), cv = *(const double2*)(c64 + 2 * j);
            dl[2 * j] = __dsub_rn(qv.x, cv.x);
            low |= (unsigned)__double2loint(dl[2 * j]);
            if (2 * j + 1 < MR) {
                dl[2 * j + 1] = __dsub_rn(qv.y, cv.y);
                low |= (unsigned)__double2loint(dl[2 * j + 1]);
            }
        }
        acc = __dmul_rn(dl[0], dl[0]);
        // differences of at most 26 significant bits have exact squares: a fused multiply-add
        // then rounds like the canonical square and sum, in one operation of the narrow FP64
        // pipe instead of two
        if (__all_sync(0xffffffffu, (low & 0x07ffffffu) == 0)) {
#pragma unroll
            for (int j = 1; j < MR; ++j) acc = __fma_rn(dl[j], dl[j], acc);
        } else {
            acc = ws_square_sum(acc, dl[1], MR > 2 ? dl[2] : 0.0, MR > 3 ? dl[3] : 0.0);
        }
    } else {
        acc = 0.0;
#pragma unroll
        for (int j = 0; j < MP / 2; ++j) {
            if (2 * j >= a.m) break;
            const double2 qv = *(const double2*)(q64 + 2 * j), cv = *(const double2*)(c64 + 2 * j);
            const double dx = __dsub_rn(qv.x, cv.x), s = __dmul_rn(dx, dx);
            acc = j == 0 ? s : __dadd_rn(acc, s);
            if (2 * j + 1 < a.m) {
                const double dy = __dsub_rn(qv.y, cv.y);
                acc = __dadd_rn(acc, __dmul_rn(dy, dy));
            }
        }
    }
    return acc;
}

// A non-negative double, given by its bits, rounded up to FP32 on the integer pipe (to 2^-126 at
// least, +inf beyond the range).
__device__ __forceinline__ float ws_up(unsigned long long bits)
{
    const int e = (int)(bits >> 52) - 1023 + 127;
    if (e <= 0) return 1.1754944e-38f;
    if (e >= 255) return INFINITY;
    const uint32_t f = (uint32_t)(bits >> 29) & 0x7fffffu;
    return __uint_as_float((((uint32_t)e << 23) | f) + ((bits & 0x1fffffffull) ? 1u : 0u));
}

// Rescores the first 32 NB ranks of the sorted list (c entries, list bu), puts them in exact order,
// certifies and writes the row of sorted point pu; the k-th FP64 distance rounded up to FP32, or -1 when
// not certified.  The certificate is evaluated in FP32 with directed rounding: a handful of FP64
// operations per row would cost as much of the narrow FP64 pipe as a quarter of the rescoring.
template <int MP, int MR, int SB, int KB, int NB>
__device__ __forceinline__ float ws_row(const TileArgs& a, int pu, float th, int c, const uint2* bu,
                                         const uint32_t* srt, int lane)
{
    const int k = a.k, nres = min(min(c, a.L), 32 * NB);
    unsigned long long d[NB];
    uint32_t o[NB];
#pragma unroll
    for (int r = 0; r < NB; ++r) {
        const int rank = r * 32 + lane;
        const bool in = rank < nres;
        const uint32_t pos = in ? bu[srt[rank] & ((1u << SB) - 1u)].y : (uint32_t)pu;
        const unsigned long long bits = (unsigned long long)__double_as_longlong(ws_canon<MP, MR>(a, pu, pos));
        d[r] = in ? bits : ~0ull;
        o[r] = in ? a.perm[pos] : ~0u;
    }
    ws_exact_order<NB>(d, o, lane);
    unsigned long long v = d[0];
#pragma unroll
    for (int r = 1; r < KB; ++r)
        if (r == (k - 1) >> 5) v = d[r];
    const float dk = ws_up(__shfl_sync(0xffffffffu, v, (k - 1) & 31));
    // every candidate left out: a later rank of the list, or beyond the threshold
    const float B = c > nres ? ws_lo<SB>(srt[nres]) : th;
    // 2 (m + 2) 2^-24 relative, and the FP32 underflow of m terms
    const float lb = __fsub_rd(__fmul_rd(B, __fsub_rd(1.f, 1.1920930e-7f * (float)(a.m + 2))), (float)a.m * 1.1754944e-38f);
    if (!(isfinite(B) && dk < lb)) return -1.f;
    const int64_t row = (int64_t)a.perm[pu] * k;
#pragma unroll
    for (int r = 0; r < KB; ++r) {
        if (r * 32 + lane < k) {
            a.nbr[row + r * 32 + lane] = (int32_t)o[r];
            a.nbr_d2[row + r * 32 + lane] = __longlong_as_double((long long)d[r]);
        }
    }
    return dk;
}
// The same with 32 more ranks, for the few rows whose candidates at rank k and beyond lie within the
// FP32 error band of each other (out of line: the kernel is long).
template <int MP, int MR, int SB, int KB>
__device__ __noinline__ float ws_row_more(const TileArgs& a, int pu, float th, int c, const uint2* bu,
                                           const uint32_t* srt, int lane)
{
    return ws_row<MP, MR, SB, KB, KB + 1>(a, pu, th, c, bu, srt, lane);
}

// Appends (d, pos) at `at`, a lane's shared-memory address, when d <= thr and pos is not the query
// itself; predicated, without a branch.
__device__ __forceinline__ void ws_append(uint32_t& at, float d, float thr, uint32_t pos, uint32_t self)
{
    asm volatile(
        "{\n .reg .pred p;\n setp.le.f32 p, %1, %2;\n setp.ne.and.u32 p, %3, %4, p;\n"
        " @p st.shared.v2.b32 [%0], {%1, %3};\n @p add.u32 %0, %0, 256;\n}"
        : "+r"(at)
        : "f"(d), "f"(thr), "r"(pos), "r"(self)
        : "memory");
}

template <int MP, int MR, int KB>
__global__ void __launch_bounds__(WS_WARPS * 32, KB <= 2 && MP == 4 ? 6 : 4) knn_warp_kernel(const __grid_constant__ TileArgs a, int G,
                                                                                              unsigned sample)
{
    using Cfg = WsCfg<KB>;
    constexpr int ROWS = Cfg::ROWS, NS = Cfg::NS, SB = Cfg::SB;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ unsigned long long s_ev;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned below = (1u << lane) - 1u;
    uint2* buf = (uint2*)(smem + warp * Cfg::BYTES);   // [2][ROWS][32] candidates (distance bits, sorted position)
    uint32_t* list = (uint32_t*)(buf + 2 * ROWS * 32);  // the group's candidate tiles
    uint32_t* srt = list + WS_LIST;                     // the sorted keys of the query being finished
    // this lane's first entries
    const uint32_t base[2] = {(uint32_t)__cvta_generic_to_shared(buf + lane),
                              (uint32_t)__cvta_generic_to_shared(buf + ROWS * 32 + lane)};
    constexpr uint32_t FULL = (ROWS - 2) * 256;   // beyond it a tile's two candidates may not fit
    if (threadIdx.x == 0) s_ev = 0;
    __syncthreads();

    const int n = (int)a.n, k = a.k;
    // the first WS_SAMPLE blocks take every `sample`-th block of the cloud, the others what lies between (0: in order)
    unsigned blk = blockIdx.x;
    if (blk < sample * WS_SAMPLE)
        blk = blk < WS_SAMPLE ? blk * sample : blk - WS_SAMPLE + (blk - WS_SAMPLE) / (sample - 1u) + 1u;
    const int64_t g64 = ((int64_t)blk * WS_WARPS + warp) * G;
    unsigned tests = 0;   // candidate tiles x queries scanned
    if (g64 < n) {
        const int gp0 = (int)g64, gp1 = min(n, gp0 + G);
        const int own = gp0 / TILE;
        const bool rmode = a.r2 != nullptr;
        // do the groups counted so far say that the tiled search is the faster one?
        auto wide = [&]() {
            const int v = lane < 2 ? *(volatile int*)(a.reach + lane) : 0;
            const int c = __shfl_sync(0xffffffffu, v, 0);
            return c >= WS_REACH_MIN && __shfl_sync(0xffffffffu, v, 1) / c > WS_REACH;
        };
        bool dead = sample && wide();
        for (int s0 = gp0; s0 < gp1 && !dead;) {
            // the group's points of one cloud
            int qlo = 0, qhi = n;
            if (a.cl.B > 1) {
                const int b = cloud_id(a.cl, s0);
                qlo = (int)a.cl.ptr[b];
                qhi = (int)a.cl.ptr[b + 1];
            }
            const int s1 = min(gp1, qhi);
            const int ct_lo = qlo / TILE, ct_hi = (qhi + TILE - 1) / TILE;
            const int g_lo = ct_lo / TILE, g_hi = (ct_hi + TILE - 1) / TILE;

            float2 nq[2][MP / 2];            // the pair's coordinates, negated
            float thr[2] = {-1.f, -1.f};     // candidates at or below it are kept (-1: query not scanned)
            uint32_t at[2] = {base[0], base[1]};   // where this lane's lists go on
            int p[2] = {s0, s0};
            bool norelist = false;           // the group's tiles do not fit the list
            bool full = false;               // a list cannot hold its candidates
            const int whole_lo = (qlo + TILE - 1) / TILE, whole_hi = qhi / TILE;   // tiles wholly in the cloud

            auto load_query = [&](int u, int pu) {
                p[u] = pu;
                const float4* row = (const float4*)(a.xs + (int64_t)pu * MP);
#pragma unroll
                for (int j = 0; j < MP / 4; ++j) {
                    const float4 v = row[j];
                    nq[u][2 * j] = make_float2(-v.x, -v.y);
                    nq[u][2 * j + 1] = make_float2(-v.z, -v.w);
                }
            };
            auto nrows = [&](int u) { return (int)((at[u] - base[u]) >> 8); };
            uint32_t hash = 2654435769u;
            // this lane's candidates of tile ct: rotated by a hash of the tile, as a far query finds its
            // neighbours at the same end of many tiles, of those at the corners of the curve's cells
            auto first_of = [&](int ct) { return ct * TILE + (int)((lane + ((uint32_t)ct * hash >> 27)) & 31u); };
            auto load_tile = [&](int ct, float4 (&v)[2][MP / 4]) {
                const float4* row = (const float4*)(a.xs + (int64_t)first_of(ct) * MP);
#pragma unroll
                for (int j = 0; j < MP / 4; ++j) {
                    v[0][j] = row[j];
                    v[1][j] = row[32 * (MP / 4) + j];
                }
            };
            // cuts the list of query u
            auto tighten = [&](int u) {
                if ((int)__reduce_add_sync(0xffffffffu, nrows(u)) >= k) {
                    const WsCut c = ws_tighten<ROWS>(buf + u * ROWS * 32, nrows(u), k, a.band, lane);
                    at[u] = base[u] + c.rows * 256u;
                    thr[u] = fminf(thr[u], c.thr);
                }
                if (__any_sync(0xffffffffu, at[u] - base[u] > FULL)) {   // ties, or one lane's share too large
                    full = true;
                    at[u] = base[u];
                    thr[u] = -1.f;
                }
            };
            // folds the 64 candidates of tile ct into the lists of the queries under scan
            auto take_tile = [&](int ct, float4 (&v)[2][MP / 4], bool two) {
                const int c0 = first_of(ct), c1 = c0 + 32;
                if (ct < whole_lo || ct >= whole_hi) {   // points of other clouds, padding: no distance
                    if (c0 < qlo || c0 >= qhi) v[0][0].x = __uint_as_float(0x7fffffffu);
                    if (c1 < qlo || c1 >= qhi) v[1][0].x = __uint_as_float(0x7fffffffu);
                }
                ws_append(at[0], ws_dist<MP, MR>(nq[0], v[0]), thr[0], (uint32_t)c0, (uint32_t)p[0]);
                ws_append(at[0], ws_dist<MP, MR>(nq[0], v[1]), thr[0], (uint32_t)c1, (uint32_t)p[0]);
                ++tests;
                if (two) {
                    ws_append(at[1], ws_dist<MP, MR>(nq[1], v[0]), thr[1], (uint32_t)c0, (uint32_t)p[1]);
                    ws_append(at[1], ws_dist<MP, MR>(nq[1], v[1]), thr[1], (uint32_t)c1, (uint32_t)p[1]);
                    ++tests;
                }
                if (__any_sync(0xffffffffu, at[0] - base[0] > FULL || at[1] - base[1] > FULL)) {
                    tighten(0);
                    tighten(1);
                }
            };
            // does the box (lo, hi)[idx] reach under the threshold of a query under scan?
            auto reaches = [&](const float* lo, const float* hi, int idx) {
                const float4* l4 = (const float4*)(lo + (int64_t)idx * MP);
                const float4* h4 = (const float4*)(hi + (int64_t)idx * MP);
                float acc[2] = {0.f, 0.f};
#pragma unroll
                for (int j = 0; j < MP / 4; ++j) {
                    const float4 l = l4[j], h = h4[j];
                    const float lv[4] = {l.x, l.y, l.z, l.w}, hv[4] = {h.x, h.y, h.z, h.w};
#pragma unroll
                    for (int u = 0; u < 2; ++u) {
                        const float qv[4] = {nq[u][2 * j].x, nq[u][2 * j].y, nq[u][2 * j + 1].x, nq[u][2 * j + 1].y};
#pragma unroll
                        for (int r = 0; r < 4; ++r) {
                            if (4 * j + r >= MR) continue;
                            const float g = fmaxf(fmaxf(lv[r] + qv[r], -(hv[r] + qv[r])), 0.f);
                            acc[u] = fmaf(g, g, acc[u]);
                        }
                    }
                }
                return __fmul_rd(acc[0], a.lb_factor) <= thr[0] || __fmul_rd(acc[1], a.lb_factor) <= thr[1];
            };
            // takes the tiles ct of the lanes in m.  8-wide rows are loaded a tile ahead (1.40 -> 1.23 ms on
            // 20,011 points in R^8); 4-wide rows are not: the 16 registers cost a third of the warps per SM
            // (3.6 -> 3.0 ms on the torus of 1M points without them)
            auto take_masked = [&](unsigned m, int ct, bool two) {
                if (!m) return;
                int cur = __shfl_sync(0xffffffffu, ct, __ffs(m) - 1);
                if constexpr (MP > 4) {
                    float4 v[2][MP / 4], w[2][MP / 4];
                    load_tile(cur, v);
                    for (;;) {
                        m &= m - 1u;
                        int nxt = 0;
                        if (m) {
                            nxt = __shfl_sync(0xffffffffu, ct, __ffs(m) - 1);
                            load_tile(nxt, w);
                        }
                        take_tile(cur, v, two);
                        if (!m) break;
                        m &= m - 1u;
                        if (m) {
                            cur = __shfl_sync(0xffffffffu, ct, __ffs(m) - 1);
                            load_tile(cur, v);
                        }
                        take_tile(nxt, w, two);
                        if (!m) break;
                    }
                } else {
                    float4 v[2][MP / 4];
                    for (;;) {
                        load_tile(cur, v);
                        take_tile(cur, v, two);
                        m &= m - 1u;
                        if (!m) break;
                        cur = __shfl_sync(0xffffffffu, ct, __ffs(m) - 1);
                    }
                }
            };
            int nlist = -1;   // tiles in the group's list (-1: none, scan the boxes)
            float rl2 = INFINITY;   // the list holds every tile that close to the group's box (squared): no
                                    // threshold under scan is above it while there is a list
            auto scan = [&](bool two) {
                // 32 tiles per step: the next of the list, or half of the next super-tile in reach
                unsigned ms = 0;
                int nx = nlist >= 0 ? 0 : g_lo, half = 0, t0 = 0;
                for (;;) {
                    int ct;
                    if (nlist >= 0) {
                        if (nx >= nlist) break;
                        ct = nx + lane < nlist ? (int)list[nx + lane] : -1;
                        nx += 32;
                    } else {
                        if (half == 0) {
                            while (!ms && nx < g_hi) {
                                const bool in = nx + lane < g_hi;
                                ms = __ballot_sync(0xffffffffu, in && reaches(a.slo, a.shi, in ? nx + lane : g_lo));
                                t0 = nx;
                                nx += 32;
                            }
                            if (!ms) break;
                        }
                        ct = (t0 + __ffs(ms) - 1) * TILE + 32 * half + lane;
                        if (half) ms &= ms - 1u;
                        half ^= 1;
                        if (ct < ct_lo || ct >= ct_hi) ct = -1;
                    }
                    take_masked(__ballot_sync(0xffffffffu, ct >= 0 && reaches(a.tlo, a.thi, max(ct, 0))), ct, two);
                }
            };
            // sorts, rescores, certifies and writes the row of the query at sorted position pu; the k-th
            // FP64 distance, or -1 when the row is not settled
            auto finish = [&](int pu, float th, int nrow, uint2* bu) -> float {
                int c = __reduce_add_sync(0xffffffffu, nrow);
                if (c > 64 * KB) {
                    const WsCut cut = ws_tighten<ROWS>(bu, nrow, k, a.band, lane);
                    nrow = cut.rows;
                    th = fminf(th, cut.thr);
                    c = __reduce_add_sync(0xffffffffu, nrow);
                    if (c > 64 * KB) return -1.f;
                }
                int place = nrow;   // of this lane's keys among all lanes'
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int y = __shfl_up_sync(0xffffffffu, place, o);
                    if (lane >= o) place += y;
                }
                place -= nrow;
                for (int r = 0; __any_sync(0xffffffffu, r < nrow); ++r)
                    if (r < nrow) srt[place + r] = ws_key<SB>(bu[r * 32 + lane].x, (uint32_t)(r * 32 + lane));
                __syncwarp();
                if (c <= 64) ws_sort_keys<2>(srt, c, NS, lane);
                else if (KB == 4 && c > 128) ws_sort_keys256(srt, c, NS, lane);
                else if constexpr (KB > 1) ws_sort_keys<4>(srt, c, NS, lane);
                __syncwarp();
                const float dk = ws_row<MP, MR, SB, KB, KB>(a, pu, th, c, bu, srt, lane);
                if (dk >= 0.f || min(c, a.L) <= 32 * KB) return dk;
                return ws_row_more<MP, MR, SB, KB>(a, pu, th, c, bu, srt, lane);
            };

            // the predecessors whose k-th distance is known, for the next queries' bounds
            int pp[2] = {-1, -1};
            float pr[2] = {0.f, 0.f};   // their k-th distances, rounded up
            float pd = 0.f;             // the squared k-th distance of the last one

            // scans and finishes the queries p[u] of `todo`; pmax[u]: proven bound on the squared k-th
            // distance, guess: threshold tried first.  False: the tile goes to the tiled search.
            auto settle = [&](int todo, const float (&pmax)[2], float guess) -> bool {
                float r2q[2] = {INFINITY, INFINITY}, tmax[2];
                int level[2] = {0, 0};
                bool redo[2] = {false, false};
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    if (rmode && (todo >> u & 1)) r2q[u] = __fmul_ru(a.r2[p[u]], a.r2_scale);
                    tmax[u] = fminf(pmax[u], r2q[u]);
                    thr[u] = (todo >> u & 1) ? fminf(fminf(guess, tmax[u]), rl2) : -1.f;
                }
                int np = 0, tries = 0;
                while (todo) {
                    const float tried[2] = {thr[0], thr[1]};
                    at[0] = base[0];
                    at[1] = base[1];
                    scan(todo != 1);
                    if (full) {
                        // one lane's list ran out (a few rows in a million): once more with the candidates dealt
                        // to other lanes; ties fill every lane's
                        if (tries++ == 2) return false;
                        hash = hash * 747796405u + 2891336452u | 1u;
                        full = false;
#pragma unroll
                        for (int u = 0; u < 2; ++u) thr[u] = (todo >> u & 1) ? tried[u] : -1.f;
                        continue;
                    }
                    __syncwarp();
                    int got = 0;
#pragma unroll 1
                    for (int u = 0; u < 2; ++u) {
                        if (!(todo >> u & 1)) continue;
                        const int nr = u ? nrows(1) : nrows(0);
                        if ((int)__reduce_add_sync(0xffffffffu, nr) < k) continue;
                        const int pu = u ? p[1] : p[0];
                        const float dk = finish(pu, u ? thr[1] : thr[0], nr, buf + u * ROWS * 32);
                        __syncwarp();   // the sorted keys and the lists are written again
                        if (dk < 0.f) continue;
                        got |= 1 << u;
                        pd = dk;
                        const float r = __fsqrt_ru(pd);
                        if (np) { pp[1] = pu; pr[1] = r; }
                        else { pp[0] = pu; pr[0] = r; pp[1] = -1; }
                        np = 1;
                    }
                    todo &= ~got;
#pragma unroll
                    for (int u = 0; u < 2; ++u) {
                        if (!(todo >> u & 1)) {
                            thr[u] = -1.f;
                            continue;
                        }
                        // fewer than k candidates, or the k-th too close to the threshold: a larger one
                        if (tried[u] < tmax[u]) {
                            thr[u] = level[u] == 0 ? fminf(1.7f * tried[u], tmax[u]) : tmax[u];
                            ++level[u];
                            continue;
                        }
                        if (redo[u] || !(r2q[u] <= pmax[u])) return false;
                        redo[u] = true;   // the radius guess does not settle the row: once more at twice the radius
                        if (lane == 0) {
                            atomicAdd(&a.rep->knn_rows_short, 1ull);
                            if (atomicExch(&a.fail_flag[a.ntiles + own], 1) == 0) atomicAdd(&a.rep->knn_redo_tiles, 1ull);
                        }
                        tmax[u] = fminf(pmax[u], 4.f * r2q[u]);
                        thr[u] = tmax[u];
                    }
                    if (!(fmaxf(thr[0], thr[1]) <= rl2)) nlist = -1;   // beyond the list's reach
                }
                return true;
            };
            // proven bound of a query from the predecessors, squared
            auto bound = [&](int u) {
                float best = INFINITY;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    if (pp[h] < 0) continue;
                    const float4* row = (const float4*)(a.xs + (int64_t)pp[h] * MP);
                    float4 v[MP / 4];
#pragma unroll
                    for (int j = 0; j < MP / 4; ++j) v[j] = row[j];
                    const float r = __fadd_ru(pr[h], __fsqrt_ru(__fmul_ru(ws_dist<MP, MR>(nq[u], v), 1.00001f)));
                    best = fminf(best, __fmul_ru(__fmul_ru(r, r), 1.00001f));
                }
                return best;
            };

            for (int i = s0; i < s1 && !dead;) {
                int todo = 1;
                float pm[2] = {INFINITY, INFINITY};
                load_query(0, i);
                if (i == s0) {
                    // ---- the first query: the k-th distance within its own and the neighbouring tiles
                    load_query(1, i);
                    if (!rmode) {
                        thr[0] = INFINITY;
                        at[0] = base[0];
                        at[1] = base[1];
                        int done = 0;
                        for (int h = 0; h < 2 * (ct_hi - ct_lo) && !full; ++h) {
                            if (done >= Cfg::SEEDS && (int)__reduce_add_sync(0xffffffffu, nrows(0)) >= k) break;
                            const int ct = (h & 1) ? own + ((h + 1) >> 1) : own - (h >> 1);
                            if (ct < ct_lo || ct >= ct_hi) continue;
                            float4 v[2][MP / 4];
                            load_tile(ct, v);
                            take_tile(ct, v, false);
                            ++done;
                        }
                        if (full || (int)__reduce_add_sync(0xffffffffu, nrows(0)) < k) { dead = true; break; }
                        pm[0] = ws_tighten<ROWS>(buf, nrows(0), k, a.band, lane).thr;
                    }
                } else {
                    // ---- the others, two at a time
                    const bool two = i + 1 < s1;
                    load_query(1, two ? i + 1 : i);
                    pm[0] = bound(0);
                    pm[1] = bound(1);
                    if (two) todo = 3;
                }
                // ---- the group's candidate tiles: boxes within the queries' bound + the reach of the rest of the group.
                // A later query with a larger bound (a radius guess proves nothing about its neighbours') starts at the
                // list's reach; if it needs more, the boxes are scanned and the next pair makes a new list.
                if (nlist < 0 && !norelist && s1 - i > 3) {
                    const bool mine = lane < s1 - i;
                    float4 v[MP / 4];
                    const float4* row = (const float4*)(a.xs + (int64_t)(i + (mine ? lane : 0)) * MP);
#pragma unroll
                    for (int j = 0; j < MP / 4; ++j) v[j] = row[j];
                    float reach = ws_dist<MP, MR>(nq[0], v);
                    float blo[MR], bhi[MR];
#pragma unroll
                    for (int r = 0; r < MR; ++r) {
                        const float4 w = v[r / 4];
                        blo[r] = bhi[r] = r % 4 == 0 ? w.x : r % 4 == 1 ? w.y : r % 4 == 2 ? w.z : w.w;
                    }
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) {
                        reach = fmaxf(reach, __shfl_xor_sync(0xffffffffu, reach, o));
#pragma unroll
                        for (int r = 0; r < MR; ++r) {
                            blo[r] = fminf(blo[r], __shfl_xor_sync(0xffffffffu, blo[r], o));
                            bhi[r] = fmaxf(bhi[r], __shfl_xor_sync(0xffffffffu, bhi[r], o));
                        }
                    }
                    // the larger of the thresholds that the queries at hand may start with: guesses differ
                    float base = fminf(pm[0], rmode ? __fmul_ru(a.r2[i], a.r2_scale) : INFINITY);
                    if (todo == 3)
                        base = fmaxf(base, fminf(pm[1], rmode ? __fmul_ru(a.r2[i + 1], a.r2_scale) : INFINITY));
                    const float rl = __fadd_ru(__fsqrt_ru(base), __fsqrt_ru(__fmul_ru(reach, 1.00001f)));
                    const float near2 = __fmul_ru(__fmul_ru(rl, rl), 1.00001f);
                    auto near = [&](const float* lo, const float* hi, int idx) {
                        const float4* l4 = (const float4*)(lo + (int64_t)idx * MP);
                        const float4* h4 = (const float4*)(hi + (int64_t)idx * MP);
                        float acc = 0.f;
#pragma unroll
                        for (int j = 0; j < MP / 4; ++j) {
                            const float4 l = l4[j], h = h4[j];
                            const float lv[4] = {l.x, l.y, l.z, l.w}, hv[4] = {h.x, h.y, h.z, h.w};
#pragma unroll
                            for (int r = 0; r < 4; ++r) {
                                if (4 * j + r >= MR) continue;
                                const int q = 4 * j + r < MR ? 4 * j + r : 0;
                                const float g = fmaxf(fmaxf(lv[r] - bhi[q], blo[q] - hv[r]), 0.f);
                                acc = fmaf(g, g, acc);
                            }
                        }
                        return __fmul_rd(acc, a.lb_factor) <= near2;
                    };
                    int nl = 0;
                    for (int g0 = g_lo; g0 < g_hi && nl <= WS_LIST; g0 += 32) {
                        unsigned ms = __ballot_sync(0xffffffffu, g0 + lane < g_hi && near(a.slo, a.shi, min(g0 + lane, g_hi - 1)));
                        while (ms && nl <= WS_LIST) {
                            const int t0 = (g0 + __ffs(ms) - 1) * TILE;
                            ms &= ms - 1u;
#pragma unroll 1
                            for (int h = 0; h < 2; ++h) {
                                const int ct = t0 + 32 * h + lane;
                                const bool in = ct >= ct_lo && ct < ct_hi;
                                const unsigned b = __ballot_sync(0xffffffffu, in && near(a.tlo, a.thi, in ? ct : ct_lo));
                                const int to = nl + __popc(b & below);
                                if ((b >> lane & 1u) && to < WS_LIST) list[to] = (uint32_t)ct;
                                nl += __popc(b);
                            }
                        }
                    }
                    if (nl <= WS_LIST) { nlist = nl; rl2 = near2; }
                    else norelist = true;
                    __syncwarp();
                }
                dead = !settle(todo, pm, i == s0 ? INFINITY : 1.3f * pd);
                if (nlist < 0) rl2 = INFINITY;
                i += todo == 3 ? 2 : 1;
                if (sample && tests > (unsigned)(WS_REACH * (i - s0)) && wide()) dead = true;
                if (i - s0 == 3 && blockIdx.x < WS_SAMPLE && sample && lane < 2)
                    atomicAdd(a.reach + lane, lane == 0 ? 1 : (int)min(tests / 3, 65535u));
            }
            s0 = s1;
        }
        if (dead && lane == 0 && atomicExch(&a.fail_flag[own], 1) == 0) {
            a.fail_list[atomicAdd(a.fail_count, 1)] = own;
            atomicAdd(&a.rep->knn_retry_tiles, 1ull);
        }
    }
    if (lane == 0 && tests) atomicAdd(&s_ev, (unsigned long long)tests * TILE);
    __syncthreads();
    if (threadIdx.x == 0 && s_ev) atomicAdd(&a.rep->knn_candidates, s_ev);
}

template <int MP, int MR, int KB>
static vb_status launch_ws(const TileArgs& a, cudaStream_t s)
{
    constexpr size_t sm = WS_WARPS * WsCfg<KB>::BYTES;
    static bool attr_set[16] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    if (!attr_set[dev & 15]) {
        if (cudaFuncSetAttribute(knn_warp_kernel<MP, MR, KB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm) !=
            cudaSuccess)
            return VB_ERR_CUDA;
        attr_set[dev & 15] = true;
    }
    // points per warp: as many as leave the grid 32 warps for every SM, of which 24 are resident (16 with 8-wide rows
    // or k > 64).  A longer group shares its first query's seeds and the tile list among more queries; a short
    // cloud needs the warps.
    int G = 1;
    while (G < WS_MAX_G && a.n / (2 * G) >= 152 * 32) G *= 2;
    const int64_t groups = (a.n + G - 1) / G;
    const int64_t blocks = (groups + WS_WARPS - 1) / WS_WARPS;
    // a cloud in which a query can reach that many tiles (a batch by its mean cloud)
    const bool large = a.n / a.cl.B > (int64_t)WS_REACH * TILE && blocks >= 2 * WS_SAMPLE;
    const unsigned sample = large ? (unsigned)(blocks / WS_SAMPLE) : 0u;
    knn_warp_kernel<MP, MR, KB><<<(unsigned)blocks, WS_WARPS * 32, sm, s>>>(a, G, sample);
    return last_launch();
}

template <int MP, int MR>
static vb_status launch_ws_k(const TileArgs& a, cudaStream_t s)
{
    if (a.k <= 32) return launch_ws<MP, MR, 1>(a, s);
    if (a.k <= 64) return launch_ws<MP, MR, 2>(a, s);
    return launch_ws<MP, MR, 4>(a, s);
}

// k <= 128: four ranks per lane, and lists of at most 256 entries.
bool warp_search_takes(int mp, const vb_knn_params* p)
{
    return mp <= 8 && p->k <= 128 && p->prune != VB_PRUNE_NONE && p->heap_keys != VB_KEYS_FULL;
}

vb_status launch_warp_search(const TileArgs& a, int mp, cudaStream_t s)
{
    if (mp == 8) return launch_ws_k<8, 8>(a, s);
    if (a.m <= 2) return launch_ws_k<4, 2>(a, s);
    if (a.m == 3) return launch_ws_k<4, 3>(a, s);
    return launch_ws_k<4, 4>(a, s);
}

}  // namespace vb
