// Symmetric sparsity pattern (step a6) and the bandwidth function (step a8).
//
// a6: E = {(i, i)} U {(i, j): j in N_k(i) or i in N_k(j)} as CSR with rows
//     sorted by column.  Algorithm 1 keeps the diagonal (its inner loop
//     starts at j = i) and sets K^ij and K^ji together, so every kNN pair
//     enters in both directions.  The FP32 squared distance of every entry is
//     the FP32 rounding of the canonical FP64 value, identical for (i, j) and
//     (j, i).  Construction below (sorted own lists, filtered reverse entries,
//     merge by rank).
// a8: b_i^2 = sum_{r=1}^{k_bw} d2(i, I(i, r)) in rank order, FP64 (Eq.
//     bandwidth parameter).
#include "vb_internal.cuh"

#include <algorithm>

namespace vb {

constexpr int BIG_CAP = 8192;       // block path: reverse entries per row
constexpr int SCAN_T = 1024;
constexpr int SCAN_ITEMS = 8;       // counts per thread per scan block

// ------------------------------------------------------------------ exclusive scan int32 -> int64[n+1]
size_t scan_ws_bytes(int64_t n)
{
    int64_t nb = (n + SCAN_T * SCAN_ITEMS - 1) / (SCAN_T * SCAN_ITEMS);
    return (size_t)(nb + 1) * sizeof(int64_t) + 256;
}

__device__ __forceinline__ int64_t block_excl_scan(int64_t v, int64_t* sh, int64_t* total)
{
    // 1024 threads: warp inclusive scans, then a scan of the 32 warp totals
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    int64_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int64_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) sh[w] = x;
    __syncthreads();
    if (w == 0) {
        int64_t s = sh[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int64_t y = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += y;
        }
        sh[lane] = s;
    }
    __syncthreads();
    int64_t r = x - v + (w ? sh[w - 1] : 0);
    if (total) *total = sh[31];
    __syncthreads();
    return r;
}

__global__ void __launch_bounds__(SCAN_T) scan_reduce_kernel(const int32_t* __restrict__ c, int64_t n, int add, int64_t* bsum)
{
    __shared__ int64_t sh[32];
    int64_t base = (int64_t)blockIdx.x * SCAN_T * SCAN_ITEMS;
    int64_t s = 0;
    for (int i = 0; i < SCAN_ITEMS; ++i) {
        int64_t e = base + (int64_t)i * SCAN_T + threadIdx.x;
        if (e < n) s += c[e] + add;
    }
    int64_t tot;
    block_excl_scan(s, sh, &tot);
    if (threadIdx.x == 0) bsum[blockIdx.x] = tot;
}

__global__ void __launch_bounds__(SCAN_T) scan_top_kernel(int64_t* bsum, int64_t nb)
{
    __shared__ int64_t sh[32];
    __shared__ int64_t carry;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    for (int64_t b0 = 0; b0 < nb; b0 += SCAN_T) {
        int64_t i = b0 + threadIdx.x;
        int64_t v = i < nb ? bsum[i] : 0;
        int64_t tot;
        int64_t ex = block_excl_scan(v, sh, &tot);
        if (i < nb) bsum[i] = carry + ex;
        __syncthreads();
        if (threadIdx.x == 0) carry += tot;
        __syncthreads();
    }
    if (threadIdx.x == 0) bsum[nb] = carry;
}

__global__ void __launch_bounds__(SCAN_T) scan_apply_kernel(const int32_t* __restrict__ c, int64_t n, int add,
                                                           const int64_t* __restrict__ bsum, int64_t nb, int64_t* out)
{
    __shared__ int64_t sh[32];
    // each thread owns SCAN_ITEMS consecutive counts of the block's chunk
    int64_t base = (int64_t)blockIdx.x * SCAN_T * SCAN_ITEMS + (int64_t)threadIdx.x * SCAN_ITEMS;
    int32_t v[SCAN_ITEMS];
    int64_t s = 0;
#pragma unroll
    for (int i = 0; i < SCAN_ITEMS; ++i) {
        v[i] = base + i < n ? c[base + i] + add : 0;
        s += v[i];
    }
    int64_t run = bsum[blockIdx.x] + block_excl_scan(s, sh, nullptr);
#pragma unroll
    for (int i = 0; i < SCAN_ITEMS; ++i) {
        if (base + i < n) out[base + i] = run;
        run += v[i];
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) out[n] = bsum[nb];
}

vb_status scan_counts(cudaStream_t s, const int32_t* counts, int64_t n, int64_t* out, void* ws, int add)
{
    int64_t nb = (n + SCAN_T * SCAN_ITEMS - 1) / (SCAN_T * SCAN_ITEMS);
    int64_t* bsum = (int64_t*)ws;
    scan_reduce_kernel<<<(unsigned)nb, SCAN_T, 0, s>>>(counts, n, add, bsum);
    scan_top_kernel<<<1, SCAN_T, 0, s>>>(bsum, nb);
    scan_apply_kernel<<<(unsigned)nb, SCAN_T, 0, s>>>(counts, n, add, bsum, nb, out);
    return last_launch();
}

// ------------------------------------------------------------------ a6
// Row j of E is the disjoint union of {j}, its own kNN list N(j), and the reverse
// entries R(j) = {i : j in N(i), i not in N(j)}.  Construction: every kNN list is
// sorted by column (one warp per row); a reverse candidate (i -> j) is kept unless i is
// in N(j), which for exact lists ordered by (d2, index) holds exactly when
// (d2(i, j), i) <= (d2 and index of j's k-th neighbour), one 16-byte load instead of a
// search, so mutual pairs enter once; the counts
// 1 + k + |R(j)| give row_ptr directly (one scan).  A kept reverse entry goes straight into one of
// row j's RBUCKET slots as it is counted; what overflows them is listed (and marked in the sorted list, for
// when the list overflows too) and scattered behind row_ptr in a second pass.  Finally one warp per row sorts
// R(j) and places every entry by its rank (own index + reverse entries below it + the diagonal),
// which merges the three sorted sets with no duplicates left to remove.
constexpr int RCAP = 256;           // warp path: reverse entries per row held in shared memory
constexpr int OWN_CAP = 256;        // longest kNN list (k + margin <= 256)
// Reverse entries a row takes without the second pass.  Clouds in many dimensions have hubs: 100k points in R^16,
// k = 64 and 128, take 0.42 and 1.12 ms with 32, 0.38 and 1.02 ms with 64 (without buckets 0.36 and 0.99 ms, but
// 1.49 against 1.04 ms on 1M torus points, whose rows have few reverse entries).
constexpr int RBUCKET = 64;
constexpr int RSMALL = 32;          // reverse entries that a warp merges without sorting them
constexpr int OVER_CAP = 1 << 16;   // entries beyond the buckets that are listed (more: every list is scanned)

struct Kth {
    double d2;         // j's k-th neighbour distance and index
    int32_t idx, pad;
};

struct GraphWs {
    Kth* kth;          // n
    int32_t* own_col;  // n k: kNN lists sorted by column
    float* own_d2;     // n k
    int32_t* rcnt;     // n reverse entries per row
    int32_t* fill;     // n scatter cursors of the entries beyond RBUCKET
    int2* bucket;      // n RBUCKET reverse entries (row, distance bits)
    int32_t* rev_col;  // n k: those beyond RBUCKET, entry e of row j at row_ptr[j] - j (1 + k) + e
    float* rev_d2;     // n k
    int32_t* big;      // n rows for the block path
    int32_t* nbig;     // rows for the block path
    unsigned long long* nover;   // entries beyond RBUCKET (n k of them at most: they can pass 2^32)
    int4* over;        // OVER_CAP of those: (i, j, distance bits, -)
    void* scan;        // scan_ws_bytes(n)
};

static size_t graph_plan(Carve& c, int64_t n, int32_t k, GraphWs* w)
{
    GraphWs t;
    t.kth = c.take<Kth>(n);
    t.own_col = c.take<int32_t>(n * (int64_t)k);
    t.own_d2 = c.take<float>(n * (int64_t)k);
    t.rcnt = c.take<int32_t>(n);
    t.fill = c.take<int32_t>(n);
    t.bucket = c.take<int2>(n * RBUCKET);
    t.rev_col = c.take<int32_t>(n * (int64_t)k);
    t.rev_d2 = c.take<float>(n * (int64_t)k);
    t.big = c.take<int32_t>(n);
    t.nbig = c.take<int32_t>(1);
    t.nover = c.take<unsigned long long>(1);
    t.over = c.take<int4>(OVER_CAP);
    t.scan = c.take<char>(scan_ws_bytes(n));
    if (w) *w = t;
    return c.off;
}
size_t graph_plan_bytes(int64_t n, int32_t k)
{
    Carve c(nullptr);
    return graph_plan(c, n, k, nullptr);
}

// bitonic sort of P (power of two) 64-bit keys in shared memory by `nthr` threads
__device__ __forceinline__ void bitonic_smem(uint64_t* a, int P, int tid, int nthr, bool warp_only)
{
    for (int size = 2; size <= P; size <<= 1) {
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            for (int i = tid; i < P / 2; i += nthr) {
                int lo = 2 * i - (i & (stride - 1));
                int hi = lo + stride;
                bool up = (lo & size) == 0;
                uint64_t x = a[lo], y = a[hi];
                if ((x > y) == up) { a[lo] = y; a[hi] = x; }
            }
            if (warp_only) __syncwarp(); else __syncthreads();
        }
    }
}

// Number of entries of the ascending list a[0..len) below v.
__device__ __forceinline__ int lower_bound_i32(const int32_t* a, int len, int32_t v)
{
    int lo = 0, hi = len;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (a[mid] < v) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}
__device__ __forceinline__ int lower_bound_key(const uint64_t* a, int len, int32_t v)
{
    int lo = 0, hi = len;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if ((int32_t)(a[mid] >> 32) < v) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

constexpr int SORT_WARPS = 4;

// Clears the counters, and the k-th pair (distance, index) of every list, 16 bytes per point: the table the mutual
// test below reads at random stays in L2, where the lists themselves (12 k bytes per point)
// do not.
__global__ void kth_kernel(const int32_t* __restrict__ nbr, const double* __restrict__ nbr_d2, int64_t n, int k,
                           Kth* kth, int32_t* rcnt, int32_t* fill, int32_t* nbig, unsigned long long* nover)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i == 0) {
        *nbig = 0;
        *nover = 0;
    }
    if (i >= n) return;
    rcnt[i] = 0;
    fill[i] = 0;
    Kth q;
    q.d2 = nbr_d2[i * k + k - 1];
    q.idx = nbr[i * k + k - 1];
    q.pad = 0;
    kth[i] = q;
}

// Own kNN lists sorted by column, one warp per row; the FP32 value of each entry is the
// rounding of its canonical FP64 distance (identical for (i, j) and (j, i)).  The same pass finds, for
// every point j, the lists that name j without j naming their owner (the reverse entries of row j):
// (i -> j) is mutual exactly when (d2(i, j), i) does not exceed the k-th pair of j's own list
// (kth[j]).  A non-mutual entry is counted and put into row j's bucket in one atomic; beyond
// RBUCKET it is listed and carries the sign bit in own_d2 (distances are >= 0) for the second pass.  (Marking
// all of them and scattering in a pass over every entry took 0.48 ms more at 1M torus points, k = 64.)
// SORT: the list is sorted as 32-bit keys column << (5 + log2 KL) | position (columns distinct, so the order is
// the columns' order) by a bitonic network across the warp, for k <= 32 KL <= 128 and columns that fit;
// else an entry's place is the number of columns below its own: every column is broadcast to the warp
// once and each lane counts for the KL entries it holds.
__device__ __forceinline__ float own_entry(int64_t i, int32_t j, double d, int k, const Kth* __restrict__ kth,
                                           int32_t* rcnt, int2* bucket, unsigned long long* nover, int4* over)
{
    const Kth q = kth[j];
    const float f = (float)d;
    if (d < q.d2 || (d == q.d2 && (int32_t)i <= q.idx)) return f;
    const int slot = atomicAdd(&rcnt[j], 1);
    if (slot < RBUCKET) {
        bucket[(int64_t)j * RBUCKET + slot] = make_int2((int32_t)i, __float_as_int(f));
        return f;
    }
    const unsigned long long at = atomicAdd(nover, 1ull);
    if (at < OVER_CAP) over[at] = make_int4((int32_t)i, j, __float_as_int(f), 0);
    return -f;
}

template <int KL, bool SORT>
__global__ void __launch_bounds__(SORT_WARPS * 32) own_sort_kernel(const int32_t* __restrict__ nbr,
                                                                    const double* __restrict__ nbr_d2, int64_t n,
                                                                    int k, int32_t* own_col, float* own_d2,
                                                                    const Kth* __restrict__ kth, int32_t* rcnt,
                                                                    int2* bucket, unsigned long long* nover, int4* over)
{
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int64_t i = (int64_t)blockIdx.x * SORT_WARPS + w; i < n; i += (int64_t)gridDim.x * SORT_WARPS) {
        const int32_t* row = nbr + i * k;
        if constexpr (SORT) {
            constexpr int PB = KL == 1 ? 5 : KL == 2 ? 6 : 7;
            uint32_t key[KL];
#pragma unroll
            for (int s = 0; s < KL; ++s) {
                const int e = lane + 32 * s;
                key[s] = e < k ? ((uint32_t)row[e] << PB) | (uint32_t)e : 0xffffffffu;
            }
            warp_sort<KL>(key, lane);
#pragma unroll
            for (int s = 0; s < KL; ++s) {
                const int pos = lane * KL + s;   // the key's place in the sorted list
                if (pos < k) {
                    const int32_t j = (int32_t)(key[s] >> PB);
                    const double d = nbr_d2[i * k + (key[s] & ((1u << PB) - 1u))];
                    own_col[i * k + pos] = j;
                    own_d2[i * k + pos] = own_entry(i, j, d, k, kth, rcnt, bucket, nover, over);
                }
            }
        } else {
            int32_t c[KL];
            int rank[KL];
#pragma unroll
            for (int s = 0; s < KL; ++s) {
                const int e = lane + 32 * s;
                c[s] = e < k ? row[e] : INT32_MAX;
                rank[s] = 0;
            }
#pragma unroll
            for (int s2 = 0; s2 < KL; ++s2) {
                const int32_t v = c[s2];
                const int lim = min(32, k - 32 * s2);
                for (int l = 0; l < lim; ++l) {
                    const int32_t cb = __shfl_sync(0xffffffffu, v, l);
#pragma unroll
                    for (int s = 0; s < KL; ++s) rank[s] += cb < c[s] ? 1 : 0;
                }
            }
#pragma unroll
            for (int s = 0; s < KL; ++s) {
                const int e = lane + 32 * s;
                if (e < k) {
                    own_col[i * k + rank[s]] = c[s];
                    own_d2[i * k + rank[s]] = own_entry(i, c[s], nbr_d2[i * k + e], k, kth, rcnt, bucket, nover, over);
                }
            }
        }
    }
}

// The entries (i -> j) beyond row j's bucket, from the list, or all with the sign bit set in own_d2,
// scattered behind row_ptr.
__global__ void reverse_kernel(const int32_t* __restrict__ own_col, const float* __restrict__ own_d2, int64_t n, int k,
                               const int64_t* __restrict__ row_ptr, int32_t* fill, int32_t* rev_col, float* rev_d2,
                               const unsigned long long* __restrict__ nover, const int4* __restrict__ over)
{
    const unsigned long long no = *nover;
    if (no == 0) return;
    if (no <= OVER_CAP) {
        for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < (int)no; e += gridDim.x * blockDim.x) {
            const int4 v = over[e];
            const int64_t off = row_ptr[v.y] - (int64_t)v.y * (1 + k) + RBUCKET + atomicAdd(&fill[v.y], 1);
            rev_col[off] = v.x;
            rev_d2[off] = __int_as_float(v.z);
        }
        return;
    }
    const int lane = threadIdx.x & 31;
    const int64_t step = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t i = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; i < n; i += step) {   // a warp per list
        for (int e = lane; e < k; e += 32) {
            const float d = own_d2[i * k + e];
            if (!signbit(d)) continue;
            const int32_t j = own_col[i * k + e];
            const int slot = RBUCKET + atomicAdd(&fill[j], 1);
            const int64_t off = row_ptr[j] - (int64_t)j * (1 + k) + slot;
            rev_col[off] = (int32_t)i;
            rev_d2[off] = -d;
        }
    }
}

// Row j: sort R(j) in shared memory, then write every entry at its rank.
// oc_s: shared-memory room for the row's own columns (k ints), or nullptr to search them in
// global memory (the block path).
__device__ void merge_row(int64_t j, int k, int r, uint64_t* rb, const int64_t* __restrict__ row_ptr,
                          const int32_t* __restrict__ own_col, const float* __restrict__ own_d2,
                          const int2* __restrict__ bucket, const int32_t* __restrict__ rev_col,
                          const float* __restrict__ rev_d2, int32_t* col, float* ed2, int tid, int nthr,
                          bool warp_only, int32_t* oc_s = nullptr)
{
    int P = 32;
    while (P < r) P <<= 1;
    const int64_t roff = row_ptr[j] - j * (1 + k);
    for (int e = tid; e < P; e += nthr) {
        if (e < min(r, RBUCKET)) {
            const int2 v = bucket[j * RBUCKET + e];
            rb[e] = ((uint64_t)(uint32_t)v.x << 32) | (uint32_t)v.y;
        } else {
            rb[e] = e < r ? ((uint64_t)(uint32_t)rev_col[roff + e] << 32) | __float_as_uint(rev_d2[roff + e]) : ~0ull;
        }
    }
    const int32_t* oc = own_col + j * k;
    if (oc_s) {   // the own columns, searched once per reverse entry, from shared memory
        for (int e = tid; e < k; e += nthr) oc_s[e] = oc[e];
        oc = oc_s;
    }
    if (warp_only) __syncwarp(); else __syncthreads();
    if (r > 1) bitonic_smem(rb, P, tid, nthr, warp_only);
    const int64_t ob = row_ptr[j];
    const float* od = own_d2 + j * k;
    for (int a = tid; a < k; a += nthr) {
        const int32_t c = oc[a];   // (own_col + j k)[a]
        const int rank = a + lower_bound_key(rb, r, c) + ((int32_t)j < c ? 1 : 0);
        col[ob + rank] = c;
        ed2[ob + rank] = fabsf(od[a]);   // without the non-mutual mark
    }
    for (int b = tid; b < r; b += nthr) {
        const int32_t c = (int32_t)(rb[b] >> 32);
        const int rank = b + lower_bound_i32(oc, k, c) + ((int32_t)j < c ? 1 : 0);
        col[ob + rank] = c;
        ed2[ob + rank] = __uint_as_float((uint32_t)rb[b]);
    }
    if (tid == 0) {
        const int rank = lower_bound_i32(oc, k, (int32_t)j) + lower_bound_key(rb, r, (int32_t)j);
        col[ob + rank] = (int32_t)j;
        ed2[ob + rank] = 0.f;
    }
}

// The same for a row with at most 32 reverse entries (nearly every row), one per lane, without
// sorting them: every reverse column is broadcast to the warp once, and each lane counts the
// reverse columns below its own reverse entry (its rank among them; the columns of R(j) are
// distinct) and below each of its own-list entries; a reverse entry's place among the own
// entries is a binary search of the sorted own columns in shared memory.
template <int OWN_PER_LANE>   // own-list entries per lane: k <= 32 OWN_PER_LANE
__device__ void merge_row_small(int64_t j, int k, int r, const int64_t* __restrict__ row_ptr,
                                const int32_t* __restrict__ own_col, const float* __restrict__ own_d2,
                                const int2* __restrict__ bucket, int32_t* col, float* ed2, int lane, int32_t* oc_s)
{
    int32_t rc = INT32_MAX;
    float rd = 0.f;
    if (lane < r) {
        const int2 v = bucket[j * RBUCKET + lane];
        rc = v.x;
        rd = __int_as_float(v.y);
    }
    const int32_t* oc = own_col + j * k;
    int32_t c[OWN_PER_LANE];
    int below[OWN_PER_LANE];
#pragma unroll
    for (int s = 0; s < OWN_PER_LANE; ++s) {
        const int a = lane + 32 * s;
        c[s] = a < k ? oc[a] : INT32_MAX;
        below[s] = 0;
        if (a < k) oc_s[a] = c[s];
    }
    int rrank = 0;
    for (int b = 0; b < r; ++b) {
        const int32_t cb = __shfl_sync(0xffffffffu, rc, b);
        rrank += cb < rc ? 1 : 0;
#pragma unroll
        for (int s = 0; s < OWN_PER_LANE; ++s) below[s] += cb < c[s] ? 1 : 0;
    }
    const int rev_below_j = __popc(__ballot_sync(0xffffffffu, lane < r && rc < (int32_t)j));
    __syncwarp();   // the own columns in shared memory, for the searches below
    const int64_t ob = row_ptr[j];
    const float* od = own_d2 + j * k;
#pragma unroll
    for (int s = 0; s < OWN_PER_LANE; ++s) {
        const int a = lane + 32 * s;
        if (a < k) {
            const int rank = a + below[s] + ((int32_t)j < c[s] ? 1 : 0);
            col[ob + rank] = c[s];
            ed2[ob + rank] = fabsf(od[a]);   // without the non-mutual mark
        }
    }
    if (lane < r) {
        const int rank = rrank + lower_bound_i32(oc_s, k, rc) + ((int32_t)j < rc ? 1 : 0);
        col[ob + rank] = rc;
        ed2[ob + rank] = rd;
    }
    if (lane == 0) {
        const int rank = lower_bound_i32(oc_s, k, (int32_t)j) + rev_below_j;
        col[ob + rank] = (int32_t)j;
        ed2[ob + rank] = 0.f;
    }
}

template <int KL>   // own-list entries per lane, k <= 32 KL
__global__ void __launch_bounds__(SORT_WARPS * 32) merge_kernel(const int64_t* __restrict__ row_ptr, int64_t n, int k,
                                                                 const int32_t* __restrict__ own_col,
                                                                 const float* __restrict__ own_d2,
                                                                 const int2* __restrict__ bucket,
                                                                 const int32_t* __restrict__ rev_col,
                                                                 const float* __restrict__ rev_d2, int32_t* col,
                                                                 float* ed2, int64_t cap, int32_t* big, int32_t* nbig,
                                                                 int64_t* nnz_dev, DevReport* rep)
{
    __shared__ uint64_t buf[SORT_WARPS][RCAP];
    __shared__ int32_t ocs[SORT_WARPS][OWN_CAP];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        *nnz_dev = row_ptr[n];
        if (row_ptr[n] > cap) report_error(rep, VB_ERR_BOUNDS);
    }
    if (row_ptr[n] > cap) return;
    for (int64_t j = (int64_t)blockIdx.x * SORT_WARPS + w; j < n; j += (int64_t)gridDim.x * SORT_WARPS) {
        const int r = (int)(row_ptr[j + 1] - row_ptr[j]) - 1 - k;
        if (r > RCAP) {
            if (lane == 0) {
                big[atomicAdd(nbig, 1)] = (int32_t)j;
                atomicAdd(&rep->union_big_rows, 1ull);
            }
            continue;
        }
        if (r <= RSMALL)
            merge_row_small<KL>(j, k, r, row_ptr, own_col, own_d2, bucket, col, ed2, lane, ocs[w]);
        else
            merge_row(j, k, r, buf[w], row_ptr, own_col, own_d2, bucket, rev_col, rev_d2, col, ed2, lane, 32, true, ocs[w]);
        __syncwarp();
    }
}

__global__ void __launch_bounds__(1024) big_merge_kernel(const int64_t* __restrict__ row_ptr, int64_t n, int k,
                                                        const int32_t* __restrict__ own_col,
                                                        const float* __restrict__ own_d2,
                                                        const int2* __restrict__ bucket,
                                                        const int32_t* __restrict__ rev_col,
                                                        const float* __restrict__ rev_d2, int32_t* col, float* ed2,
                                                        int64_t cap, const int32_t* __restrict__ big,
                                                        const int32_t* __restrict__ nbig, DevReport* rep)
{
    extern __shared__ uint64_t bbuf[];
    if (row_ptr[n] > cap) return;
    const int nb = *nbig;
    for (int f = blockIdx.x; f < nb; f += gridDim.x) {
        const int64_t j = big[f];
        const int r = (int)(row_ptr[j + 1] - row_ptr[j]) - 1 - k;
        if (r > BIG_CAP) {   // a hub point in more than BIG_CAP other lists
            if (threadIdx.x == 0) report_error(rep, VB_ERR_UNSUPPORTED);
            continue;
        }
        merge_row(j, k, r, bbuf, row_ptr, own_col, own_d2, bucket, rev_col, rev_d2, col, ed2, threadIdx.x, blockDim.x, false);
        __syncthreads();
    }
}

vb_status graph_run(Ctx* ctx, int64_t n, int32_t k, const int32_t* nbr, const double* nbr_d2, int64_t* row_ptr,
                    int32_t* col, float* ed2, int64_t cap, int64_t* nnz_dev, void* ws, size_t ws_bytes)
{
    if (n < 2 || k < 1 || k > n - 1 || k > OWN_CAP || !nbr || !nbr_d2 || !row_ptr || !col || !ed2 || !nnz_dev)
        return VB_ERR_ARG;
    if (cap < n * (2 * (int64_t)k + 1)) return VB_ERR_ARG;
    GraphWs w;
    Carve c(ws);
    size_t need = graph_plan(c, n, k, &w);
    if (!ws || ws_bytes < need) return VB_ERR_WORKSPACE;
    cudaStream_t s = ctx->stream;
    mark(ctx, VB_STAGE_GRAPH, 0);
    kth_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(nbr, nbr_d2, n, k, w.kth, w.rcnt, w.fill, w.nbig, w.nover);
    // sorted by keys of a column and a position while those fit 32 bits, else ranked by counting
    const int pb = k <= 32 ? 5 : k <= 64 ? 6 : 7;
    const bool keys = k <= 128 && n <= (int64_t)1 << (32 - pb);
#define VB_OWN(KL, SORT)                                                                                            \
    own_sort_kernel<KL, SORT><<<152 * 16, SORT_WARPS * 32, 0, s>>>(nbr, nbr_d2, n, k, w.own_col, w.own_d2, w.kth,     \
                                                                w.rcnt, w.bucket, w.nover, w.over)
    if (k <= 32) {
        if (keys) VB_OWN(1, true); else VB_OWN(1, false);
    } else if (k <= 64) {
        if (keys) VB_OWN(2, true); else VB_OWN(2, false);
    } else if (k <= 128) {
        if (keys) VB_OWN(4, true); else VB_OWN(4, false);
    } else {
        VB_OWN(8, false);
    }
#undef VB_OWN
    vb_status st = scan_counts(s, w.rcnt, n, row_ptr, w.scan, 1 + k);
    if (st != VB_OK) return st;
    reverse_kernel<<<152 * 8, 256, 0, s>>>(w.own_col, w.own_d2, n, k, row_ptr, w.fill, w.rev_col, w.rev_d2, w.nover, w.over);
#define VB_MERGE(KL)                                                                                                 \
    merge_kernel<KL><<<152 * 16, SORT_WARPS * 32, 0, s>>>(row_ptr, n, k, w.own_col, w.own_d2, w.bucket, w.rev_col,      \
                                                         w.rev_d2, col, ed2, cap, w.big, w.nbig, nnz_dev, ctx->rep)
    if (k <= 32) VB_MERGE(1);
    else if (k <= 64) VB_MERGE(2);
    else if (k <= 128) VB_MERGE(4);
    else VB_MERGE(OWN_CAP / 32);
#undef VB_MERGE
    static bool big_attr[16] = {};
    int dev = ctx->device & 15;
    if (!big_attr[dev]) {
        if (cudaFuncSetAttribute(big_merge_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, BIG_CAP * 8) !=
            cudaSuccess)
            return VB_ERR_CUDA;
        big_attr[dev] = true;
    }
    big_merge_kernel<<<152, 1024, BIG_CAP * 8, s>>>(row_ptr, n, k, w.own_col, w.own_d2, w.bucket, w.rev_col, w.rev_d2, col, ed2,
                                                    cap, w.big, w.nbig, ctx->rep);
    mark(ctx, VB_STAGE_GRAPH, 1);
    ctx->launches += 8;
    return last_launch();
}

// ------------------------------------------------------------------ a8
// One thread per row, the rows' distances staged through shared memory 16 at a time, so that the loads are
// whole 128-byte lines (a thread reading its own row directly touches one line per load: 0.22 ms for
// 1M rows of 64); the sums stay in rank order.  A chunk's loads fly while the one before is summed: a whole
// build of 2,000 points 202.7 -> 197.3 us, of 50k 576 -> 560 us, of 1M 7.19 -> 7.16 ms (each k <= 64).  Blocks of
// 64 rows, so that 20,000 points fill the chip (k = 200: 25 us with 128 rows, 21 us with a thread reading its row,
// 19 us so; 100k, k = 32: 15 -> 13 us).  Bound by the narrow FP64 pipe (n k additions, 0.11 ms at 1M) and by the
// length of its chain in small clouds.
constexpr int BW_T = 64, BW_C = 16, BW_R = BW_T / BW_C;   // a chunk: BW_T rows by BW_C columns, BW_C loads a thread
__global__ void __launch_bounds__(BW_T) bandwidth_kernel(const double* __restrict__ nbr_d2, int64_t n, int k, int k_bw,
                                                         double* b, float* ib, DevReport* rep)
{
    __shared__ double sh[BW_T][BW_C + 1];
    const int t = threadIdx.x;
    const int64_t r0 = (int64_t)blockIdx.x * BW_T;
    const int nr = (int)min((int64_t)BW_T, n - r0);
    const int c = t % BW_C, rt = t / BW_C;   // the thread's column of a chunk and its first row
    const double* src = nbr_d2 + (r0 + rt) * k + c;
    double v[BW_C] = {}, s = 0.0;
    auto load = [&](int c0) {
#pragma unroll
        for (int u = 0; u < BW_C; ++u)
            if (rt + u * BW_R < nr && c0 + c < k_bw) v[u] = src[(int64_t)u * BW_R * k + c0];
    };
    load(0);
    for (int c0 = 0; c0 < k_bw; c0 += BW_C) {
        const int nc = min(BW_C, k_bw - c0);
#pragma unroll
        for (int u = 0; u < BW_C; ++u) sh[rt + u * BW_R][c] = v[u];
        __syncthreads();
        load(c0 + BW_C);
        if (t < nr)
            for (int e = 0; e < nc; ++e) s = c0 + e == 0 ? sh[t][e] : __dadd_rn(s, sh[t][e]);
        __syncthreads();
    }
    if (t >= nr) return;
    const double bw = sqrt(s);
    b[r0 + t] = bw;
    if (ib) ib[r0 + t] = (float)(1.0 / bw);
    if (!(bw > 0.0) || !isfinite(bw)) report_error(rep, VB_ERR_DEGENERATE);
}

vb_status bandwidth_run(Ctx* ctx, int64_t n, int32_t k, int32_t k_bw, const double* nbr_d2, double* b, float* ib)
{
    if (n < 1 || k < 1 || k_bw < 1 || k_bw > k || !nbr_d2 || !b) return VB_ERR_ARG;
    mark(ctx, VB_STAGE_BANDWIDTH, 0);
    bandwidth_kernel<<<(unsigned)((n + BW_T - 1) / BW_T), BW_T, 0, ctx->stream>>>(nbr_d2, n, k, k_bw, b, ib, ctx->rep);
    mark(ctx, VB_STAGE_BANDWIDTH, 1);
    ctx->launches += 1;
    return last_launch();
}

}  // namespace vb
