// Device-side format conversion: COO triplets -> CSR -> ELL / COO / HYB / BSR.
//
// The paper converts the input COO matrix to the chosen format on the CPU
// (Section 5.3 step 4; overhead in Section 7.5).  Here every step runs on
// the GPU: validation, a stable LSD radix sort on the (row, col) key,
// merging of duplicate pairs, the row-pointer array, and the packs of the
// other formats from CSR (Section 2.3 layouts).
#include <algorithm>
#include <climits>
#include <initializer_list>
#include <vector>

#include "combine.cuh"

namespace spmv {

namespace {

constexpr unsigned FULL = 0xffffffffu;

// ---------------------------------------------------------------------------
// temporary device buffer, freed (stream-ordered) when it goes out of scope
// ---------------------------------------------------------------------------
template <typename T>
struct Tmp {
    T *p = nullptr;
    cudaStream_t s = nullptr;
    Tmp() = default;
    Tmp(const Tmp &) = delete;
    Tmp &operator=(const Tmp &) = delete;
    ~Tmp() { if (p) cudaFreeAsync(p, s); }
    int alloc(size_t count, cudaStream_t stream) {
        s = stream;
        cudaError_t e = dev_malloc_async(reinterpret_cast<void **>(&p),
                                        std::max<size_t>(count, 1) * sizeof(T), stream);
        if (e != cudaSuccess) { p = nullptr; return cuda_status(e, "dev_malloc_async(temp)"); }
        return SPMV_OK;
    }
};

template <typename T>
int dalloc(T **p, size_t count) {
    cudaError_t e = dev_malloc(reinterpret_cast<void **>(p), std::max<size_t>(count, 1) * sizeof(T));
    if (e != cudaSuccess) { *p = nullptr; return cuda_status(e, "cudaMalloc"); }
    return SPMV_OK;
}
int dalloc_bytes(void **p, size_t bytes) {
    cudaError_t e = dev_malloc(p, std::max<size_t>(bytes, 1));
    if (e != cudaSuccess) { *p = nullptr; return cuda_status(e, "cudaMalloc"); }
    return SPMV_OK;
}

// The CSR arrays are allocated CSR_PAD entries longer than needed: the
// staged tile kernel copies whole multiples of 8 column/value entries and
// 16-byte windows of row pointers, so the last tile may read up to 7 entries
// past nnz and 3 past m (never used).
constexpr size_t CSR_PAD = 8;

inline int bits_for(int64_t count) {  // bits to hold 0 .. count-1
    int b = 0;
    while ((int64_t(1) << b) < count) ++b;
    return b;
}
// One block of several arrays, each on a 256-byte boundary; the first is the
// owner, the one to free.  (Mapping and unmapping cost by the block as well as
// by the byte.)
struct Slab {
    void **p;
    size_t bytes;
};
int dalloc_slab(std::initializer_list<Slab> parts) {
    size_t total = 0;
    for (const Slab &q : parts) total += (std::max<size_t>(q.bytes, 1) + 255) / 256 * 256;
    char *base = nullptr;
    for (const Slab &q : parts) *q.p = nullptr;
    cudaError_t e = dev_malloc(reinterpret_cast<void **>(&base), total);
    if (e != cudaSuccess) return cuda_status(e, "cudaMalloc");
    for (const Slab &q : parts) {
        *q.p = base;
        base += (std::max<size_t>(q.bytes, 1) + 255) / 256 * 256;
    }
    return SPMV_OK;
}
template <typename T>
Slab slab(T **p, size_t count) { return Slab{reinterpret_cast<void **>(p), sizeof(T) * count}; }
inline Slab slab_bytes(void **p, size_t bytes) { return Slab{p, bytes}; }

inline unsigned grid1d(int64_t work, int threads, int cap = 152 * 32) {
    int64_t g = (work + threads - 1) / threads;
    return (unsigned)std::max<int64_t>(1, std::min<int64_t>(g, cap));
}

// sums, maxima and bitwise ors of a block end in one atomic each: an atomic
// per warp on one word held these passes up (R-MAT, 8.4M triplets: 45, 29 and
// 22 us for check, contiguous pairs and longest row; 30, 9 and 3.5 now)
__device__ __forceinline__ void block_add(unsigned v, unsigned long long *out) {
    __shared__ unsigned s_v;
    if (threadIdx.x == 0) s_v = 0;
    __syncthreads();
    v = __reduce_add_sync(FULL, v);
    if ((threadIdx.x & 31) == 0 && v) atomicAdd(&s_v, v);
    __syncthreads();
    if (threadIdx.x == 0 && s_v) atomicAdd(out, (unsigned long long)s_v);
}

// ---------------------------------------------------------------------------
// validation: bit 0 = index out of range, bit 1 = not sorted by (row, col),
// bit 2 = a repeated (row, col) pair, bit 3 = over ROW_GAP empty rows in a row.
// The same pass forms what an ordered list needs besides: the row pointers
// (each written at the entry that opens its row; not across a gap of bit 3)
// and the number of consecutive entries with consecutive columns (a pair
// across a row boundary counts too; the statistic only steers a layout
// default).  An unordered list leaves both meaningless.
// ---------------------------------------------------------------------------
constexpr int ROW_GAP = 32, CHECK_STEPS = 8;

__global__ void __launch_bounds__(256) k_check_triplets(const int *__restrict__ rows, const int *__restrict__ cols,
                                                        int64_t nnz, int64_t m, int64_t n, unsigned *flags, int *rowptr,
                                                        unsigned long long *contiguous) {
    unsigned f = 0, cnt = 0;
    const int lane = threadIdx.x & 31;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t stride = (((int64_t)gridDim.x * blockDim.x) >> 5) * (32 * CHECK_STEPS);
    const unsigned mu = (unsigned)m, nu = (unsigned)n;  // below 2^31: one unsigned comparison checks both ends
    // rows (r, r2] start at entry i
    auto open_rows = [&](int r, int r2, int64_t i) {
        if (r2 == r + 1) rowptr[r2] = (int)i;
        else if (r2 - r > ROW_GAP) f |= 8u;
        else
            for (int q = r + 1; q <= r2; ++q) rowptr[q] = (int)i;
    };
    // a warp takes 32 CHECK_STEPS consecutive entries; an entry's successor is the next lane's
    for (int64_t w0 = warp * (32 * CHECK_STEPS); w0 < nnz; w0 += stride) {
        int r[CHECK_STEPS + 1], c[CHECK_STEPS + 1];
        const int left = (int)(nnz - w0 < 32 * CHECK_STEPS + 1 ? nnz - w0 : 32 * CHECK_STEPS + 1);  // entries from w0 on
        const int *rp = rows + w0 + lane, *cp = cols + w0 + lane;
#pragma unroll
        for (int j = 0; j <= CHECK_STEPS; ++j) {
            const bool read = (j < CHECK_STEPS || lane == 0) && 32 * j + lane < left;
            r[j] = read ? __ldg(rp + 32 * j) : 0;
            c[j] = read ? __ldg(cp + 32 * j) : 0;
        }
#pragma unroll
        for (int j = 0; j < CHECK_STEPS; ++j) {
            const int ru = __shfl_down_sync(FULL, r[j], 1), cu = __shfl_down_sync(FULL, c[j], 1);
            const int rn = __shfl_sync(FULL, r[j + 1], 0), cn = __shfl_sync(FULL, c[j + 1], 0);
            const int r2 = lane == 31 ? rn : ru, c2 = lane == 31 ? cn : cu;
            if (32 * j + lane < left) {
                const bool more = 32 * j + lane + 1 < left, in = (unsigned)r[j] < mu;
                if (!in || (unsigned)c[j] >= nu) f |= 1u;
                if (more) {
                    if (r2 < r[j] || (r2 == r[j] && c2 < c[j])) f |= 2u;
                    else if (r2 == r[j] && c2 == c[j]) f |= 4u;
                    cnt += c2 == c[j] + 1;
                }
                if (rowptr && in && (r2 != r[j] || !more || (j == 0 && lane == 0))) {
                    const int64_t i = w0 + 32 * j + lane;
                    if (i == 0) open_rows(-1, r[j], 0);
                    const unsigned next = more ? (unsigned)r2 : mu;
                    if (next <= mu && (int)next > r[j]) open_rows(r[j], (int)next, i + 1);
                }
            }
        }
    }
    __shared__ unsigned s_f;
    if (threadIdx.x == 0) s_f = 0;
    __syncthreads();
    f = __reduce_or_sync(FULL, f);
    if ((threadIdx.x & 31) == 0 && f) atomicOr(&s_f, f);
    if (contiguous) block_add(cnt, contiguous);
    __syncthreads();
    if (threadIdx.x == 0 && s_f) atomicOr(flags, s_f);
}

// rowptr[r] = first position whose row is >= r, over rows sorted ascending
__global__ void k_rowptr_from_sorted(const int *rows, int64_t nnz, int64_t m, int *rowptr) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r <= m; r += stride) {
        int64_t lo = 0, hi = nnz;
        while (lo < hi) {
            int64_t mid = (lo + hi) >> 1;
            if (rows[mid] < r) lo = mid + 1; else hi = mid;
        }
        rowptr[r] = (int)lo;
    }
}

// row of entry k: the r with rowptr[r] <= k < rowptr[r+1]
__device__ __forceinline__ int row_of(const int *rowptr, int64_t m, int64_t k) {
    int64_t lo = 0, hi = m;  // answer in [0, m-1]
    while (lo < hi) {
        int64_t mid = (lo + hi + 1) >> 1;
        if (rowptr[mid] <= k) lo = mid; else hi = mid - 1;
    }
    return (int)lo;
}

__global__ void k_expand_rows(const int *rowptr, int64_t m, int64_t nnz, int *rows) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < nnz; k += stride)
        rows[k] = row_of(rowptr, m, k);
}

// longest row, and the sum over groups of 32 rows of the group's longest row
// (counted up to 512 entries): what a warp with a lane per row waits for
__global__ void __launch_bounds__(1024) k_max_row(const int *rowptr, int64_t m, unsigned long long *longest,
                                                  unsigned long long *group_sum) {
    int best = 0;
    unsigned sum = 0;
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t mr = (m + 31) / 32 * 32;
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < mr; r += stride) {
        const int len = r < m ? rowptr[r + 1] - rowptr[r] : 0;
        best = max(best, len);
        sum += (unsigned)__reduce_max_sync(FULL, min(len, 512));
    }
    __shared__ int s_best;
    if (threadIdx.x == 0) s_best = 0;
    __syncthreads();
    best = __reduce_max_sync(FULL, best);
    if ((threadIdx.x & 31) == 0) atomicMax(&s_best, best);
    block_add((threadIdx.x & 31) == 0 ? sum : 0u, group_sum);
    if (threadIdx.x == 0) atomicMax(longest, (unsigned long long)s_best);
}

// consecutive stored entries whose columns are consecutive (as k_check_triplets counts them)
__global__ void __launch_bounds__(256) k_contiguous_pairs(const int *__restrict__ colidx, int64_t nnz,
                                                          unsigned long long *out) {
    unsigned cnt = 0;
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
#pragma unroll 4
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x + 1; k < nnz; k += stride)
        cnt += __ldg(colidx + k) == __ldg(colidx + k - 1) + 1;
    block_add(cnt, out);
}

// ---------------------------------------------------------------------------
// exclusive scan of int32 (three passes: tile sums, scan of sums, tiles)
// ---------------------------------------------------------------------------
constexpr int SC_THREADS = 256, SC_ITEMS = 8, SC_TILE = SC_THREADS * SC_ITEMS;

__device__ __forceinline__ int block_exclusive_scan(int v, int *total) {
    __shared__ int warp_sums[SC_THREADS / 32];
    int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int incl = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        int t = __shfl_up_sync(FULL, incl, d);
        if (lane >= d) incl += t;
    }
    if (lane == 31) warp_sums[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        int w = lane < SC_THREADS / 32 ? warp_sums[lane] : 0;
        int wi = w;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            int t = __shfl_up_sync(FULL, wi, d);
            if (lane >= d) wi += t;
        }
        if (lane < SC_THREADS / 32) warp_sums[lane] = wi - w;
        if (lane == SC_THREADS / 32 - 1) *total = wi;
    }
    __syncthreads();
    int r = incl - v + warp_sums[warp];
    __syncthreads();
    return r;
}

__global__ void __launch_bounds__(SC_THREADS) k_scan_reduce(const int *in, int64_t n, int *sums) {
    int64_t base = (int64_t)blockIdx.x * SC_TILE;
    int s = 0;
    for (int k = threadIdx.x; k < SC_TILE; k += SC_THREADS) {
        int64_t i = base + k;
        if (i < n) s += in[i];
    }
    s = __reduce_add_sync(FULL, s);
    __shared__ int ws[SC_THREADS / 32];
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        int t = 0;
        for (int w = 0; w < SC_THREADS / 32; ++w) t += ws[w];
        sums[blockIdx.x] = t;
    }
}

// single block: exclusive scan of nb tile sums in place, their total in
// sums[nb]
__global__ void __launch_bounds__(SC_THREADS) k_scan_sums(int *sums, int64_t nb) {
    __shared__ int total_s;
    int carry = 0;
    for (int64_t base = 0; base < nb; base += SC_TILE) {
        const int64_t at = base + (int64_t)threadIdx.x * SC_ITEMS;
        int v[SC_ITEMS], t = 0;
#pragma unroll
        for (int j = 0; j < SC_ITEMS; ++j) {
            v[j] = at + j < nb ? sums[at + j] : 0;
            t += v[j];
        }
        int ex = block_exclusive_scan(t, &total_s) + carry;
#pragma unroll
        for (int j = 0; j < SC_ITEMS; ++j) {
            if (at + j < nb) sums[at + j] = ex;
            ex += v[j];
        }
        carry += total_s;
        __syncthreads();
    }
    if (threadIdx.x == 0) sums[nb] = carry;
}

__global__ void __launch_bounds__(SC_THREADS) k_scan_down(const int *in, int *out, int64_t n,
                                                          const int *sums) {
    __shared__ int total_s;
    int64_t base = (int64_t)blockIdx.x * SC_TILE + (int64_t)threadIdx.x * SC_ITEMS;
    int v[SC_ITEMS];
    int t = 0;
#pragma unroll
    for (int j = 0; j < SC_ITEMS; ++j) {
        int64_t i = base + j;
        v[j] = i < n ? in[i] : 0;
        t += v[j];
    }
    int ex = block_exclusive_scan(t, &total_s) + sums[blockIdx.x];
#pragma unroll
    for (int j = 0; j < SC_ITEMS; ++j) {
        int64_t i = base + j;
        if (i < n) out[i] = ex;
        ex += v[j];
    }
}

// exclusive scan in -> out (may alias); returns the total through *total_host
// when non-null (synchronises the stream in that case)
int exclusive_scan(const int *in, int *out, int64_t n, cudaStream_t s, int64_t *total_host) {
    if (n <= 0) {
        if (total_host) *total_host = 0;
        return SPMV_OK;
    }
    int64_t nb = (n + SC_TILE - 1) / SC_TILE;
    Tmp<int> sums;
    SPMV_TRY(sums.alloc(nb + 1, s));
    k_scan_reduce<<<(unsigned)nb, SC_THREADS, 0, s>>>(in, n, sums.p);
    int last_in = 0;
    if (total_host) {
        SPMV_CUDA_TRY(cudaMemcpyAsync(&last_in, in + n - 1, sizeof(int), cudaMemcpyDeviceToHost, s));
    }
    k_scan_sums<<<1, SC_THREADS, 0, s>>>(sums.p, nb);
    k_scan_down<<<(unsigned)nb, SC_THREADS, 0, s>>>(in, out, n, sums.p);
    SPMV_CUDA_TRY(cudaGetLastError());
    if (total_host) {
        int last_out = 0;
        SPMV_CUDA_TRY(cudaMemcpyAsync(&last_out, out + n - 1, sizeof(int), cudaMemcpyDeviceToHost, s));
        SPMV_CUDA_TRY(cudaStreamSynchronize(s));
        *total_host = (int64_t)last_out + last_in;
    }
    return SPMV_OK;
}

// ---------------------------------------------------------------------------
// stable LSD radix sort of (uint64 key, value) pairs, at most 8 bits a pass.
// A pass is three kernels: digit counts per tile, a scan of each digit's
// counts over the tiles (one block per digit), and the scatter.  The
// scatter is the cost: its blocks order their tile in shared memory first, so
// that consecutive threads write runs of a digit to consecutive addresses.
// Writing each pair from where it was read touched a sector per pair: 161 us
// a pass on 8.4M pairs (and 49 counting, 23 scanning); now 63, 12.5 and 3.
// ---------------------------------------------------------------------------
constexpr int RS_BITS = 8, RS_BINS = 1 << RS_BITS;
constexpr int RS_THREADS = 512, RS_WARPS = RS_THREADS / 32;
// keys per thread: two scatter blocks per SM by shared memory
template <typename W>
constexpr int RS_ITEMS = sizeof(W) <= 4 ? 16 : 8;
template <typename W>
constexpr int RS_TILE = RS_THREADS * RS_ITEMS<W>;

// dynamic shared memory of the scatter: the tile's keys and values, the
// warps' digit counts, the digits' offsets
template <typename W>
constexpr size_t RS_SMEM = RS_TILE<W> * (sizeof(uint64_t) + sizeof(W)) + sizeof(unsigned) * RS_BINS +
                           sizeof(uint16_t) * RS_WARPS * RS_BINS;

__device__ __forceinline__ unsigned rs_digit(uint64_t key, int shift, unsigned mask) {
    return (unsigned)(key >> shift) & mask;
}

// lanes whose digit equals this lane's (RS_BINS: no key): one ballot per bit
// (match.any takes some 50 cycles of the SM for 32 different digits)
__device__ __forceinline__ unsigned rs_peers(unsigned d) {
    unsigned peers = FULL;
#pragma unroll
    for (int b = 0; b <= RS_BITS; ++b) {
        const unsigned set = __ballot_sync(FULL, (d >> b) & 1u);
        peers &= (d >> b) & 1u ? set : ~set;
    }
    return peers;
}

// hist[d * nblocks + b]: keys of tile b with digit d
template <int ITEMS>
__global__ void __launch_bounds__(RS_THREADS) k_radix_hist(const uint64_t *keys, int64_t n, int shift, unsigned mask,
                                                           unsigned *hist, int nblocks) {
    __shared__ unsigned h[RS_BINS];
    for (int i = threadIdx.x; i < RS_BINS; i += RS_THREADS) h[i] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * (RS_THREADS * ITEMS);
    unsigned d[ITEMS];
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
        const int64_t i = base + r * RS_THREADS + threadIdx.x;
        d[r] = i < n ? rs_digit(__ldg(keys + i), shift, mask) : RS_BINS;
    }
#pragma unroll
    for (int r = 0; r < ITEMS; ++r)
        if (d[r] < RS_BINS) atomicAdd(&h[d[r]], 1u);  // grouping equal digits first costs more than their conflicts
    __syncthreads();
    for (int d = threadIdx.x; d < RS_BINS; d += RS_THREADS) hist[(int64_t)d * nblocks + blockIdx.x] = h[d];
}

// block d: exclusive scan of digit d's counts over the tiles, and their total
__global__ void __launch_bounds__(SC_THREADS) k_radix_scan(int *hist, int nblocks, int *totals) {
    __shared__ int total_s;
    int *row = hist + (int64_t)blockIdx.x * nblocks;
    int carry = 0;
    for (int base = 0; base < nblocks; base += SC_TILE) {
        const int at = base + threadIdx.x * SC_ITEMS;
        int v[SC_ITEMS], t = 0;
#pragma unroll
        for (int j = 0; j < SC_ITEMS; ++j) {
            v[j] = at + j < nblocks ? row[at + j] : 0;
            t += v[j];
        }
        int ex = block_exclusive_scan(t, &total_s) + carry;
#pragma unroll
        for (int j = 0; j < SC_ITEMS; ++j) {
            if (at + j < nblocks) row[at + j] = ex;
            ex += v[j];
        }
        carry += total_s;
        __syncthreads();
    }
    if (threadIdx.x == 0) totals[blockIdx.x] = carry;
}

// exclusive scan of RS_BINS values by the block's first RS_BINS threads (the
// whole block calls it)
__device__ __forceinline__ unsigned scan_bins(unsigned v) {
    __shared__ unsigned ws[RS_BINS / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned incl = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const unsigned t = __shfl_up_sync(FULL, incl, d);
        if (lane >= d) incl += t;
    }
    __syncthreads();
    if (warp < RS_BINS / 32 && lane == 31) ws[warp] = incl;
    __syncthreads();
    unsigned before = 0;
    for (int w = 0; w < RS_BINS / 32 && w < warp; ++w) before += ws[w];
    return before + incl - v;
}

template <typename W>
__global__ void __launch_bounds__(RS_THREADS, 2)
k_radix_scatter(const uint64_t *__restrict__ kin, const W *__restrict__ vin, uint64_t *__restrict__ kout,
                W *__restrict__ vout, int64_t n, int shift, unsigned mask, const int *__restrict__ offsets,
                const int *__restrict__ totals, int nblocks) {
    constexpr int ITEMS = RS_ITEMS<W>, TILE = RS_TILE<W>;
    extern __shared__ __align__(16) unsigned char rs_smem[];
    uint64_t *sk = reinterpret_cast<uint64_t *>(rs_smem);
    W *sv = reinterpret_cast<W *>(sk + TILE);
    unsigned *delta = reinterpret_cast<unsigned *>(sv + TILE);  // global minus local position of a digit's first pair
    uint16_t *wh = reinterpret_cast<uint16_t *>(delta + RS_BINS);  // [warp][digit]: counts, then local positions
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    for (int i = tid; i < RS_WARPS * RS_BINS / 2; i += RS_THREADS) reinterpret_cast<unsigned *>(wh)[i] = 0;
    const int64_t base = (int64_t)blockIdx.x * TILE;
    const int count = (int)(n - base < TILE ? n - base : TILE);
    const int wbase = warp * 32 * ITEMS;
    const unsigned lt = (1u << lane) - 1u;
    uint16_t *mine = wh + warp * RS_BINS;
    uint64_t k[ITEMS];
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
        const int i = wbase + r * 32 + lane;
        k[r] = i < count ? kin[base + i] : 0;
    }
    __syncthreads();
    unsigned loc[ITEMS / 2];  // ranks among the warp's earlier pairs of the digit (below 2^16, two a word)
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
        const bool valid = wbase + r * 32 + lane < count;
        const unsigned d = valid ? rs_digit(k[r], shift, mask) : RS_BINS;
        const unsigned peers = rs_peers(d);
        const unsigned cnt = valid ? mine[d] : 0u;
        __syncwarp();
        if (valid && lane == 31 - __clz(peers)) mine[d] = (uint16_t)(cnt + __popc(peers));
        __syncwarp();
        const unsigned rank = cnt + __popc(peers & lt);
        loc[r / 2] = r % 2 ? loc[r / 2] | (rank << 16) : rank;
    }
    __syncthreads();
    // per digit: pairs of earlier warps, of the tile, and where the digit starts
    unsigned run = 0;
    if (tid < RS_BINS)
        for (int w = 0; w < RS_WARPS; ++w) {
            const unsigned c = wh[w * RS_BINS + tid];
            wh[w * RS_BINS + tid] = (uint16_t)run;
            run += c;
        }
    const unsigned local = scan_bins(tid < RS_BINS ? run : 0u);
    const unsigned global = scan_bins(tid < RS_BINS ? (unsigned)totals[tid] : 0u);
    if (tid < RS_BINS) {
        for (int w = 0; w < RS_WARPS; ++w) wh[w * RS_BINS + tid] = (uint16_t)(wh[w * RS_BINS + tid] + local);
        delta[tid] = global + (unsigned)offsets[(int64_t)tid * nblocks + blockIdx.x] - local;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
        const int i = wbase + r * 32 + lane;
        if (i < count) {
            const unsigned pos = mine[rs_digit(k[r], shift, mask)] + ((loc[r / 2] >> (r % 2 * 16)) & 0xffffu);
            sk[pos] = k[r];
            sv[pos] = vin[base + i];
        }
    }
    __syncthreads();
#pragma unroll 4
    for (int i = tid; i < count; i += RS_THREADS) {
        const uint64_t key = sk[i];
        const unsigned at = delta[rs_digit(key, shift, mask)] + (unsigned)i;
        kout[at] = key;
        vout[at] = sv[i];
    }
}

// Sorts keys[0..n) with their values of type W, read from vin and left, as the
// keys, in one of the two buffers of (keys, kalt) and (v0, v1).  vin may be v0.
template <typename W>
int radix_sort_pairs(uint64_t *keys, const W *vin, uint64_t *kalt, W *v0, W *v1, int64_t n, int total_bits,
                     cudaStream_t s, uint64_t **kres, W **vres) {
    const int nblocks = (int)((n + RS_TILE<W> - 1) / RS_TILE<W>);
    Tmp<int> hist;
    SPMV_TRY(hist.alloc((size_t)RS_BINS * nblocks + RS_BINS, s));
    int *totals = hist.p + (size_t)RS_BINS * nblocks;
    SPMV_CUDA_TRY(cudaFuncSetAttribute((const void *)k_radix_scatter<W>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)RS_SMEM<W>));
    uint64_t *ka = keys, *kb = kalt;
    W *vb = v1, *vo = v0;
    // passes of nearly equal width
    const int passes = (total_bits + RS_BITS - 1) / RS_BITS;
    int shift = 0;
    for (int p = 0; p < passes; ++p) {
        const int bits = (total_bits - shift + passes - p - 1) / (passes - p);
        const unsigned mask = (1u << bits) - 1u;
        k_radix_hist<RS_ITEMS<W>><<<nblocks, RS_THREADS, 0, s>>>(ka, n, shift, mask,
                                                                 reinterpret_cast<unsigned *>(hist.p), nblocks);
        k_radix_scan<<<RS_BINS, SC_THREADS, 0, s>>>(hist.p, nblocks, totals);
        k_radix_scatter<W><<<nblocks, RS_THREADS, RS_SMEM<W>, s>>>(ka, vin, kb, vb, n, shift, mask, hist.p, totals,
                                                                   nblocks);
        SPMV_CUDA_TRY(cudaGetLastError());
        std::swap(ka, kb);
        vin = vb;
        std::swap(vb, vo);
        shift += bits;
    }
    *kres = ka;
    *vres = vo;
    return SPMV_OK;
}

// ---------------------------------------------------------------------------
// unsorted / duplicated triplets: sort by (row, col), merge duplicates
// ---------------------------------------------------------------------------
__global__ void k_make_keys(const int *rows, const int *cols, int64_t nnz, int colbits, uint64_t *keys) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
#pragma unroll 4
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nnz; i += stride)
        keys[i] = ((uint64_t)(uint32_t)__ldg(rows + i) << colbits) | (uint32_t)__ldg(cols + i);
}

__global__ void k_heads(const uint64_t *keys, int64_t n, int *head) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride)
        head[i] = (i == 0 || keys[i] != keys[i - 1]) ? 1 : 0;
}

__device__ __forceinline__ double to_acc(double v) { return v; }
__device__ __forceinline__ float to_acc(float v) { return v; }
__device__ __forceinline__ float to_acc(__nv_bfloat16 v) { return __bfloat162float(v); }
__device__ __forceinline__ void from_acc(double a, double *o) { *o = a; }
__device__ __forceinline__ void from_acc(float a, float *o) { *o = a; }
__device__ __forceinline__ void from_acc(float a, __nv_bfloat16 *o) { *o = __float2bfloat16_rn(a); }

// Each run of equal keys becomes one entry; its value is the sum of the run's
// values in original triplet order (the sort is stable).  Two passes over the
// keys: heads per tile, then (after a scan of the tiles) the entries
// themselves; no head or position array is written.  A warp takes 256
// consecutive keys, 32 a step, so that loads and the stores of the entries
// (mostly one per key) are contiguous (eight keys in a row per thread: 160 us
// on 8.4M triplets, bound by partial-sector writes; 50 now,
// and 11 counting, against 156 with head and position arrays and a gather of
// the values through a sorted index).
__device__ __forceinline__ void head_masks(const uint64_t *__restrict__ keys, int64_t w0, int64_t n,
                                           uint64_t (&k)[SC_ITEMS], unsigned (&mask)[SC_ITEMS]) {
    const int lane = threadIdx.x & 31;
    uint64_t prev = lane == 0 && w0 > 0 && w0 < n ? __ldg(keys + w0 - 1) : 0;  // of lane 0: the key before the step
#pragma unroll
    for (int j = 0; j < SC_ITEMS; ++j) k[j] = w0 + 32 * j + lane < n ? __ldg(keys + w0 + 32 * j + lane) : 0;
#pragma unroll
    for (int j = 0; j < SC_ITEMS; ++j) {
        const int64_t i = w0 + 32 * j + lane;
        const uint64_t up = __shfl_up_sync(FULL, k[j], 1), last = __shfl_sync(FULL, k[j], 31);
        const uint64_t before = lane == 0 ? prev : up;
        mask[j] = __ballot_sync(FULL, i < n && (i == 0 || k[j] != before));
        prev = last;
    }
}

__global__ void __launch_bounds__(SC_THREADS) k_merge_count(const uint64_t *keys, int64_t n, int *sums) {
    __shared__ int ws[SC_THREADS / 32];
    const int warp = threadIdx.x >> 5;
    uint64_t k[SC_ITEMS];
    unsigned mask[SC_ITEMS];
    head_masks(keys, (int64_t)blockIdx.x * SC_TILE + 32 * SC_ITEMS * warp, n, k, mask);
    int c = 0;
#pragma unroll
    for (int j = 0; j < SC_ITEMS; ++j) c += __popc(mask[j]);
    if ((threadIdx.x & 31) == 0) ws[warp] = c;
    __syncthreads();
    if (threadIdx.x == 0) {
        int t = 0;
        for (int w = 0; w < SC_THREADS / 32; ++w) t += ws[w];
        sums[blockIdx.x] = t;
    }
}

template <typename V, typename T>
__global__ void __launch_bounds__(SC_THREADS)
k_merge_runs(const uint64_t *__restrict__ keys, const V *__restrict__ vin, const int *__restrict__ sums, int64_t n, int colbits, int *urows, int *ucols, V *uvals) {
    __shared__ int ws[SC_THREADS / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t w0 = (int64_t)blockIdx.x * SC_TILE + 32 * SC_ITEMS * warp;
    const uint64_t colmask = (uint64_t(1) << colbits) - 1;
    uint64_t k[SC_ITEMS];
    unsigned mask[SC_ITEMS];
    head_masks(keys, w0, n, k, mask);
    T v[SC_ITEMS];
    int c = 0;
#pragma unroll
    for (int j = 0; j < SC_ITEMS; ++j) {
        c += __popc(mask[j]);
        if ((mask[j] >> lane) & 1u) v[j] = to_acc(vin[w0 + 32 * j + lane]);
    }
    if (lane == 0) ws[warp] = c;
    __syncthreads();
    int u0 = sums[blockIdx.x];
    for (int w = 0; w < warp; ++w) u0 += ws[w];
#pragma unroll
    for (int j = 0; j < SC_ITEMS; ++j) {
        if ((mask[j] >> lane) & 1u) {
            T acc = v[j];
            for (int64_t i = w0 + 32 * j + lane + 1; i < n && keys[i] == k[j]; ++i) acc += to_acc(vin[i]);
            const int u = u0 + __popc(mask[j] & ((1u << lane) - 1u));
            urows[u] = (int)(k[j] >> colbits);
            ucols[u] = (int)(k[j] & colmask);
            from_acc(acc, &uvals[u]);
        }
        u0 += __popc(mask[j]);
    }
}

// The unordered path of build_csr: triplets sorted by (row, col) with their
// values as the sort's payload (a gather through a sorted index cost more than
// the values' way through the passes), then merged.  Sets h->nnz, h->colidx,
// h->vals and the row of every entry in `urows`.
template <typename V>
int sort_and_merge(spmv_matrix *h, const int32_t *d_rows, const int32_t *d_cols, const void *d_vals, int64_t nnz,
                   cudaStream_t s, Tmp<int> *urows) {
    using T = typename std::conditional<std::is_same<V, double>::value, double, float>::type;
    using W = typename std::conditional<sizeof(V) == 8, uint64_t,
                                        typename std::conditional<sizeof(V) == 4, uint32_t, uint16_t>::type>::type;
    const int colbits = std::max(1, bits_for(h->n));
    Tmp<uint64_t> k0, k1;
    Tmp<W> v0, v1;
    SPMV_TRY(k0.alloc(nnz, s));
    SPMV_TRY(k1.alloc(nnz, s));
    SPMV_TRY(v0.alloc(nnz, s));
    SPMV_TRY(v1.alloc(nnz, s));
    k_make_keys<<<grid1d(nnz, 256, 152 * 16), 256, 0, s>>>(d_rows, d_cols, nnz, colbits, k0.p);
    uint64_t *ks;
    W *vsorted;
    SPMV_TRY(radix_sort_pairs<W>(k0.p, static_cast<const W *>(d_vals), k1.p, v0.p, v1.p, nnz, bits_for(h->m) + colbits,
                                 s, &ks, &vsorted));
    const int64_t nb = (nnz + SC_TILE - 1) / SC_TILE;
    Tmp<int> sums;
    SPMV_TRY(sums.alloc(nb + 1, s));
    k_merge_count<<<(unsigned)nb, SC_THREADS, 0, s>>>(ks, nnz, sums.p);
    k_scan_sums<<<1, SC_THREADS, 0, s>>>(sums.p, nb);
    SPMV_CUDA_TRY(cudaGetLastError());
    int nu = 0;
    SPMV_CUDA_TRY(cudaMemcpyAsync(&nu, sums.p + nb, sizeof(int), cudaMemcpyDeviceToHost, s));
    SPMV_CUDA_TRY(cudaStreamSynchronize(s));
    h->nnz = nu;
    SPMV_TRY(urows->alloc(nu, s));
    SPMV_TRY(dalloc_slab({slab_bytes(&h->vals, sizeof(V) * (nu + CSR_PAD)), slab(&h->colidx, (size_t)nu + CSR_PAD)}));
    k_merge_runs<V, T><<<(unsigned)nb, SC_THREADS, 0, s>>>(ks, reinterpret_cast<const V *>(vsorted), sums.p, nnz, colbits,
                                                           urows->p, h->colidx, (V *)h->vals);
    SPMV_CUDA_TRY(cudaGetLastError());
    return SPMV_OK;
}

// ---------------------------------------------------------------------------
// format packs from CSR
// ---------------------------------------------------------------------------
// ELL columns as stored: int32 column (padding -1), or the 16-bit offset
// column - row (padding INT16_MIN) when every offset fits
__device__ __forceinline__ void ell_code(int *p, int c, int64_t r) { *p = c; }
__device__ __forceinline__ void ell_code(int16_t *p, int c, int64_t r) {
    *p = c < 0 ? (int16_t)INT16_MIN : (int16_t)(c - r);
}

// A warp packs 32 rows.  Their entries are contiguous in CSR: they are staged
// in shared memory with contiguous loads (at most `cap` entries; longer ranges
// are read in place, a row per lane) and leave column by column, 32 slots a
// store.  Reading a row per lane touched 32 lines a load: 27-point stencil
// 101^3, fp64, 216 us, 156 now (its bytes at the HBM rate: 98), bound by
// load latency at the 20 warps per SM that the staging leaves room for.
// One padding word per 32 spreads rows of one length over the banks.
constexpr int ELL_PACK_CAP = 4608, ELL_PACK_SMEM = 96 * 1024;
__host__ __device__ constexpr size_t ell_pack_words(int cap) { return (size_t)cap + cap / 32 + 1; }

// Entries of a slice that k_dia_slices stages, at most: 20480, less where their
// columns and values (12 bytes an entry for fp64) would not fit in the 227 KB a
// block may have.  A slice of more entries is read in place.
constexpr size_t DIA_PACK_SMEM = 224 * 1024;
template <typename V>
constexpr size_t dia_pack_smem(int cap, bool values) {
    return (4 * ell_pack_words(cap) + 15) / 16 * 16 + (values ? sizeof(V) * ell_pack_words(cap) : 0);
}
template <typename V>
constexpr int dia_pack_cap() {
    int cap = 20480;
    while (dia_pack_smem<V>(cap, true) > DIA_PACK_SMEM) cap -= 32;
    return cap;
}

template <typename V, typename CI>
__global__ void __launch_bounds__(128) k_ell_pack(const int *__restrict__ rowptr, const int *__restrict__ colidx,
                                                  const V *__restrict__ vals, int64_t m, int64_t width, int64_t pitch,
                                                  int cap, CI *ell_col, V *ell_val) {
    extern __shared__ __align__(16) unsigned char pack_smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const size_t words = ell_pack_words(cap);
    V *sv = reinterpret_cast<V *>(pack_smem) + warp * words;
    int *sc = reinterpret_cast<int *>(pack_smem + (sizeof(V) * words * nw + 15) / 16 * 16) + warp * words;
    const int64_t stride = (int64_t)gridDim.x * nw * 32;
    for (int64_t base = ((int64_t)blockIdx.x * nw + warp) * 32; base < pitch; base += stride) {
        const int64_t r = base + lane;
        const int s = __ldg(rowptr + (r < m ? r : m)), e = __ldg(rowptr + (r + 1 < m ? r + 1 : m));
        const int w0 = __shfl_sync(FULL, s, 0), w1 = __shfl_sync(FULL, e, 31);
        const bool staged = w1 - w0 <= cap;
        __syncwarp();
        if (staged) {
#pragma unroll 8
            for (int o = lane; o < w1 - w0; o += 32) {
                sc[o + (o >> 5)] = __ldg(colidx + w0 + o);
                sv[o + (o >> 5)] = vals[w0 + o];
            }
        }
        __syncwarp();
        const int len = e - s, first = s - w0;
#pragma unroll 4
        for (int k = 0; k < (int)width; ++k) {
            int c = -1;
            V v = V(0.0f);
            if (k < len) {
                const int o = first + k;
                c = staged ? sc[o + (o >> 5)] : __ldg(colidx + s + k);
                v = staged ? sv[o + (o >> 5)] : vals[s + k];
            }
            ell_code(ell_col + k * pitch + r, c, r);
            ell_val[k * pitch + r] = v;
        }
    }
}

// Diagonals of a slice (32 R rows, of each row its first `width` entries): a
// merge of the rows' ascending offsets, one step per distinct offset.  Without
// FILL the steps are counted and summed (sums[0], the entries in sums[1]); a
// slice of more than `most` offsets is given up and counted in sums[2], since
// its count is then too small to fill by.  With FILL each step writes its
// offset, row masks and values.  A block of R warps takes a slice
// (warp w the rows 32 w .. 32 w + 31, a row per lane), every step_s-th slice;
// the slice's columns and values are staged as in k_ell_pack, at most cap.
template <typename V, int R, bool FILL>
__global__ void __launch_bounds__(32 * R)
k_dia_slices(const int *__restrict__ rowptr, const int *__restrict__ colidx, const V *__restrict__ vals, int64_t m,
             int64_t width, int64_t nslices, int64_t step_s, int most, int cap, const int *__restrict__ ptr, int *count,
             unsigned long long *sums, int *off, uint32_t *mask, V *val) {
    extern __shared__ __align__(16) unsigned char pack_smem[];
    __shared__ int s_min[2][R];
    __shared__ unsigned s_entries;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    int *sc = reinterpret_cast<int *>(pack_smem);
    V *sv = reinterpret_cast<V *>(pack_smem + (4 * ell_pack_words(cap) + 15) / 16 * 16);
    if (!FILL && tid == 0) s_entries = 0;
    unsigned diags = 0, entries = 0, cut = 0;
    for (int64_t sl = (int64_t)blockIdx.x * step_s; sl < nslices; sl += (int64_t)gridDim.x * step_s) {
        const int64_t first = sl * (32 * R), row = first + tid, end = first + 32 * R < m ? first + 32 * R : m;
        const int w0 = __ldg(rowptr + first), w1 = __ldg(rowptr + end);
        int p = __ldg(rowptr + (row < m ? row : m)), e = __ldg(rowptr + (row + 1 < m ? row + 1 : m));
        const bool staged = w1 - w0 <= cap;
        __syncthreads();  // the previous slice's staging is read
        if (staged) {
#pragma unroll 8
            for (int o = tid; o < w1 - w0; o += 32 * R) {
                sc[o + (o >> 5)] = __ldg(colidx + w0 + o);
                if (FILL) sv[o + (o >> 5)] = vals[w0 + o];
            }
        }
        __syncthreads();
        auto col = [&](int k) -> int { return staged ? sc[(k - w0) + ((k - w0) >> 5)] : __ldg(colidx + k); };
        if (e - p > width) e = p + (int)width;
        entries += e - p;
        int d = p < e ? (int)(col(p) - row) : INT_MAX;
        int64_t at = FILL ? __ldg(ptr + sl) : 0;
        int n = 0;
        for (;; ++n) {
            int lo = __reduce_min_sync(FULL, d);
            if (R > 1) {  // over the block's warps; two sets, so one barrier a step
                if (lane == 0) s_min[n & 1][w] = lo;
                __syncthreads();
#pragma unroll
                for (int i = 0; i < R; ++i) lo = min(lo, s_min[n & 1][i]);
            }
            if (lo == INT_MAX) break;
            if (!FILL && n == most) {
                ++cut;
                break;
            }
            const bool hit = d == lo;
            if (FILL) {
                const uint32_t bits = __ballot_sync(FULL, hit);
                V v = V(0.0f);
                if (hit) v = staged ? sv[(p - w0) + ((p - w0) >> 5)] : vals[p];
                if (tid == 0) off[at] = lo;
                if (lane == 0) mask[at * R + w] = bits;
                val[(at * 32 + lane) * R + w] = v;
                ++at;
            }
            if (hit) {
                ++p;
                d = p < e ? (int)(col(p) - row) : INT_MAX;
            }
        }
        if (!FILL) {
            if (tid == 0 && count) count[sl] = n;
            diags += n;
        }
    }
    if (!FILL) {
        __syncthreads();
        entries = __reduce_add_sync(FULL, entries);
        if (lane == 0) atomicAdd(&s_entries, entries);
        __syncthreads();
        if (tid == 0) {
            atomicAdd(sums, (unsigned long long)diags);
            atomicAdd(sums + 1, (unsigned long long)s_entries);
            if (cut) atomicAdd(sums + 2, (unsigned long long)cut);
        }
    }
}

// rows of the diagonal layout as ELL columns and values (either may be null)
template <typename V>
__global__ void k_ell_from_csr(const int *rowptr, const int *colidx, const V *vals, int64_t m, int64_t width,
                               int64_t pitch, int *cols, V *out) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < pitch; r += stride) {
        const int s = r < m ? rowptr[r] : 0, len = r < m ? rowptr[r + 1] - s : 0;
        for (int64_t k = 0; k < width; ++k) {
            if (cols) cols[k * pitch + r] = k < len ? colidx[s + k] : -1;
            if (out) out[k * pitch + r] = k < len ? vals[s + k] : V(0.0f);
        }
    }
}

// largest |column - row| of the matrix (columns ascend within a row, so a
// row's first and last entries bound it)
__global__ void k_max_offset(const int *rowptr, const int *colidx, int64_t m, int *out) {
    int best = 0;
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < m; r += stride) {
        const int b = rowptr[r], e = rowptr[r + 1];
        if (b < e) {
            const int64_t lo = colidx[b] - r, hi = colidx[e - 1] - r;
            const int64_t d = max(lo < 0 ? -lo : lo, hi < 0 ? -hi : hi);
            best = max(best, (int)min(d, (int64_t)0x7fffffff));
        }
    }
    best = __reduce_max_sync(FULL, best);
    if ((threadIdx.x & 31) == 0) atomicMax(out, best);
}

// int32 columns of a 16-bit-offset ELL (for export)
__global__ void k_ell_decode(const int16_t *d16, int64_t width, int64_t pitch, int *out) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < width * pitch; i += stride) {
        const int v = d16[i];
        out[i] = v == INT16_MIN ? -1 : (int)(i % pitch) + v;
    }
}

// histogram of min(row length, cap)
__global__ void k_len_hist(const int *rowptr, int64_t m, int cap, unsigned *hist) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    unsigned lane = threadIdx.x & 31;
    int64_t mr = (m + 31) / 32 * 32;
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < mr; r += stride) {
        bool valid = r < m;
        int len = valid ? min(rowptr[r + 1] - rowptr[r], cap) : -1;
        unsigned peers = __match_any_sync(__activemask(), len);
        if (valid && lane == (unsigned)(31 - __clz(peers))) atomicAdd(&hist[len], (unsigned)__popc(peers));
    }
}

__global__ void k_tail_counts(const int *rowptr, int64_t m, int width, int *cnt) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < m; r += stride)
        cnt[r] = max(0, rowptr[r + 1] - rowptr[r] - width);
}

// tail entry o belongs to the row r with tptr[r] <= o < tptr[r+1]; entries
// are spread over the threads (long rows do not serialise on one thread)
template <typename V>
__global__ void k_hyb_tail(const int *rowptr, const int *colidx, const V *vals, int64_t m, int width,
                           const int *tptr, int64_t tail, int *trows, int *tcols, V *tvals) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t o = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; o < tail; o += stride) {
        const int r = row_of(tptr, m, o);
        const int64_t k = (int64_t)rowptr[r] + width + (o - tptr[r]);
        trows[o] = r;
        tcols[o] = colidx[k];
        tvals[o] = vals[k];
    }
}

__global__ void k_block_keys(const int *rows, const int *cols, int64_t nnz, int r, int bcbits,
                             uint64_t *keys, uint32_t *idx) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nnz; i += stride) {
        keys[i] = ((uint64_t)(rows[i] / r) << bcbits) | (uint64_t)(cols[i] / r);
        idx[i] = (uint32_t)i;
    }
}

template <typename V>
__global__ void k_bsr_fill(const uint64_t *keys, const uint32_t *perm, const int *head, const int *pos,
                           int64_t n, const int *rows, const int *cols, const V *vals, int r, int bcbits,
                           int *bcol, int *brow_of_block, V *bval) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const uint64_t mask = (uint64_t(1) << bcbits) - 1;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        int b = pos[i] + head[i] - 1;
        if (head[i]) {
            bcol[b] = (int)(keys[i] & mask);
            brow_of_block[b] = (int)(keys[i] >> bcbits);
        }
        uint32_t e = perm[i];
        int rr = rows[e] % r, cc = cols[e] % r;
        bval[(int64_t)b * r * r + rr * r + cc] = vals[e];
    }
}

// segmented-kernel chunk metadata (COO and HYB tail): first chunk of the
// chunk's head row and last chunk of its tail row
__global__ void k_seg_meta_coo(const int *rows, const int *rowptr, int64_t nnz, int C,
                               int64_t nchunks, int *meta0, int *meta1) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < nchunks; c += stride) {
        int64_t e0 = c * C, e1 = min(e0 + C, nnz);
        int hrow = rows[e0], trow = rows[e1 - 1];
        meta0[c] = rowptr[hrow] / C;
        meta1[c] = (rowptr[trow + 1] - 1) / C;
    }
}

// split CSR: row holding each chunk's first entry; entry nchunks = m - 1
__global__ void k_seg_meta_split(const int *rowptr, int64_t m, int64_t nnz, int C, int64_t nchunks,
                                 int *meta0) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c <= nchunks; c += stride) {
        if (c == nchunks) { meta0[c] = (int)(m - 1); continue; }
        meta0[c] = row_of(rowptr, m, c * C);
    }
}

// split CSR by warp chunks: first row starting at or after each chunk's
// first entry (lower bound of c*C in rowptr[0..m)); entry nchunks = m
__global__ void k_seg_meta_merge(const int *rowptr, int64_t m, int C, int64_t nchunks, int *meta) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c <= nchunks; c += stride) {
        if (c == nchunks) { meta[c] = (int)m; continue; }
        const int64_t k = c * (int64_t)C;
        int64_t lo = 0, hi = m;  // first r in [0, m] with r == m or rowptr[r] >= k
        while (lo < hi) {
            const int64_t mid = lo + ((hi - lo) >> 1);
            if (rowptr[mid] >= k) hi = mid; else lo = mid + 1;
        }
        meta[c] = (int)lo;
    }
}

__global__ void k_fill_u64(unsigned long long *p, int64_t n, unsigned long long v) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) p[i] = v;
}

// segments per long row: ceil(len / seg) if len > threshold, else 0
__global__ void k_long_count(const int *rowptr, int64_t nrows, int64_t threshold, int64_t seg, int *cnt) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < nrows; r += stride) {
        const int64_t len = rowptr[r + 1] - rowptr[r];
        cnt[r] = len > threshold ? (int)((len + seg - 1) / seg) : 0;
    }
}

__global__ void k_long_fill(const int *rowptr, int64_t nrows, int64_t threshold, int64_t seg, const int *off,
                            int *seg_row, int *seg_begin, int *seg_end, int *seg_c0, int *seg_c1) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < nrows; r += stride) {
        const int64_t b = rowptr[r], e = rowptr[r + 1];
        if (e - b <= threshold) continue;
        const int64_t ns = (e - b + seg - 1) / seg;
        const int o = off[r];
        for (int64_t j = 0; j < ns; ++j) {
            seg_row[o + j] = (int)r;
            seg_begin[o + j] = (int)(b + j * seg);
            seg_end[o + j] = (int)min(b + (j + 1) * seg, e);
            seg_c0[o + j] = o;
            seg_c1[o + j] = (int)(o + ns - 1);
        }
    }
}

// SELL: sort key per row = descending length (the sort is stable, so rows of
// equal length keep their order)
__global__ void k_sell_keys(const int *rowptr, int64_t m, int longest, uint64_t *keys, uint32_t *idx) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < m; r += stride) {
        const int len = rowptr[r + 1] - rowptr[r];
        keys[r] = (uint64_t)(uint32_t)(longest - len);
        idx[r] = (uint32_t)r;
    }
}

// slice width = length of its first (longest) sorted row; slots = 32 * width
__global__ void k_sell_widths(const int *rowptr, const uint32_t *perm, int64_t m, int64_t nslices, int *slots) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t sl = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; sl < nslices; sl += stride) {
        const uint32_t r = perm[sl * 32];
        slots[sl] = 32 * (rowptr[r + 1] - rowptr[r]);
    }
}

// Slot of entry k of lane l in a slice of width w starting at slot base:
// the first w & ~3 columns in groups of four, each group 32 lanes x 4
// consecutive entries (a lane's four entries of a group contiguous), then
// the remaining w & 3 columns column-major (32 lanes each).
// (grouped = false: every column column-major, entry k at base + 32 k + l)
__host__ __device__ __forceinline__ int64_t sell_slot(int64_t base, int64_t w, int64_t k, int l, bool grouped) {
    const int64_t w4 = grouped ? (w & ~int64_t(3)) : 0;
    return k < w4 ? base + 128 * (k >> 2) + 4 * l + (k & 3) : base + 32 * w4 + 32 * (k - w4) + l;
}

// A warp fills a work item (at most kmax columns of a slice): lane l walks its
// row's entries in order, so that its loads stay in one line for a while, and
// the stores of a column are contiguous.  (A warp per column found its slice
// by a binary search for every 32 slots.)
template <typename V>
__global__ void k_sell_fill(const int *__restrict__ rowptr, const int *__restrict__ colidx, const V *__restrict__ vals,
                            const uint32_t *__restrict__ perm, int64_t m, const int *__restrict__ sptr, int64_t nitems,
                            const int *__restrict__ it_slice, const int *__restrict__ it_base,
                            const int *__restrict__ it_len, int *scol, V *sval, int *sperm, bool grouped) {
    const int lane = threadIdx.x & 31;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t it = warp; it < nitems; it += nwarps) {
        const int sl = __ldg(it_slice + it), len = __ldg(it_len + it);
        const int sbase = __ldg(sptr + sl), w = (__ldg(sptr + sl + 1) - sbase) / 32, k0 = (__ldg(it_base + it) - sbase) / 32;
        const int64_t q = (int64_t)sl * 32 + lane;
        int rs = 0, n = 0;  // the lane's row
        if (q < m) {
            const uint32_t r = __ldg(perm + q);
            rs = __ldg(rowptr + r);
            n = __ldg(rowptr + r + 1) - rs;
        }
#pragma unroll 4
        for (int k = k0; k < k0 + len; ++k) {
            const bool have = k < n;
            const int c = have ? __ldg(colidx + rs + k) : -1;
            const V v = have ? vals[rs + k] : V(0.0f);
            const int64_t at = sell_slot(sbase, w, k, lane, grouped);
            scol[at] = c;
            sval[at] = v;
        }
    }
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < m; q += stride) sperm[q] = (int)perm[q];
}

// work items per slice: ceil(width / kmax), at least one
__global__ void k_sell_item_count(const int *sptr, int64_t nslices, int kmax, int *cnt) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t sl = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; sl < nslices; sl += stride) {
        const int width = (sptr[sl + 1] - sptr[sl]) / 32;
        cnt[sl] = (width + kmax - 1) / kmax;  // zero-width slices (empty rows) get no item
    }
}

// first zero-width slice: the first s with ptr[s] == ptr[nslices] (rows are
// sorted by descending length, so every later slice is empty too)
__global__ void k_sell_first_empty(const int *sptr, int64_t nslices, int *out) {
    const int total = sptr[nslices];
    int64_t lo = 0, hi = nslices;
    while (lo < hi) {
        const int64_t mid = lo + ((hi - lo) >> 1);
        if (sptr[mid] >= total) hi = mid; else lo = mid + 1;
    }
    *out = (int)lo;
}

// item j of a slice: its slice, the slot offset of its first column
// (ptr[slice] + 32 j kmax), its column count, and the slice's item range
__global__ void k_sell_item_fill(const int *sptr, int64_t nslices, int kmax, const int *off, int *it_slice,
                                 int *it_base, int *it_len, int *it_c0, int *it_c1) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t sl = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; sl < nslices; sl += stride) {
        const int width = (sptr[sl + 1] - sptr[sl]) / 32;
        const int n = (width + kmax - 1) / kmax;
        const int o = off[sl];
        for (int j = 0; j < n; ++j) {
            it_slice[o + j] = (int)sl;
            it_base[o + j] = sptr[sl] + 32 * j * kmax;
            it_len[o + j] = min((j + 1) * kmax, width) - j * kmax;
            it_c0[o + j] = o;
            it_c1[o + j] = o + n - 1;
        }
    }
}

// ---------------------------------------------------------------------------
// row panels: more triplets than one handle indexes with int32 offsets
// ---------------------------------------------------------------------------
constexpr int PANEL_CHUNK_SHIFT = 18;  // 2^18-row chunks, a multiple of 4 rows
constexpr int PC_THREADS = SC_THREADS, PC_ITEMS = 16, PC_TILE = PC_THREADS * PC_ITEMS;

// triplets per 2^18-row chunk; lanes of a warp on the same chunk add once
__global__ void k_chunk_hist(const int *rows, int64_t nnz, int nchunks, unsigned long long *counts) {
    extern __shared__ unsigned sh_chunks[];
    for (int c = threadIdx.x; c < nchunks; c += blockDim.x) sh_chunks[c] = 0;
    __syncthreads();
    const unsigned lane = threadIdx.x & 31;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t nr = (nnz + 31) / 32 * 32;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nr; i += stride) {
        const int c = i < nnz ? rows[i] >> PANEL_CHUNK_SHIFT : -1;
        const unsigned peers = __match_any_sync(FULL, c);
        if (c >= 0 && lane == (unsigned)(__ffs(peers) - 1)) atomicAdd(&sh_chunks[c], (unsigned)__popc(peers));
    }
    __syncthreads();
    for (int c = threadIdx.x; c < nchunks; c += blockDim.x)
        if (sh_chunks[c]) atomicAdd(&counts[c], (unsigned long long)sh_chunks[c]);
}

// triplets per 4-row group of rows [lo, hi)
__global__ void k_group_hist(const int *rows, int64_t nnz, int lo, int hi, unsigned long long *counts) {
    const unsigned lane = threadIdx.x & 31;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t nr = (nnz + 31) / 32 * 32;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nr; i += stride) {
        const int r = i < nnz ? rows[i] : -1;
        const int g = r >= lo && r < hi ? (r - lo) >> 2 : -1;
        const unsigned peers = __match_any_sync(FULL, g);
        if (g >= 0 && lane == (unsigned)(__ffs(peers) - 1)) atomicAdd(&counts[g], (unsigned long long)__popc(peers));
    }
}

// per 4096-triplet tile: triplets with row in [r0, r1)
__global__ void __launch_bounds__(PC_THREADS) k_panel_tile_count(const int *rows, int64_t nnz, int r0, int r1,
                                                                 int *cnt) {
    const int64_t base = (int64_t)blockIdx.x * PC_TILE;
    int c = 0;
    for (int k = threadIdx.x; k < PC_TILE; k += PC_THREADS) {
        const int64_t i = base + k;
        if (i < nnz) {
            const int r = rows[i];
            c += r >= r0 && r < r1;
        }
    }
    c = __reduce_add_sync(FULL, c);
    __shared__ int ws[PC_THREADS / 32];
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = c;
    __syncthreads();
    if (threadIdx.x == 0) {
        int t = 0;
        for (int w = 0; w < PC_THREADS / 32; ++w) t += ws[w];
        cnt[blockIdx.x] = t;
    }
}

// stable scatter of the tile's in-panel triplets to off[tile] + rank
template <typename W>
__global__ void __launch_bounds__(PC_THREADS) k_panel_scatter(const int *rows, const int *cols, const W *vals,
                                                              int64_t nnz, int r0, int r1, const int *off,
                                                              int *orow, int *ocol, W *oval) {
    __shared__ int total_s;
    const int64_t base = (int64_t)blockIdx.x * PC_TILE + (int64_t)threadIdx.x * PC_ITEMS;
    int c = 0;
#pragma unroll
    for (int j = 0; j < PC_ITEMS; ++j) {
        const int64_t i = base + j;
        if (i < nnz) {
            const int r = rows[i];
            c += r >= r0 && r < r1;
        }
    }
    int pos = block_exclusive_scan(c, &total_s) + off[blockIdx.x];
#pragma unroll
    for (int j = 0; j < PC_ITEMS; ++j) {
        const int64_t i = base + j;
        if (i < nnz) {
            const int r = rows[i];
            if (r >= r0 && r < r1) {
                orow[pos] = r - r0;
                ocol[pos] = cols[i];
                oval[pos] = vals[i];
                ++pos;
            }
        }
    }
}

}  // namespace

// ---------------------------------------------------------------------------
// public (library-internal) entry points
// ---------------------------------------------------------------------------

int decode_ell_columns(const spmv_matrix *h, int32_t *d_out, cudaStream_t s) {
    const int64_t n = h->ell_width * h->ell_pitch;
    if (n == 0) return SPMV_OK;
    k_ell_decode<<<grid1d(n, 256), 256, 0, s>>>(h->ell_d16, h->ell_width, h->ell_pitch, d_out);
    SPMV_CUDA_TRY(cudaGetLastError());
    return SPMV_OK;
}

// the ELL arrays of a handle that keeps diagonals, in the documented layout
int export_dia_as_ell(spmv_matrix *h, int32_t *cols, void *vals, cudaStream_t s) {
    const unsigned g = grid1d(h->ell_pitch, 256);
    auto go = [&](auto *v) {
        using V = std::remove_pointer_t<decltype(v)>;
        k_ell_from_csr<V><<<g, 256, 0, s>>>(h->rowptr, h->colidx, (const V *)h->vals, h->m, h->ell_width, h->ell_pitch,
                                            cols, (V *)vals);
    };
    if (h->vt == SPMV_F64) go((double *)nullptr);
    else if (h->vt == SPMV_F32) go((float *)nullptr);
    else go((__nv_bfloat16 *)nullptr);
    SPMV_CUDA_TRY(cudaGetLastError());
    return SPMV_OK;
}

int expand_rows(const int32_t *rowptr, int64_t m, int64_t nnz, int32_t *rows_out, cudaStream_t s) {
    if (nnz == 0) return SPMV_OK;
    k_expand_rows<<<grid1d(nnz, 256), 256, 0, s>>>(rowptr, m, nnz, rows_out);
    SPMV_CUDA_TRY(cudaGetLastError());
    return SPMV_OK;
}

int check_triplet_bounds(const int32_t *d_rows, const int32_t *d_cols, int64_t nnz, int64_t m, int64_t n,
                         cudaStream_t s) {
    if (nnz == 0) return SPMV_OK;
    Tmp<unsigned> flags;
    SPMV_TRY(flags.alloc(1, s));
    SPMV_CUDA_TRY(cudaMemsetAsync(flags.p, 0, sizeof(unsigned), s));
    k_check_triplets<<<grid1d(nnz, 256 * CHECK_STEPS, 152 * 8), 256, 0, s>>>(d_rows, d_cols, nnz, m, n, flags.p, nullptr,
                                                                         nullptr);
    SPMV_CUDA_TRY(cudaGetLastError());
    unsigned hflags = 0;
    SPMV_CUDA_TRY(cudaMemcpyAsync(&hflags, flags.p, sizeof(unsigned), cudaMemcpyDeviceToHost, s));
    SPMV_CUDA_TRY(cudaStreamSynchronize(s));
    if (hflags & 1u) {
        set_error("spmv_create: a triplet lies outside the %lld x %lld matrix", (long long)m, (long long)n);
        return SPMV_ERR_INVALID;
    }
    return SPMV_OK;
}

int plan_panels(const int32_t *d_rows, int64_t nnz, int64_t m, int64_t limit, cudaStream_t s,
                std::vector<int64_t> *bounds) {
    const int64_t chunk = int64_t(1) << PANEL_CHUNK_SHIFT;
    const int nchunks = (int)((m + chunk - 1) / chunk);
    Tmp<unsigned long long> counts;
    SPMV_TRY(counts.alloc(nchunks, s));
    SPMV_CUDA_TRY(cudaMemsetAsync(counts.p, 0, sizeof(unsigned long long) * nchunks, s));
    k_chunk_hist<<<grid1d(nnz, 256, 152 * 8), 256, sizeof(unsigned) * nchunks, s>>>(d_rows, nnz, nchunks, counts.p);
    SPMV_CUDA_TRY(cudaGetLastError());
    std::vector<unsigned long long> hc(nchunks);
    SPMV_CUDA_TRY(cudaMemcpyAsync(hc.data(), counts.p, sizeof(unsigned long long) * nchunks,
                                  cudaMemcpyDeviceToHost, s));
    SPMV_CUDA_TRY(cudaStreamSynchronize(s));
    bounds->assign(1, 0);
    int64_t cur = 0;  // triplets in the open panel
    for (int c = 0; c < nchunks; ++c) {
        const int64_t lo = (int64_t)c * chunk, hi = std::min<int64_t>(m, lo + chunk);
        if ((int64_t)hc[c] <= limit) {
            if (cur > 0 && cur + (int64_t)hc[c] > limit) {
                bounds->push_back(lo);
                cur = 0;
            }
            cur += (int64_t)hc[c];
            continue;
        }
        // a chunk over the limit: split it at 4-row groups
        const int64_t ng = (hi - lo + 3) / 4;
        Tmp<unsigned long long> g;
        SPMV_TRY(g.alloc(ng, s));
        SPMV_CUDA_TRY(cudaMemsetAsync(g.p, 0, sizeof(unsigned long long) * ng, s));
        k_group_hist<<<grid1d(nnz, 256, 152 * 8), 256, 0, s>>>(d_rows, nnz, (int)lo, (int)hi, g.p);
        SPMV_CUDA_TRY(cudaGetLastError());
        std::vector<unsigned long long> hg(ng);
        SPMV_CUDA_TRY(cudaMemcpyAsync(hg.data(), g.p, sizeof(unsigned long long) * ng, cudaMemcpyDeviceToHost, s));
        SPMV_CUDA_TRY(cudaStreamSynchronize(s));
        for (int64_t k = 0; k < ng; ++k) {
            if ((int64_t)hg[k] > limit) {
                set_error("spmv_create: rows %lld..%lld hold %llu triplets, more than one panel (%lld) holds",
                          (long long)(lo + 4 * k), (long long)std::min<int64_t>(m, lo + 4 * k + 4) - 1,
                          hg[k], (long long)limit);
                return SPMV_ERR_UNSUPPORTED;
            }
            if (cur > 0 && cur + (int64_t)hg[k] > limit) {
                bounds->push_back(lo + 4 * k);
                cur = 0;
            }
            cur += (int64_t)hg[k];
        }
    }
    bounds->push_back(m);
    return SPMV_OK;
}

int gather_panel(const int32_t *d_rows, const int32_t *d_cols, const void *d_vals, size_t vs, int64_t nnz,
                 int64_t r0, int64_t r1, int32_t **orow, int32_t **ocol, void **oval, int64_t *count,
                 cudaStream_t s) {
    *orow = *ocol = nullptr;
    *oval = nullptr;
    const int64_t ntiles = (nnz + PC_TILE - 1) / PC_TILE;
    Tmp<int> cnt, off;
    SPMV_TRY(cnt.alloc(ntiles, s));
    SPMV_TRY(off.alloc(ntiles, s));
    k_panel_tile_count<<<(unsigned)ntiles, PC_THREADS, 0, s>>>(d_rows, nnz, (int)r0, (int)r1, cnt.p);
    SPMV_CUDA_TRY(cudaGetLastError());
    int64_t total = 0;
    SPMV_TRY(exclusive_scan(cnt.p, off.p, ntiles, s, &total));
    *count = total;
    SPMV_TRY(dalloc(orow, (size_t)total));
    SPMV_TRY(dalloc(ocol, (size_t)total));
    SPMV_TRY(dalloc_bytes(oval, vs * (size_t)std::max<int64_t>(total, 1)));
    if (vs == 8)
        k_panel_scatter<uint64_t><<<(unsigned)ntiles, PC_THREADS, 0, s>>>(
            d_rows, d_cols, (const uint64_t *)d_vals, nnz, (int)r0, (int)r1, off.p, *orow, *ocol, (uint64_t *)*oval);
    else if (vs == 4)
        k_panel_scatter<uint32_t><<<(unsigned)ntiles, PC_THREADS, 0, s>>>(
            d_rows, d_cols, (const uint32_t *)d_vals, nnz, (int)r0, (int)r1, off.p, *orow, *ocol, (uint32_t *)*oval);
    else
        k_panel_scatter<uint16_t><<<(unsigned)ntiles, PC_THREADS, 0, s>>>(
            d_rows, d_cols, (const uint16_t *)d_vals, nnz, (int)r0, (int)r1, off.p, *orow, *ocol, (uint16_t *)*oval);
    SPMV_CUDA_TRY(cudaGetLastError());
    SPMV_CUDA_TRY(cudaStreamSynchronize(s));
    return SPMV_OK;
}

int build_csr(spmv_matrix *h, const int32_t *d_rows, const int32_t *d_cols, const void *d_vals,
              cudaStream_t s) {
    const int64_t m = h->m, n = h->n, nnz_in = h->nnz;
    const size_t vs = value_size(h->vt);
    SPMV_TRY(dalloc(&h->rowptr, (size_t)m + 1 + CSR_PAD));  // staged windows may read 3 past m
    if (nnz_in == 0) {
        SPMV_CUDA_TRY(cudaMemsetAsync(h->rowptr, 0, sizeof(int) * (m + 1), s));
        SPMV_TRY(dalloc_slab({slab_bytes(&h->vals, vs), slab(&h->colidx, 1)}));
        h->max_row = 0;
        SPMV_CUDA_TRY(cudaStreamSynchronize(s));
        return SPMV_OK;
    }
    // [0] flags, [1] longest row, [2] contiguous pairs, [3] longest rows of 32-row groups; for an
    // ordered list the first look at the triplets gives them all
    Tmp<unsigned long long> st;
    SPMV_TRY(st.alloc(4, s));
    unsigned long long hst[4] = {0, 0, 0, 0};
    auto row_statistics = [&]() {
        k_max_row<<<grid1d(m, 1024, 152), 1024, 0, s>>>(h->rowptr, m, st.p + 1, st.p + 3);
    };
    auto read_statistics = [&]() -> int {
        SPMV_CUDA_TRY(cudaGetLastError());
        SPMV_CUDA_TRY(cudaMemcpyAsync(hst, st.p, sizeof(hst), cudaMemcpyDeviceToHost, s));
        SPMV_CUDA_TRY(cudaStreamSynchronize(s));
        return SPMV_OK;
    };
    SPMV_CUDA_TRY(cudaMemsetAsync(st.p, 0, sizeof(hst), s));
    k_check_triplets<<<grid1d(nnz_in, 256 * CHECK_STEPS, 152 * 8), 256, 0, s>>>(
        d_rows, d_cols, nnz_in, m, n, reinterpret_cast<unsigned *>(st.p), h->rowptr, st.p + 2);
    row_statistics();
    SPMV_TRY(read_statistics());
    const unsigned hflags = (unsigned)hst[0];
    if (hflags & 1u) {
        set_error("spmv_create: a triplet lies outside the %lld x %lld matrix", (long long)m,
                  (long long)n);
        return SPMV_ERR_INVALID;
    }
    if (!(hflags & 6u)) {
        // already sorted by (row, col) with no repeated pair: copy and index
        h->nnz = nnz_in;
        SPMV_TRY(dalloc_slab({slab_bytes(&h->vals, vs * (nnz_in + CSR_PAD)), slab(&h->colidx, (size_t)nnz_in + CSR_PAD)}));
        SPMV_CUDA_TRY(cudaMemcpyAsync(h->colidx, d_cols, sizeof(int) * nnz_in, cudaMemcpyDeviceToDevice, s));
        SPMV_CUDA_TRY(cudaMemcpyAsync(h->vals, d_vals, vs * nnz_in, cudaMemcpyDeviceToDevice, s));
        if (hflags & 8u) {  // long runs of empty rows: every row pointer by a search
            SPMV_CUDA_TRY(cudaMemsetAsync(st.p + 1, 0, sizeof(unsigned long long), s));
            SPMV_CUDA_TRY(cudaMemsetAsync(st.p + 3, 0, sizeof(unsigned long long), s));
            k_rowptr_from_sorted<<<grid1d(m + 1, 256), 256, 0, s>>>(d_rows, nnz_in, m, h->rowptr);
            row_statistics();
            SPMV_TRY(read_statistics());
        }
    } else {
        Tmp<int> urows;
        if (h->vt == SPMV_F64) SPMV_TRY(sort_and_merge<double>(h, d_rows, d_cols, d_vals, nnz_in, s, &urows));
        else if (h->vt == SPMV_F32) SPMV_TRY(sort_and_merge<float>(h, d_rows, d_cols, d_vals, nnz_in, s, &urows));
        else SPMV_TRY(sort_and_merge<__nv_bfloat16>(h, d_rows, d_cols, d_vals, nnz_in, s, &urows));
        const int64_t nu = h->nnz;
        k_rowptr_from_sorted<<<grid1d(m + 1, 256), 256, 0, s>>>(urows.p, nu, m, h->rowptr);
        SPMV_CUDA_TRY(cudaMemsetAsync(st.p, 0, sizeof(hst), s));
        row_statistics();
        if (nu > 1) k_contiguous_pairs<<<grid1d(nu, 256, 152 * 8), 256, 0, s>>>(h->colidx, nu, st.p + 2);
        SPMV_TRY(read_statistics());
    }
    h->max_row = (int64_t)hst[1];
    h->group_max = (double)hst[3] / (double)((m + 31) / 32);
    h->contig = h->nnz > 1 ? (double)hst[2] / (double)(h->nnz - 1) : 0.0;
    return SPMV_OK;
}

int alloc_partials(Partials *p, int64_t units, int stride, int vt, cudaStream_t s) {
    *p = Partials{};
    p->units = units;
    p->stride = stride;
    const int64_t n = (units + 1) * stride;
    const size_t ts = vec_size(vt);
    SPMV_TRY(dalloc_bytes(&p->head, ts * n));
    SPMV_TRY(dalloc_bytes(&p->tail, ts * n));
    SPMV_TRY(dalloc(&p->count, (size_t)n));
    SPMV_TRY(dalloc(&p->xslot, (size_t)n));
    SPMV_CUDA_TRY(cudaMemsetAsync(p->count, 0, sizeof(uint32_t) * n, s));
    const unsigned long long empty = vt == SPMV_F64 ? XEnc<double>::EMPTY : XEnc<float>::EMPTY;
    k_fill_u64<<<grid1d(n, 256), 256, 0, s>>>(p->xslot, n, empty);
    SPMV_CUDA_TRY(cudaGetLastError());
    return SPMV_OK;
}

void free_partials(Partials *p) {
    auto f = [](void *q) { dev_free(q); };
    f(p->head); f(p->tail); f(p->count); f(p->xslot);
    *p = Partials{};
}

static void free_long_rows(spmv_matrix *h) {
    LongRows &L = h->lng;
    auto f = [](void *q) { dev_free(q); };
    f(L.seg_row); f(L.seg_begin); f(L.seg_end); f(L.seg_c0); f(L.seg_c1);
    free_partials(&L.part);
    L = LongRows{};
}

int build_long_rows(spmv_matrix *h, const int32_t *rowptr, int64_t nrows, int64_t longest, int64_t threshold,
                    int64_t seg, int stride, cudaStream_t s) {
    free_long_rows(h);
    LongRows &L = h->lng;
    L.threshold = threshold;
    if (nrows == 0 || longest <= threshold) return SPMV_OK;
    Tmp<int> cnt, off;
    SPMV_TRY(cnt.alloc(nrows, s));
    SPMV_TRY(off.alloc(nrows, s));
    k_long_count<<<grid1d(nrows, 256), 256, 0, s>>>(rowptr, nrows, threshold, seg, cnt.p);
    SPMV_CUDA_TRY(cudaGetLastError());
    int64_t total = 0;
    SPMV_TRY(exclusive_scan(cnt.p, off.p, nrows, s, &total));
    L.nseg = total;
    if (total == 0) return SPMV_OK;
    SPMV_TRY(dalloc(&L.seg_row, (size_t)total));
    SPMV_TRY(dalloc(&L.seg_begin, (size_t)total));
    SPMV_TRY(dalloc(&L.seg_end, (size_t)total));
    SPMV_TRY(dalloc(&L.seg_c0, (size_t)total));
    SPMV_TRY(dalloc(&L.seg_c1, (size_t)total));
    k_long_fill<<<grid1d(nrows, 256), 256, 0, s>>>(rowptr, nrows, threshold, seg, off.p, L.seg_row, L.seg_begin,
                                                   L.seg_end, L.seg_c0, L.seg_c1);
    SPMV_CUDA_TRY(cudaGetLastError());
    SPMV_TRY(alloc_partials(&L.part, total, stride, h->vt, s));
    return SPMV_OK;
}

void free_packed(spmv_matrix *h) {
    auto f = [](void *p) { dev_free(p); };
    f(h->coo_rows); h->coo_rows = nullptr;
    f(h->ell_val); h->ell_val = nullptr;  // index arrays go with the values
    h->ell_col = nullptr;
    h->ell_d16 = nullptr;
    f(h->dia_ptr); h->dia_ptr = nullptr;
    f(h->dia_val); h->dia_val = nullptr;
    h->dia_off = nullptr;
    h->dia_mask = nullptr;
    h->dia_total = 0;
    h->ell_width = h->ell_pitch = 0;
    f(h->hyb_rows); h->hyb_rows = nullptr;
    f(h->hyb_cols); h->hyb_cols = nullptr;
    f(h->hyb_vals); h->hyb_vals = nullptr;
    f(h->hyb_ptr); h->hyb_ptr = nullptr;
    h->hyb_nnz = 0;
    f(h->bsr_rowptr); h->bsr_rowptr = nullptr;
    f(h->bsr_col); h->bsr_col = nullptr;
    f(h->bsr_val); h->bsr_val = nullptr;
    f(h->sell_ptr); h->sell_ptr = nullptr;
    f(h->sell_val); h->sell_val = nullptr;
    h->sell_col = nullptr;
    f(h->sell_perm); h->sell_perm = nullptr;
    h->sell_nslices = h->sell_slots = 0;
    h->bsr_r = 0;
    h->bsr_mb = h->bsr_blocks = 0;
    f(h->seg.meta0); f(h->seg.meta1);
    free_partials(&h->seg.part);
    h->seg = SegScratch{};
    free_long_rows(h);
}

namespace {

// The most dynamic shared memory a kernel is ever launched with.  Always the
// same amount for a kernel: the limit is the process's, and a thread that set
// it to what its own launch needs would take from another thread's.
int allow_smem(const void *kernel, size_t most) {
    SPMV_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most));
    return SPMV_OK;
}

template <typename V, typename CI>
int launch_ell_pack_t(spmv_matrix *h, int64_t width, int64_t pitch, CI *cols, cudaStream_t s) {
    auto kern = k_ell_pack<V, CI>;
    const int cap = (int)std::min<int64_t>(ELL_PACK_CAP, 32 * width);
    const size_t per_warp = ell_pack_words(cap) * (sizeof(V) + 4);
    const int nw = (int)std::max<size_t>(1, std::min<size_t>(4, ELL_PACK_SMEM / per_warp));
    const size_t smem = (sizeof(V) * ell_pack_words(cap) * nw + 15) / 16 * 16 + 4 * ell_pack_words(cap) * nw;
    SPMV_TRY(allow_smem((const void *)kern, ELL_PACK_SMEM));
    kern<<<grid1d(pitch, 32 * nw, 1 << 20), 32 * nw, smem, s>>>(h->rowptr, h->colidx, (const V *)h->vals, h->m, width,
                                                                pitch, cap, cols, (V *)h->ell_val);
    SPMV_CUDA_TRY(cudaGetLastError());
    return SPMV_OK;
}

template <typename CI>
int launch_ell_pack(spmv_matrix *h, int64_t width, int64_t pitch, CI *cols, cudaStream_t s) {
    if (h->vt == SPMV_F64) return launch_ell_pack_t<double, CI>(h, width, pitch, cols, s);
    if (h->vt == SPMV_F32) return launch_ell_pack_t<float, CI>(h, width, pitch, cols, s);
    return launch_ell_pack_t<__nv_bfloat16, CI>(h, width, pitch, cols, s);
}

// Diagonals instead of columns, where that makes the product read clearly
// fewer bytes: at most 0.8 of the column-major layout's, and with fp64 values
// (one multiply-add per slot of a diagonal, entry or not, on the pipe that
// bounds them) at most 1.06 slots per entry; and from 2^20 entries on (a
// smaller product lasts as long as its launch either way), fp64 from 160 MB of
// columns and values on: those that stay in L2 (126 MB) do not gain by fewer
// bytes (27-point stencil, columns / diagonals, us: 216,000 rows 17.3 / 19.6,
// 300,000 20.8 / 21.8, 400,000 29.9 / 28.3, 1,000,000 61.3 / 56.6; band of 41,
// 300,000 rows 28.7 / 29.9, 400,000 42.1 / 37.9).
// A sample of 256 slices says whether it is worth counting them all.  One slice
// of more than 4 width + 16 offsets (irregular rows among regular ones) keeps
// the column layout.  *done: the handle keeps diagonals.
template <typename V>
int pack_dia(spmv_matrix *h, int64_t width, int index_bytes, cudaStream_t s, bool *done) {
    constexpr int R = DIA_ROWS<V>;
    *done = false;
    const int64_t m = h->m, nslices = (m + 32 * R - 1) / (32 * R);
    if (width == 0 || h->nnz < (1 << 20)) return SPMV_OK;
    if (sizeof(V) == 8 && (double)width * (double)m * (8.0 + index_bytes) < 160e6) return SPMV_OK;
    // staging for a slice's entries: read in place, long rows fall out of L1
    // between steps (band of half-width 32, bf16, 300,000 rows: 198 us a count and
    // 335 a fill with a warp per slice in place, 29 and 147 staged, a warp per 32 rows)
    const int cap = (int)std::min<int64_t>(dia_pack_cap<V>(), 32 * R * width);
    auto smem_of = [&](bool values) { return dia_pack_smem<V>(cap, values); };
    Tmp<unsigned long long> sums;
    Tmp<int> count;
    SPMV_TRY(sums.alloc(3, s));
    auto count_kernel = k_dia_slices<V, R, false>;
    SPMV_TRY(allow_smem((const void *)count_kernel, DIA_PACK_SMEM));
    // the diagonals of `slices` slices (one in step_s) and the entries on them
    auto counted = [&](int64_t step_s, int *out, bool *worth) -> int {
        const int64_t slices = (nslices + step_s - 1) / step_s;
        unsigned long long hs[3];
        SPMV_CUDA_TRY(cudaMemsetAsync(sums.p, 0, sizeof(hs), s));
        count_kernel<<<grid1d(slices, 1, 152 * 32), 32 * R, smem_of(false), s>>>(
            h->rowptr, h->colidx, (const V *)h->vals, m, width, nslices, step_s, (int)std::min<int64_t>(4 * width + 16, 1 << 20),
            cap, nullptr, out, sums.p, nullptr, nullptr, nullptr);
        SPMV_CUDA_TRY(cudaGetLastError());
        SPMV_CUDA_TRY(cudaMemcpyAsync(hs, sums.p, sizeof(hs), cudaMemcpyDeviceToHost, s));
        SPMV_CUDA_TRY(cudaStreamSynchronize(s));
        const double slots = 32.0 * R * (double)hs[0], entries = (double)hs[1];
        const double dia = slots * sizeof(V) + (double)hs[0] * (4 + 4 * R), ell = entries * (double)(sizeof(V) + index_bytes);
        *worth = hs[2] == 0 && entries > 0 && dia <= 0.8 * ell && (sizeof(V) < 8 || slots <= 1.06 * entries);
        return SPMV_OK;
    };
    bool worth = false;
    if (nslices > 512) {
        SPMV_TRY(counted(nslices / 256, nullptr, &worth));
        if (!worth) return SPMV_OK;
    }
    SPMV_TRY(count.alloc(nslices + 1, s));
    SPMV_CUDA_TRY(cudaMemsetAsync(count.p + nslices, 0, sizeof(int), s));
    SPMV_TRY(counted(1, count.p, &worth));
    if (!worth) return SPMV_OK;
    int64_t total = 0;
    SPMV_TRY(dalloc(&h->dia_ptr, (size_t)nslices + 1));
    SPMV_TRY(exclusive_scan(count.p, h->dia_ptr, nslices + 1, s, &total));
    h->dia_total = total;
    SPMV_TRY(dalloc_slab({slab_bytes(&h->dia_val, sizeof(V) * (size_t)total * 32 * R), slab(&h->dia_off, (size_t)total),
                          slab(&h->dia_mask, (size_t)total * R)}));
    auto fill = k_dia_slices<V, R, true>;
    SPMV_TRY(allow_smem((const void *)fill, DIA_PACK_SMEM));
    fill<<<grid1d(nslices, 1, 1 << 30), 32 * R, smem_of(true), s>>>(h->rowptr, h->colidx, (const V *)h->vals, m, width, nslices, 1,
                                                             INT_MAX, cap, h->dia_ptr, nullptr, nullptr, h->dia_off,
                                                             h->dia_mask, (V *)h->dia_val);
    SPMV_CUDA_TRY(cudaGetLastError());
    *done = true;
    return SPMV_OK;
}

// bf16 values: columns are stored as 16-bit offsets from the row when
// every |column - row| of the matrix is at most 32767 (stencils, banded and
// block-diagonal matrices), 2 index bytes per slot instead of 4.  Measured
// on GB300 at the default unroll: bf16 13% faster (27-point stencil 76.5
// against 88.1 us); fp32 only gains at unroll 8 and loses 18% at its
// default 4; fp64 loses 8-10% (its ELL kernel is held by the fp64 pipe and
// the decode sits between the column load and the x gather).  fp32 and
// fp64 keep int32 columns.
int pack_ell(spmv_matrix *h, int64_t width, cudaStream_t s) {
    const int64_t m = h->m;
    const int64_t pitch = (m + 31) / 32 * 32;
    const size_t vs = value_size(h->vt);
    h->ell_width = width;
    h->ell_pitch = pitch;
    int maxoff = 0x7fffffff;
    if (width > 0 && m > 0 && h->vt == SPMV_BF16) {
        Tmp<int> mo;
        SPMV_TRY(mo.alloc(1, s));
        SPMV_CUDA_TRY(cudaMemsetAsync(mo.p, 0, sizeof(int), s));
        k_max_offset<<<grid1d(m, 256), 256, 0, s>>>(h->rowptr, h->colidx, m, mo.p);
        SPMV_CUDA_TRY(cudaGetLastError());
        SPMV_CUDA_TRY(cudaMemcpyAsync(&maxoff, mo.p, sizeof(int), cudaMemcpyDeviceToHost, s));
        SPMV_CUDA_TRY(cudaStreamSynchronize(s));
    }
    bool dia = false;
    const int index_bytes = maxoff <= 32767 ? 2 : 4;
    if (h->vt == SPMV_F64) SPMV_TRY(pack_dia<double>(h, width, index_bytes, s, &dia));
    else if (h->vt == SPMV_F32) SPMV_TRY(pack_dia<float>(h, width, index_bytes, s, &dia));
    else SPMV_TRY(pack_dia<__nv_bfloat16>(h, width, index_bytes, s, &dia));
    if (dia) return SPMV_OK;
    if (maxoff <= 32767) {
        SPMV_TRY(dalloc_slab({slab_bytes(&h->ell_val, vs * width * pitch), slab(&h->ell_d16, (size_t)(width * pitch))}));
        if (width > 0 && pitch > 0) SPMV_TRY(launch_ell_pack<int16_t>(h, width, pitch, h->ell_d16, s));
    } else {
        SPMV_TRY(dalloc_slab({slab_bytes(&h->ell_val, vs * width * pitch), slab(&h->ell_col, (size_t)(width * pitch))}));
        if (width > 0 && pitch > 0) SPMV_TRY(launch_ell_pack<int>(h, width, pitch, h->ell_col, s));
    }
    return SPMV_OK;
}

// HYB ELL width: the largest k >= 1 with at least max(4096, m/3) rows of
// length >= k (0 if none)
int hyb_width_rule(spmv_matrix *h, cudaStream_t s, int64_t *width) {
    const int64_t m = h->m;
    const int cap = (int)std::min<int64_t>(h->max_row, 1 << 20);
    if (m == 0 || cap == 0) { *width = 0; return SPMV_OK; }
    Tmp<unsigned> hist;
    SPMV_TRY(hist.alloc(cap + 1, s));
    SPMV_CUDA_TRY(cudaMemsetAsync(hist.p, 0, sizeof(unsigned) * (cap + 1), s));
    k_len_hist<<<grid1d(m, 256), 256, 0, s>>>(h->rowptr, m, cap, hist.p);
    std::vector<unsigned> hh(cap + 1);
    SPMV_CUDA_TRY(cudaMemcpyAsync(hh.data(), hist.p, sizeof(unsigned) * (cap + 1), cudaMemcpyDeviceToHost, s));
    SPMV_CUDA_TRY(cudaStreamSynchronize(s));
    int64_t ge = m;  // rows with length >= k, k = 0
    int64_t best = 0;
    for (int k = 1; k <= cap; ++k) {
        ge -= hh[k - 1];
        if (ge >= 4096 && 3 * ge >= m) best = k;
        else break;
    }
    *width = best;
    return SPMV_OK;
}

int pack_hyb(spmv_matrix *h, int64_t width, cudaStream_t s) {
    const int64_t m = h->m;
    SPMV_TRY(pack_ell(h, width, s));
    SPMV_TRY(dalloc(&h->hyb_ptr, (size_t)m + 1));
    Tmp<int> cnt;
    SPMV_TRY(cnt.alloc(m + 1, s));
    SPMV_CUDA_TRY(cudaMemsetAsync(cnt.p, 0, sizeof(int) * (m + 1), s));
    if (m > 0) k_tail_counts<<<grid1d(m, 256), 256, 0, s>>>(h->rowptr, m, (int)width, cnt.p);
    int64_t tail = 0;
    SPMV_TRY(exclusive_scan(cnt.p, h->hyb_ptr, m + 1, s, &tail));
    h->hyb_nnz = tail;
    const size_t vs = value_size(h->vt);
    SPMV_TRY(dalloc(&h->hyb_rows, (size_t)tail));
    SPMV_TRY(dalloc(&h->hyb_cols, (size_t)tail));
    SPMV_TRY(dalloc_bytes(&h->hyb_vals, vs * tail));
    if (tail > 0) {
        unsigned g = grid1d(tail, 256);
        if (h->vt == SPMV_F64)
            k_hyb_tail<double><<<g, 256, 0, s>>>(h->rowptr, h->colidx, (const double *)h->vals, m, (int)width,
                                                 h->hyb_ptr, tail, h->hyb_rows, h->hyb_cols, (double *)h->hyb_vals);
        else if (h->vt == SPMV_F32)
            k_hyb_tail<float><<<g, 256, 0, s>>>(h->rowptr, h->colidx, (const float *)h->vals, m, (int)width,
                                                h->hyb_ptr, tail, h->hyb_rows, h->hyb_cols, (float *)h->hyb_vals);
        else
            k_hyb_tail<__nv_bfloat16><<<g, 256, 0, s>>>(h->rowptr, h->colidx, (const __nv_bfloat16 *)h->vals, m,
                                                        (int)width, h->hyb_ptr, tail, h->hyb_rows, h->hyb_cols,
                                                        (__nv_bfloat16 *)h->hyb_vals);
        SPMV_CUDA_TRY(cudaGetLastError());
    }
    return SPMV_OK;
}

int pack_bsr(spmv_matrix *h, int r, cudaStream_t s) {
    const int64_t m = h->m, n = h->n, nnz = h->nnz;
    const int64_t mb = (m + r - 1) / r, nb = (n + r - 1) / r;
    const size_t vs = value_size(h->vt);
    h->bsr_r = r;
    h->bsr_mb = mb;
    SPMV_TRY(dalloc(&h->bsr_rowptr, (size_t)mb + 1));
    if (nnz == 0) {
        h->bsr_blocks = 0;
        SPMV_CUDA_TRY(cudaMemsetAsync(h->bsr_rowptr, 0, sizeof(int) * (mb + 1), s));
        SPMV_TRY(dalloc(&h->bsr_col, 1));
        SPMV_TRY(dalloc_bytes(&h->bsr_val, vs));
        return SPMV_OK;
    }
    const int bcbits = std::max(1, bits_for(nb));
    const int total_bits = bits_for(mb) + bcbits;
    Tmp<int> rows;
    SPMV_TRY(rows.alloc(nnz, s));
    SPMV_TRY(expand_rows(h->rowptr, m, nnz, rows.p, s));
    Tmp<uint64_t> k0, k1;
    Tmp<uint32_t> v0, v1;
    SPMV_TRY(k0.alloc(nnz, s));
    SPMV_TRY(k1.alloc(nnz, s));
    SPMV_TRY(v0.alloc(nnz, s));
    SPMV_TRY(v1.alloc(nnz, s));
    k_block_keys<<<grid1d(nnz, 256), 256, 0, s>>>(rows.p, h->colidx, nnz, r, bcbits, k0.p, v0.p);
    uint64_t *ks;
    uint32_t *vp;
    SPMV_TRY(radix_sort_pairs<uint32_t>(k0.p, v0.p, k1.p, v0.p, v1.p, nnz, total_bits, s, &ks, &vp));
    Tmp<int> head, pos;
    SPMV_TRY(head.alloc(nnz, s));
    SPMV_TRY(pos.alloc(nnz, s));
    k_heads<<<grid1d(nnz, 256), 256, 0, s>>>(ks, nnz, head.p);
    int64_t nblk = 0;
    SPMV_TRY(exclusive_scan(head.p, pos.p, nnz, s, &nblk));
    h->bsr_blocks = nblk;
    if ((double)nblk * r * r > 8.0 * (double)nnz + (double)(1 << 24)) {
        set_error("BSR: %lld blocks of %dx%d exceed 8 x nnz + 2^24 value slots", (long long)nblk, r, r);
        return SPMV_ERR_UNSUPPORTED;
    }
    SPMV_TRY(dalloc(&h->bsr_col, (size_t)nblk));
    SPMV_TRY(dalloc_bytes(&h->bsr_val, vs * nblk * r * r));
    SPMV_CUDA_TRY(cudaMemsetAsync(h->bsr_val, 0, vs * nblk * r * r, s));
    Tmp<int> brow;
    SPMV_TRY(brow.alloc(nblk, s));
    unsigned g = grid1d(nnz, 256);
    if (h->vt == SPMV_F64)
        k_bsr_fill<double><<<g, 256, 0, s>>>(ks, vp, head.p, pos.p, nnz, rows.p, h->colidx, (const double *)h->vals,
                                             r, bcbits, h->bsr_col, brow.p, (double *)h->bsr_val);
    else if (h->vt == SPMV_F32)
        k_bsr_fill<float><<<g, 256, 0, s>>>(ks, vp, head.p, pos.p, nnz, rows.p, h->colidx, (const float *)h->vals,
                                            r, bcbits, h->bsr_col, brow.p, (float *)h->bsr_val);
    else
        k_bsr_fill<__nv_bfloat16><<<g, 256, 0, s>>>(ks, vp, head.p, pos.p, nnz, rows.p, h->colidx,
                                                    (const __nv_bfloat16 *)h->vals, r, bcbits, h->bsr_col, brow.p,
                                                    (__nv_bfloat16 *)h->bsr_val);
    k_rowptr_from_sorted<<<grid1d(mb + 1, 256), 256, 0, s>>>(brow.p, nblk, mb, h->bsr_rowptr);
    SPMV_CUDA_TRY(cudaGetLastError());
    SPMV_CUDA_TRY(cudaStreamSynchronize(s));
    return SPMV_OK;
}

}  // namespace

namespace {

// kmax: columns of a slice per work item (wider slices become several items)
int pack_sell(spmv_matrix *h, int kmax, bool grouped, cudaStream_t s) {
    const int64_t m = h->m;
    const int64_t nslices = (m + 31) / 32;
    const size_t vs = value_size(h->vt);
    h->sell_nslices = nslices;
    h->sell_grouped = grouped;
    SPMV_TRY(dalloc(&h->sell_ptr, (size_t)nslices + 1));
    SPMV_TRY(dalloc(&h->sell_perm, (size_t)std::max<int64_t>(m, 1)));
    if (m == 0) {
        SPMV_CUDA_TRY(cudaMemsetAsync(h->sell_ptr, 0, sizeof(int), s));
        SPMV_TRY(dalloc_slab({slab_bytes(&h->sell_val, vs), slab(&h->sell_col, 1)}));
        h->sell_slots = 0;
        return SPMV_OK;
    }
    // sort all rows by descending length (stable): slices group rows of
    // similar length, so padding stays small even for power-law rows
    Tmp<uint64_t> k0, k1;
    Tmp<uint32_t> v0, v1;
    SPMV_TRY(k0.alloc(m, s));
    SPMV_TRY(k1.alloc(m, s));
    SPMV_TRY(v0.alloc(m, s));
    SPMV_TRY(v1.alloc(m, s));
    k_sell_keys<<<grid1d(m, 256), 256, 0, s>>>(h->rowptr, m, (int)h->max_row, k0.p, v0.p);
    uint64_t *ks;
    uint32_t *perm;
    SPMV_TRY(radix_sort_pairs<uint32_t>(k0.p, v0.p, k1.p, v0.p, v1.p, m, std::max(1, bits_for(h->max_row + 1)), s, &ks, &perm));
    Tmp<int> slots;
    SPMV_TRY(slots.alloc(nslices + 1, s));
    SPMV_CUDA_TRY(cudaMemsetAsync(slots.p, 0, sizeof(int) * (nslices + 1), s));
    k_sell_widths<<<grid1d(nslices, 256), 256, 0, s>>>(h->rowptr, perm, m, nslices, slots.p);
    int64_t total = 0;
    SPMV_TRY(exclusive_scan(slots.p, h->sell_ptr, nslices + 1, s, &total));
    if ((double)total > 8.0 * (double)h->nnz + (double)(1 << 24) || total >= (int64_t(1) << 31)) {
        set_error("SELL: %lld padded slots exceed min(8 x nnz + 2^24, 2^31 - 1)", (long long)total);
        return SPMV_ERR_UNSUPPORTED;
    }
    h->sell_slots = total;
    SPMV_TRY(dalloc_slab({slab_bytes(&h->sell_val, vs * total), slab(&h->sell_col, (size_t)total)}));
    // work items (slice, first slot, column count <= kmax) and the partials
    // joining the items of one slice
    LongRows &L = h->lng;
    Tmp<int> cnt, off;
    SPMV_TRY(cnt.alloc(nslices, s));
    SPMV_TRY(off.alloc(nslices, s));
    k_sell_item_count<<<grid1d(nslices, 256), 256, 0, s>>>(h->sell_ptr, nslices, kmax, cnt.p);
    int64_t nitems = 0;
    SPMV_TRY(exclusive_scan(cnt.p, off.p, nslices, s, &nitems));
    L.nseg = nitems;
    L.threshold = kmax;
    SPMV_TRY(dalloc(&L.seg_row, (size_t)nitems));
    SPMV_TRY(dalloc(&L.seg_begin, (size_t)nitems));
    SPMV_TRY(dalloc(&L.seg_end, (size_t)nitems));
    SPMV_TRY(dalloc(&L.seg_c0, (size_t)nitems));
    SPMV_TRY(dalloc(&L.seg_c1, (size_t)nitems));
    k_sell_item_fill<<<grid1d(nslices, 256), 256, 0, s>>>(h->sell_ptr, nslices, kmax, off.p, L.seg_row,
                                                           L.seg_begin, L.seg_end, L.seg_c0, L.seg_c1);
    SPMV_CUDA_TRY(cudaGetLastError());
    const unsigned g = grid1d(std::max<int64_t>(32 * nitems, m), 256, 152 * 16);
    auto fill = [&](auto *v) {
        using V = std::remove_pointer_t<decltype(v)>;
        k_sell_fill<V><<<g, 256, 0, s>>>(h->rowptr, h->colidx, (const V *)h->vals, perm, m, h->sell_ptr, nitems, L.seg_row,
                                         L.seg_begin, L.seg_end, h->sell_col, (V *)h->sell_val, h->sell_perm, grouped);
    };
    if (h->vt == SPMV_F64) fill((double *)nullptr);
    else if (h->vt == SPMV_F32) fill((float *)nullptr);
    else fill((__nv_bfloat16 *)nullptr);
    SPMV_CUDA_TRY(cudaGetLastError());
    SPMV_TRY(alloc_partials(&L.part, nitems, 32, h->vt, s));
    // rows of the zero-width slices are written by a grid-stride pass
    Tmp<int> sz;
    SPMV_TRY(sz.alloc(1, s));
    k_sell_first_empty<<<1, 1, 0, s>>>(h->sell_ptr, nslices, sz.p);
    SPMV_CUDA_TRY(cudaGetLastError());
    int hz = 0;
    SPMV_CUDA_TRY(cudaMemcpyAsync(&hz, sz.p, sizeof(int), cudaMemcpyDeviceToHost, s));
    SPMV_CUDA_TRY(cudaStreamSynchronize(s));
    L.nrows = hz;
    return SPMV_OK;
}
}  // namespace

int build_coo_meta(const int32_t *rows, const int32_t *rowptr, int64_t nnz, int C, int32_t *meta0, int32_t *meta1,
                   cudaStream_t s) {
    const int64_t nchunks = (nnz + C - 1) / C;
    if (nchunks == 0) return SPMV_OK;
    k_seg_meta_coo<<<grid1d(nchunks + 1, 256), 256, 0, s>>>(rows, rowptr, nnz, C, nchunks, meta0, meta1);
    SPMV_CUDA_TRY(cudaGetLastError());
    return SPMV_OK;
}

int build_merge_meta(const int32_t *rowptr, int64_t m, int64_t nnz, int C, int32_t *meta, cudaStream_t s) {
    const int64_t nchunks = (nnz + C - 1) / C;
    k_seg_meta_merge<<<grid1d(nchunks + 1, 256), 256, 0, s>>>(rowptr, m, C, nchunks, meta);
    SPMV_CUDA_TRY(cudaGetLastError());
    return SPMV_OK;
}

int ensure_seg_scratch(spmv_matrix *h, int items, int kind, cudaStream_t s) {
    SegScratch &g = h->seg;
    const int64_t nnz = kind != SEG_COO ? h->nnz : (h->cfg.format == SPMV_FMT_HYB ? h->hyb_nnz : h->nnz);
    const int C = 32 * items;
    const int64_t nchunks = (nnz + C - 1) / C;
    auto f = [](void *p) { dev_free(p); };
    f(g.meta0); f(g.meta1);
    free_partials(&g.part);
    g = SegScratch{};
    g.items = items;
    g.nchunks = nchunks;
    SPMV_TRY(dalloc(&g.meta0, (size_t)nchunks + 1));
    SPMV_TRY(dalloc(&g.meta1, (size_t)nchunks + 1));
    SPMV_TRY(alloc_partials(&g.part, nchunks, 1, h->vt, s));
    if (nchunks > 0) {
        unsigned grid = grid1d(nchunks + 1, 256);
        if (kind == SEG_TILES) {
            k_seg_meta_split<<<grid, 256, 0, s>>>(h->rowptr, h->m, nnz, C, nchunks, g.meta0);
        } else if (kind == SEG_MERGE) {
            k_seg_meta_merge<<<grid, 256, 0, s>>>(h->rowptr, h->m, C, nchunks, g.meta0);
        } else if (h->cfg.format == SPMV_FMT_HYB) {
            k_seg_meta_coo<<<grid, 256, 0, s>>>(h->hyb_rows, h->hyb_ptr, nnz, C, nchunks, g.meta0, g.meta1);
        } else {
            k_seg_meta_coo<<<grid, 256, 0, s>>>(h->coo_rows, h->rowptr, nnz, C, nchunks, g.meta0, g.meta1);
        }
        SPMV_CUDA_TRY(cudaGetLastError());
    }
    return SPMV_OK;
}

int pack_format(spmv_matrix *h, const spmv_config &cfg, cudaStream_t s) {
    // a solver graph captured the old launches
    free_cg(h);
    // a change of launch parameters only (block size, register cap, carveout)
    // keeps the packed arrays
    const spmv_config &p = h->packed_req;
    if (h->packed && p.format == cfg.format && p.threads_per_row == cfg.threads_per_row &&
        p.unroll == cfg.unroll && p.bsr_block == cfg.bsr_block && p.hyb_ell_width == cfg.hyb_ell_width) {
        const int32_t width = h->cfg.hyb_ell_width;
        h->cfg = cfg;
        if (cfg.format == SPMV_FMT_HYB) h->cfg.hyb_ell_width = width;
        return SPMV_OK;
    }
    free_packed(h);
    h->packed = false;
    h->packed_req = cfg;
    h->cfg = cfg;
    const int items = 4 * (cfg.unroll > 4 ? 4 : cfg.unroll);  // COO parts: at most 16 entries per lane
    switch (cfg.format) {
    case SPMV_FMT_CSR:
        if (cfg.threads_per_row == SPMV_TPR_SPLIT) {
            // hyb_ell_width 0: warp chunks of 32 * items entries; else staged
            // tiles of hyb_ell_width nonzeros (a multiple of 256)
            if (cfg.hyb_ell_width == 0) SPMV_TRY(ensure_seg_scratch(h, items, SEG_MERGE, s));
            else SPMV_TRY(ensure_seg_scratch(h, cfg.hyb_ell_width / 32, SEG_TILES, s));
        } else {
            // rows needing more than 32 steps of their lane group go to whole blocks (uneven rows
            // with one or two lanes: to warps)
            const bool uneven = csr_uneven(h, cfg.threads_per_row);
            const int64_t thr =
                uneven ? CSR_WARP_ROW : std::max<int64_t>(512, 32LL * cfg.threads_per_row * cfg.unroll);
            SPMV_TRY(build_long_rows(h, h->rowptr, h->m, h->max_row, thr, uneven ? CSR_SEG_LEN : 4096, 1, s));
        }
        break;
    case SPMV_FMT_ELL: {
        const int64_t width = h->max_row;
        const int64_t pitch = (h->m + 31) / 32 * 32;
        if ((double)width * (double)pitch > 8.0 * (double)h->nnz + (double)(1 << 24)) {
            set_error("ELL: padded size %lld x %lld exceeds 8 x nnz + 2^24 entries", (long long)width,
                      (long long)pitch);
            return SPMV_ERR_UNSUPPORTED;
        }
        SPMV_TRY(pack_ell(h, width, s));
        break;
    }
    case SPMV_FMT_COO:
        SPMV_TRY(dalloc(&h->coo_rows, (size_t)h->nnz));
        SPMV_TRY(expand_rows(h->rowptr, h->m, h->nnz, h->coo_rows, s));
        SPMV_TRY(ensure_seg_scratch(h, items, SEG_COO, s));
        break;
    case SPMV_FMT_HYB: {
        int64_t width = cfg.hyb_ell_width;
        if (width <= 0) SPMV_TRY(hyb_width_rule(h, s, &width));
        width = std::min<int64_t>(width, h->max_row);
        SPMV_TRY(pack_hyb(h, width, s));
        h->cfg.hyb_ell_width = (int32_t)width;
        SPMV_TRY(ensure_seg_scratch(h, items, SEG_COO, s));
        break;
    }
    case SPMV_FMT_SELL:
        SPMV_TRY(pack_sell(h, cfg.hyb_ell_width, cfg.bsr_block == 4, s));
        break;
    case SPMV_FMT_BSR: {
        SPMV_TRY(pack_bsr(h, cfg.bsr_block, s));
        const int64_t thr = 256LL * cfg.threads_per_row;
        // a block row holds at most the entries of its rows
        SPMV_TRY(build_long_rows(h, h->bsr_rowptr, h->bsr_mb, cfg.bsr_block * h->max_row, thr, 16LL * (256 / cfg.bsr_block), cfg.bsr_block, s));
        break;
    }
    default:
        set_error("unknown format %d", cfg.format);
        return SPMV_ERR_INVALID;
    }
    SPMV_CUDA_TRY(cudaStreamSynchronize(s));
    h->packed = true;
    return SPMV_OK;
}

}  // namespace spmv
