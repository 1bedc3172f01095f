// Sparsity features on the device (Table 2, Section 5.5: n, nnz, Avg_nnz,
// Var_nnz, ELL_ratio, Median, Mode, Std_nnz) plus the selector's structural
// extras, and the fused inference kernel of the 2-layer selector MLP
// (Section 5.4: a multi-class classifier over the features).
//
// The paper extracts features on the CPU with NumPy (Section 7.5 reports
// seconds per matrix); here a few kernels read the CSR arrays once:
//   k_feat_rows     row lengths: sum of squares, min, max, empty rows and a
//                   histogram of lengths;
//   k_feat_groups   block rows of four rows, one lane each merging their
//                   columns: |i - j| (max and sum), diagonal entries and the
//                   nonempty 2x2 / 4x4 blocks;
//   k_feat_heavy    the same for block rows too long for one lane;
//   k_feat_finish   one block: median, mode, Gini and the HYB width from the
//                   histogram, then the 20 feature values.
// Counts are exact 64-bit integers; ratios are formed once at the end.
#include <algorithm>
#include <cmath>

#include "internal.cuh"

namespace spmv {

namespace {

constexpr unsigned FULL = 0xffffffffu;

__device__ __forceinline__ unsigned long long warp_sum_u64(unsigned long long v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(FULL, v, o);
    return v;  // valid in lane 0
}

struct FeatAcc {
    unsigned long long sum_len2;   // sum of squared row lengths
    unsigned long long empty;      // rows of length 0
    unsigned long long sum_dist;   // sum |i - j|
    unsigned long long diag;       // entries with i == j
    unsigned long long blocks4;    // nonempty 4x4 blocks
    unsigned long long blocks2;    // nonempty 2x2 blocks
    int min_gap, max_len, max_dist;  // min_gap: 2^31 - 1 minus the shortest row, so that zero starts every field
    unsigned list_len;               // entries of the list of heavy block rows (one panel's)
};

// Row lengths.  A matrix has few distinct lengths, so a histogram of global
// atomics makes every warp queue on the same few words (random rows of mean
// 16, 2^20 rows: 86 us, of which 2 us are the 4 MB read).  Lengths below
// ROW_BINS are counted in shared memory and added once per thread block; the
// grid is one block per SM, so a bin receives at most one global atomic per
// SM.
constexpr int ROW_BINS = 4096, ROW_THREADS = 1024;

__global__ void __launch_bounds__(ROW_THREADS) k_feat_rows(const int *rowptr, int64_t m, unsigned *hist, FeatAcc *acc) {
    __shared__ unsigned sh[ROW_BINS];
    for (int i = threadIdx.x; i < ROW_BINS; i += ROW_THREADS) sh[i] = 0;
    __syncthreads();
    unsigned long long s2 = 0, emp = 0;
    int mn = 0x7fffffff, mx = 0;
    const int lane = threadIdx.x & 31;
    const int64_t stride = (int64_t)gridDim.x * ROW_THREADS;
    const int64_t mr = (m + 31) / 32 * 32;
    for (int64_t r = (int64_t)blockIdx.x * ROW_THREADS + threadIdx.x; r < mr; r += stride) {
        const bool valid = r < m;
        const int len = valid ? rowptr[r + 1] - rowptr[r] : -1;
        if (valid) {
            s2 += (unsigned long long)len * (unsigned long long)len;
            emp += len == 0;
            mn = min(mn, len);
            mx = max(mx, len);
        }
        const unsigned peers = __match_any_sync(FULL, len);
        if (valid && lane == 31 - __clz(peers)) {
            if (len < ROW_BINS) atomicAdd(&sh[len], (unsigned)__popc(peers));
            else atomicAdd(hist + len, (unsigned)__popc(peers));
        }
    }
    s2 = warp_sum_u64(s2);
    emp = warp_sum_u64(emp);
    mn = __reduce_min_sync(FULL, mn);
    mx = __reduce_max_sync(FULL, mx);
    __shared__ unsigned long long s_s2[ROW_THREADS / 32], s_emp[ROW_THREADS / 32];
    __shared__ int s_mn[ROW_THREADS / 32], s_mx[ROW_THREADS / 32];
    if (lane == 0) {
        s_s2[threadIdx.x >> 5] = s2;
        s_emp[threadIdx.x >> 5] = emp;
        s_mn[threadIdx.x >> 5] = mn;
        s_mx[threadIdx.x >> 5] = mx;
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        s2 = warp_sum_u64(s_s2[lane]);
        emp = warp_sum_u64(s_emp[lane]);
        mn = __reduce_min_sync(FULL, s_mn[lane]);
        mx = __reduce_max_sync(FULL, s_mx[lane]);
        if (lane == 0) {
            atomicAdd(&acc->sum_len2, s2);
            atomicAdd(&acc->empty, emp);
            atomicMax(&acc->min_gap, 0x7fffffff - mn);
            atomicMax(&acc->max_len, mx);
        }
    }
    // a counted bin is the length of a row, so it is at most the histogram's last
    for (int i = threadIdx.x; i < ROW_BINS; i += ROW_THREADS)
        if (sh[i]) atomicAdd(hist + i, sh[i]);
}

// Per nonzero: |i - j|, the diagonal, and how many r x r blocks (r = 2, 4)
// hold an entry.  Rows come in block rows of four (row0, the global index of
// local row 0, is a multiple of 4 for row panels).
//
// One lane merges the four ascending column lists of a block row: a step
// takes the smallest column among the four heads, consumes it from every row
// that holds it, and opens a 4 x 4 (2 x 2) block when its column block
// differs from the last one taken (by the same pair of rows).  So a step
// costs the same few instructions whatever the structure, and a step per
// distinct column of the block row is enough.  The columns of a warp's block
// rows are contiguous in CSR and are staged in shared memory with coalesced
// loads (ranges that do not fit are read in place); where 32 block rows of
// mean length do not fit, several lanes split the columns of each.  Finding
// each entry's row and blocks by binary searches was bound by some 25
// dependent loads per entry: 450 us on random rows of mean 16 (2^20 rows),
// 102 now, bound by issue (half the slots) at the 20 warps per SM that the
// staging leaves room for.  A whole selection on a band of half-width 60
// (380,000 rows, 46M entries) went from 887 to 195 us.
//
// A block row of more than `heavy` entries would hold up its warp: it is
// listed for k_feat_heavy, once per 32 of its ranges.
constexpr int FEAT_CAP = 4096;  // most staged entries per warp (one warp per thread block)
constexpr int FEAT_WARPS = 8;   // warps per SM below which a block row gets more lanes
constexpr int UNEVEN_LANES = 4;
constexpr int HEAVY_MIN = 256, HEAVY_MAX = 4096;
constexpr int HEAVY_THREADS = 128, HEAVY_STRIDE = 32;

// pivots of a row of `len` entries in a heavy block row (k_feat_heavy)
__device__ __forceinline__ int heavy_pivots(int len) {
    return (int)(((unsigned)len + HEAVY_STRIDE - 1) / HEAVY_STRIDE);
}

// sums of one warp into the accumulators
__device__ __forceinline__ void feat_add(FeatAcc *acc, unsigned long long sd, unsigned dg, unsigned b4, unsigned b2,
                                         int md) {
    sd = warp_sum_u64(sd);
    dg = __reduce_add_sync(FULL, dg);
    b4 = __reduce_add_sync(FULL, b4);
    b2 = __reduce_add_sync(FULL, b2);
    md = __reduce_max_sync(FULL, md);
    if ((threadIdx.x & 31) == 0) {
        if (sd) atomicAdd(&acc->sum_dist, sd);
        if (dg) atomicAdd(&acc->diag, (unsigned long long)dg);
        if (b4) atomicAdd(&acc->blocks4, (unsigned long long)b4);
        if (b2) atomicAdd(&acc->blocks2, (unsigned long long)b2);
        if (md) atomicMax(&acc->max_dist, md);
    }
}

// one block row, or a lane's range of its columns (whole 4-column blocks):
// rows gi .. gi + 3 at entries [k[q], e[q]), columns by col(k)
template <typename Col>
__device__ __forceinline__ void merge_group(Col col, int (&k)[4], const int (&e)[4], int64_t gi, unsigned long long &sd, unsigned &dg,
                                            unsigned &b4, unsigned &b2, int &md) {
    constexpr int NONE = 0x7fffffff;  // a column is below 2^31 - 1
    // distances row by row (a step of the merge would carry four of them)
    int j[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int i = (int)gi + q;
        unsigned far = 0;
        if (k[q] < e[q])  // columns ascend: the ends are the farthest entries
            far = max((unsigned)abs(i - col(k[q])), (unsigned)abs(i - col(e[q] - 1)));
        md = max(md, (int)far);
        if (far < (1u << 20)) {  // at most HEAVY_MAX = 2^12 of them: the sum fits in 32 bits
            unsigned sum = 0;
#pragma unroll 4
            for (int t = k[q]; t < e[q]; ++t) {
                const unsigned d = (unsigned)abs(i - col(t));
                sum += d;
                dg += d == 0;
            }
            sd += sum;
        } else {
            for (int t = k[q]; t < e[q]; ++t) {
                const unsigned d = (unsigned)abs(i - col(t));
                sd += d;
                dg += d == 0;
            }
        }
        j[q] = k[q] < e[q] ? col(k[q]) : NONE;
    }
    int last = -4, lasta = -4, lastb = -4;
    for (;;) {
        const int c = min(min(j[0], j[1]), min(j[2], j[3]));
        if (c == NONE) break;
        bool hit[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) hit[q] = j[q] == c;
        b4 += ((c ^ last) >> 2) != 0;
        last = c;
        const bool up = hit[0] || hit[1], down = hit[2] || hit[3];
        b2 += up && ((c ^ lasta) >> 1) != 0;
        b2 += down && ((c ^ lastb) >> 1) != 0;
        lasta = up ? c : lasta;
        lastb = down ? c : lastb;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            k[q] += hit[q];
            if (hit[q]) j[q] = NONE;
            if (hit[q] && k[q] < e[q]) j[q] = col(k[q]);
        }
    }
}

// the walk of one lane, `sub` of the `lpg` lanes of block row g (entries b[0]
// .. b[4]): the lanes split the columns at quantiles of the longest row,
// rounded down to whole 4-column blocks
template <typename Col>
__device__ __forceinline__ void walk_group(Col col, const int (&b)[5], bool walk, int sub, int lpg, int64_t gi,
                                           unsigned long long &sd, unsigned &dg, unsigned &b4, unsigned &b2, int &md) {
    int k[4], e[4];
    if (lpg == 1) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            k[q] = b[q];
            e[q] = b[q + 1];
        }
    } else {
        int ls = b[0], len = b[1] - b[0];
#pragma unroll
        for (int q = 1; q < 4; ++q)
            if (b[q + 1] - b[q] > len) {
                ls = b[q];
                len = b[q + 1] - b[q];
            }
        const int from = walk && sub > 0 && len > 0 ? col(ls + (int)((unsigned)(len * sub) / (unsigned)lpg)) & ~3 : 0;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            int lo = b[q], hi = walk && sub > 0 ? b[q + 1] : lo;  // first entry of the row at or after column `from`
            while (lo < hi) {
                const int mid = lo + ((hi - lo) >> 1);
                if (col(mid) < from) lo = mid + 1; else hi = mid;
            }
            k[q] = lo;
            const int next = __shfl_down_sync(FULL, lo, 1);
            e[q] = sub == lpg - 1 ? b[q + 1] : next;
        }
    }
    if (walk) merge_group(col, k, e, gi, sd, dg, b4, b2, md);
}

// lpg: lanes per block row (a power of two); cap: entries the dynamic shared
// memory holds besides 32 words for the block rows' shifts
__global__ void __launch_bounds__(32)
k_feat_groups(const int *__restrict__ rowptr, const int *__restrict__ colidx, int64_t m, int64_t row0, int heavy, int cap,
              int lpg, int2 *list, unsigned *list_len, FeatAcc *acc) {
    extern __shared__ int sc[];
    const int lane = threadIdx.x;
    const int gpw = 32 / lpg, sub = lane & (lpg - 1), mine = lane / lpg;  // block rows per warp, this lane's
    const int64_t ngroups = (m + 3) / 4;
    unsigned long long sd = 0;
    unsigned dg = 0, b4 = 0, b2 = 0;
    int md = 0;
    for (int64_t g0 = (int64_t)blockIdx.x * gpw; g0 < ngroups; g0 += (int64_t)gridDim.x * gpw) {
        const int64_t g = g0 + mine;
        int b[5];
#pragma unroll
        for (int q = 0; q < 5; ++q) {  // rows past m are empty
            const int64_t r = 4 * g + q;
            b[q] = __ldg(rowptr + (r < m ? r : m));
        }
        const int w0 = __shfl_sync(FULL, b[0], 0), w1 = __shfl_sync(FULL, b[4], 31);
        const bool staged = w1 - w0 <= cap;
        __syncwarp();  // the walks of the previous block rows are done
        if (staged) {
            // block row l is shifted by l words, so that the lanes' walks through
            // rows of one length start on different banks
#pragma unroll 4
            for (int l = 0; l < gpw; ++l) {
                const int s = __shfl_sync(FULL, b[0], l * lpg), e = __shfl_sync(FULL, b[4], l * lpg);
                for (int k = s + lane; k < e; k += 32) sc[k - w0 + l] = __ldg(colidx + k);
            }
        }
        __syncwarp();
        const int cnt = b[4] - b[0];
        if (cnt > heavy && sub == 0) {
            int pivots = 0;
#pragma unroll
            for (int q = 0; q < 4; ++q) pivots += heavy_pivots(b[q + 1] - b[q]);
            const int nt = (pivots + 31) / 32;
            const unsigned at = atomicAdd(list_len, (unsigned)nt);
            for (int t = 0; t < nt; ++t) list[at + t] = make_int2((int)g, t);
        }
        const bool walk = cnt <= heavy;
        if (staged)
            walk_group([&](int k) { return sc[k - w0 + mine]; }, b, walk, sub, lpg, row0 + 4 * g, sd, dg, b4, b2, md);
        else
            walk_group([&](int k) { return __ldg(colidx + k); }, b, walk, sub, lpg, row0 + 4 * g, sd, dg, b4, b2, md);
    }
    __syncwarp();
    feat_add(acc, sd, dg, b4, b2, md);
}

// The listed heavy block rows, cut into column ranges of a lane each.  Every
// HEAVY_STRIDE-th entry of each row is a pivot, its column rounded down to a
// whole 4-column block; a range starts at a pivot and ends at the next larger
// one of any row, so it holds at most HEAVY_STRIDE + 3 entries of a row however
// the rows' columns are spread.  The lane of a pivot finds its range by one
// search per row (the four rows' searches run together) and merges it as
// k_feat_groups does; where rows share a pivot the first row's lane takes it.
// With a thread per 8 consecutive entries looking up the earlier rows for each
// it took 57 us on an R-MAT matrix of scale 17 (a = 0.64), 22 now; whole
// selection of scale 19 (a = 0.57) 392 and 248.
__global__ void __launch_bounds__(HEAVY_THREADS)
k_feat_heavy(const int *__restrict__ rowptr, const int *__restrict__ colidx, int64_t m, int64_t row0,
             const int2 *list, const unsigned *list_len, FeatAcc *acc) {
    constexpr int S = HEAVY_STRIDE, NONE = 0x7fffffff;
    unsigned long long sd = 0;
    unsigned dg = 0, b4 = 0, b2 = 0;
    int md = 0;
    const unsigned n = *list_len;
    const unsigned warp = (blockIdx.x * HEAVY_THREADS + threadIdx.x) >> 5, warps = gridDim.x * (HEAVY_THREADS / 32);
    auto col = [&](int k) { return __ldg(colidx + k); };
    for (unsigned it = warp; it < n; it += warps) {
        const int2 item = list[it];
        int b[5];
#pragma unroll
        for (int q = 0; q < 5; ++q) {
            const int64_t r = 4 * (int64_t)item.x + q;
            b[q] = __ldg(rowptr + (r < m ? r : m));
        }
        // this lane's pivot: entry own * S of row `row`
        int own = item.y * 32 + (threadIdx.x & 31), row = 0;
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const int pivots = heavy_pivots(b[q + 1] - b[q]);
            if (row == q && own >= pivots) {
                own -= pivots;
                row = q + 1;
            }
        }
        const int rb = row == 0 ? b[0] : row == 1 ? b[1] : row == 2 ? b[2] : b[3];
        const int re = row == 0 ? b[1] : row == 1 ? b[2] : row == 2 ? b[3] : b[4];
        if (own >= heavy_pivots(re - rb)) continue;  // past the last row's pivots
        const int from = col(rb + own * S) & ~3;
        // first entry of each row at or after column `from`
        int k[4], e[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            k[q] = b[q];
            e[q] = b[q + 1];
        }
        while (k[0] < e[0] || k[1] < e[1] || k[2] < e[2] || k[3] < e[3]) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int mid = k[q] + ((e[q] - k[q]) >> 1);
                if (k[q] < e[q]) {
                    if (col(mid) < from) k[q] = mid + 1; else e[q] = mid;
                }
            }
        }
        // the next pivot of any row, and whether an earlier row holds this one
        int next = NONE;
        bool mine = true;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            // pivot entry at or after the range's start (offsets in the row: b + S may pass 2^31)
            const int at = heavy_pivots(k[q] - b[q]), all = heavy_pivots(b[q + 1] - b[q]);
            int c = at < all ? col(b[q] + at * S) & ~3 : NONE;
            if (c == from) {
                mine = mine && q >= row;
                c = at + 1 < all ? col(b[q] + (at + 1) * S) & ~3 : NONE;
            }
            next = min(next, c);
        }
        if (!mine) continue;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            int lo = k[q], hi = k[q] + min(b[q + 1] - k[q], S + 3);
            while (lo < hi) {
                const int mid = lo + ((hi - lo) >> 1);
                if (col(mid) < next) lo = mid + 1; else hi = mid;
            }
            e[q] = lo;
        }
        merge_group(col, k, e, row0 + 4 * (int64_t)item.x, sd, dg, b4, b2, md);
    }
    __syncwarp();
    feat_add(acc, sd, dg, b4, b2, md);
}

constexpr int FIN_THREADS = 1024;

constexpr int FIN_ITEMS = 8;  // histogram bins per thread and step

// fixed-order sums over the block of two values; results valid in every thread
__device__ void block_sum2_ll(long long &a, long long &b, long long (*sh)[FIN_THREADS / 32]) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_down_sync(FULL, a, o);
        b += __shfl_down_sync(FULL, b, o);
    }
    __syncthreads();
    if (lane == 0) {
        sh[0][w] = a;
        sh[1][w] = b;
    }
    __syncthreads();
    a = sh[0][lane];
    b = sh[1][lane];
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_xor_sync(FULL, a, o);
        b += __shfl_xor_sync(FULL, b, o);
    }
}

// Single block over the histogram h[0..maxlen]: P(L) = #rows shorter than L.
// One block, so its time is the latency of its steps: a thread takes
// FIN_ITEMS bins a step (power-law matrices have 10^5 bins), and the feature
// values, each an fp64 division or two, are formed by one warp each.
__global__ void __launch_bounds__(FIN_THREADS)
k_feat_finish(const unsigned *hist, int maxlen, int64_t m, int64_t n, int64_t nnz, const FeatAcc *acc,
              double *out) {
    __shared__ long long sh[2][FIN_THREADS / 32];
    __shared__ long long median_s;
    __shared__ unsigned long long mode_key_s, K_s;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    if (tid == 0) {
        median_s = 0;
        mode_key_s = 0ull;
        K_s = 0ull;
    }
    const long long target = (m - 1) / 2;  // 0-based index of the lower middle
    long long gini_num = 0, carry = 0;     // carry: rows in the bins of earlier steps
    unsigned long long mode_key = 0ull, K_best = 0ull;
    for (int64_t base = 0; base <= maxlen; base += FIN_THREADS * FIN_ITEMS) {
        const int64_t L0 = base + (int64_t)tid * FIN_ITEMS;
        unsigned h[FIN_ITEMS];
        long long mine = 0;
#pragma unroll
        for (int u = 0; u < FIN_ITEMS; ++u) {
            h[u] = L0 + u <= maxlen ? hist[L0 + u] : 0u;
            mine += h[u];
        }
        // exclusive prefix over the step
        long long incl = mine;
        for (int o = 1; o < 32; o <<= 1) {
            const long long t = __shfl_up_sync(FULL, incl, o);
            if (lane >= o) incl += t;
        }
        __syncthreads();  // the previous step's totals are read
        if (lane == 31) sh[0][w] = incl;
        __syncthreads();
        long long tot = sh[0][lane], winc = tot;
        for (int o = 1; o < 32; o <<= 1) {
            const long long t = __shfl_up_sync(FULL, winc, o);
            if (lane >= o) winc += t;
        }
        long long P = carry + __shfl_sync(FULL, winc - tot, w) + incl - mine;  // rows shorter than L0
        carry += __shfl_sync(FULL, winc, 31);
#pragma unroll
        for (int u = 0; u < FIN_ITEMS; ++u) {
            const long long L = L0 + u, c = h[u];
            if (L <= maxlen) {
                if (c > 0) {
                    if (P <= target && target < P + c) median_s = L;
                    // mode: largest count, smallest length on ties (64-bit key)
                    const unsigned long long key = ((unsigned long long)c << 32) | (unsigned)(0x7fffffff - (int)L);
                    mode_key = key > mode_key ? key : mode_key;
                }
                gini_num += L * c * (2 * P + c - m);
                // HYB width: rows with length >= L is m - P
                const long long ge = m - P;
                if (L >= 1 && ge >= 4096 && 3 * ge >= m) K_best = (unsigned long long)L;
            }
            P += c;
        }
    }
    __syncthreads();
    if (mode_key) atomicMax(&mode_key_s, mode_key);
    if (K_best) atomicMax(&K_s, K_best);
    __syncthreads();
    const long long K = (long long)K_s;
    long long tail = 0;
    for (int64_t base = 0; base <= maxlen; base += FIN_THREADS * FIN_ITEMS) {
        const int64_t L0 = base + (int64_t)tid * FIN_ITEMS;
#pragma unroll
        for (int u = 0; u < FIN_ITEMS; ++u)
            if (L0 + u <= maxlen && L0 + u > K) tail += (L0 + u - K) * (long long)hist[L0 + u];
    }
    block_sum2_ll(gini_num, tail, sh);
    if (lane != 0) return;
    const double md = (double)m, nd = (double)n, zd = (double)nnz;
    const double mean = m ? zd / md : 0.0;
    // population variance from the exact integer numerator sum(l^2) m - nnz^2
    auto variance = [&]() {
        const __int128 num = (__int128)acc->sum_len2 * m - (__int128)nnz * nnz;
        return m ? (double)num / (md * md) : 0.0;
    };
    auto deviation = [&]() {
        const double var = variance();
        return sqrt(var > 0 ? var : 0.0);
    };
    double v = 0.0;
    switch (w) {
    case 0: v = md; break;
    case 1: v = zd; break;
    case 2: v = (m && n) ? zd / (md * nd) : 0.0; break;
    case 3: v = mean; break;
    case 4: v = variance(); break;
    case 5: v = deviation(); break;
    case 6: v = m ? (double)(0x7fffffff - acc->min_gap) : 0.0; break;
    case 7: v = (double)acc->max_len; break;
    case 8: v = (double)median_s; break;
    case 9: v = mode_key_s ? (double)(0x7fffffff - (long long)(mode_key_s & 0xffffffffull)) : 0.0; break;
    case 10: v = (m && acc->max_len) ? zd / (md * (double)acc->max_len) : 0.0; break;
    case 11: v = (m && nnz) ? (double)gini_num / (md * zd) : 0.0; break;
    case 12: v = mean > 0 ? deviation() / mean : 0.0; break;
    case 13: v = m ? (double)acc->empty / md : 0.0; break;
    case 14: v = (double)acc->max_dist; break;
    case 15: v = nnz ? (double)acc->sum_dist / zd : 0.0; break;
    case 16: v = nnz ? (double)acc->diag / zd : 0.0; break;
    case 17: v = nnz ? zd / (16.0 * (double)acc->blocks4) : 0.0; break;
    case 18: v = nnz ? zd / (4.0 * (double)acc->blocks2) : 0.0; break;
    case 19: v = nnz ? (double)tail / zd : 0.0; break;
    default: return;
    }
    out[w] = v;
}

}  // namespace

// Features of the handle's matrix into d_out[SPMV_NUM_FEATURES] (device).
int compute_features(const spmv_matrix *h, double *d_out, cudaStream_t s) {
    const int64_t m = h->m;
    const int maxlen = (int)h->max_row;
    void *buf = nullptr;
    // histogram, accumulators, list of heavy block rows (one panel's at a time): one has
    const int np = h->npanels > 0 ? h->npanels : 1;
    int64_t most = 0;
    for (int p = 0; p < np; ++p) most = std::max(most, h->npanels > 0 ? h->panels[p]->nnz : h->nnz);
    const size_t hist_bytes = (sizeof(unsigned) * ((size_t)maxlen + 1) + 127) / 128 * 128;
    // cnt > HEAVY_MIN entries, listed at most cnt / (32 HEAVY_STRIDE) + 2 times
    const size_t list_bytes = sizeof(int2) * (size_t)(2 * (most / HEAVY_MIN) + most / (32 * HEAVY_STRIDE) + 1);
    SPMV_CUDA_TRY(dev_malloc_async(&buf, hist_bytes + 128 + list_bytes, s));
    unsigned *hist = static_cast<unsigned *>(buf);
    FeatAcc *acc = reinterpret_cast<FeatAcc *>(static_cast<char *>(buf) + hist_bytes);
    int2 *list = reinterpret_cast<int2 *>(static_cast<char *>(buf) + hist_bytes + 128);
    int st = SPMV_OK;
    cudaError_t e = cudaMemsetAsync(buf, 0, hist_bytes + 128, s);
    if (e == cudaSuccess) {
        // a matrix held in row panels accumulates every panel into one set
        const int64_t sms = h->sm_count > 0 ? h->sm_count : 152;
        for (int p = 0; p < np && e == cudaSuccess; ++p) {
            const spmv_matrix *q = h->npanels > 0 ? h->panels[p] : h;
            const int64_t row0 = h->npanels > 0 ? h->panel_row0[p] : 0;
            const int64_t mq = q->m;
            if (mq == 0) continue;
            const int64_t rb = (mq + ROW_THREADS - 1) / ROW_THREADS;
            k_feat_rows<<<(unsigned)(rb < sms ? rb : sms), ROW_THREADS, 0, s>>>(q->rowptr, mq, hist, acc);
            if (q->nnz == 0) continue;
            if (p > 0) e = cudaMemsetAsync(&acc->list_len, 0, sizeof(unsigned), s);
            // heavy: over four mean block rows, within [HEAVY_MIN, HEAVY_MAX]: uniform rows stay with
            // the merge, and a warp does not last far longer than the others
            const double mean4 = 4.0 * (double)q->nnz / (double)mq;
            const int heavy = (int)std::min<double>(HEAVY_MAX, std::max<double>(HEAVY_MIN, 4.0 * mean4));
            // lanes per block row: enough that the warp's block rows fit in the staging (the mean and
            // an eighth more; shared memory sets the warps per SM)
            const int64_t ngroups = (mq + 3) / 4;
            int lpg = 1;
            while (lpg < 32 && 36.0 / lpg * mean4 + 64.0 > FEAT_CAP) lpg *= 2;
            // ... and, while the chip is not full of warps, more of them with a shorter walk each
            // (Poisson(22) of 1756 rows: 85 us a selection with one lane, 63 now)
            while (lpg < 32 && ngroups * lpg < 32 * FEAT_WARPS * sms && mean4 >= 8.0 * lpg) lpg *= 2;
            // ... or where the longest row of most 32-row groups is far above the mean: a warp is done
            // when its longest walk is (R-MAT scale 19, whole selection: 248 us with one lane, 204,
            // 197, 213 with 2, 4, 8)
            if (csr_uneven(q, 1)) lpg = std::max(lpg, UNEVEN_LANES);
            const int cap = (int)std::min<double>(FEAT_CAP, 128.0 * std::ceil((36.0 / lpg * mean4 + 64.0) / 128.0));
            const int64_t wb = (ngroups + 32 / lpg - 1) / (32 / lpg);
            k_feat_groups<<<(unsigned)(wb < 64 * sms ? wb : 64 * sms), 32, sizeof(int) * (size_t)(cap + 32), s>>>(
                q->rowptr, q->colidx, mq, row0, heavy, cap, lpg, list, &acc->list_len, acc);
            // (a block row holds at most four times the longest row)
            if (4 * h->max_row > heavy)
                k_feat_heavy<<<(unsigned)(8 * sms), HEAVY_THREADS, 0, s>>>(q->rowptr, q->colidx, mq, row0, list,
                                                                           &acc->list_len, acc);
        }
        k_feat_finish<<<1, FIN_THREADS, 0, s>>>(hist, maxlen, m, h->n, h->nnz, acc, d_out);
        if (e == cudaSuccess) e = cudaGetLastError();
    }
    if (e != cudaSuccess) st = cuda_status(e, "feature kernels");
    cudaFreeAsync(buf, s);
    return st;
}

}  // namespace spmv
