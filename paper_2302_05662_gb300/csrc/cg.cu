// Conjugate gradients on the device with the handle's SpMV (spmv_cg).
//
// Section 7.5 of the paper names preconditioned CG as the iterative setting
// in which one matrix is multiplied many times, so that feature extraction,
// selection and conversion are paid once.  The iteration is Hestenes and
// Stiefel's (1952):
//
//   r0 = b - A x0, p0 = r0, rho_k = r_k.r_k
//   while k < maxit and rho_k > tol^2 (b.b):
//     q = A p_k; alpha = rho_k / (p_k.q)          (stop on p_k.q <= 0)
//     x_{k+1} = x_k + alpha p_k; r_{k+1} = r_k - alpha q
//     beta = rho_{k+1} / rho_k; p_{k+1} = r_{k+1} + beta p_k
//
// GB300 layout of the loop: the whole solve is one launch, and the device
// alone decides when to stop, so no iteration waits for the host.  There are
// two forms.
//
// Graph (any size): a prologue forms r0, p0, rho_0 and b.b; a WHILE
// conditional node repeats the body
//   SpMV (the handle's format) -> p.q, alpha -> r update, r.r, beta, stop
//   -> x and p updates.
// The thread block that finishes a dot product last sums the blocks'
// partials in block order and leaves the scalar the next kernel reads, and x
// is updated where p is read anyway: eight vector passes in three kernels,
// against eleven in four when every block summed the partials for itself
// (27-point Laplacian 128^3, fp64, per iteration besides the product: 58 us
// then, 40 now, of which the vector passes' bytes take 25 at the HBM rate).
//
// Cluster (small systems, see cluster_fits): one thread-block cluster keeps
// x, r, p and q on the SMs for the whole solve and replaces kernel
// boundaries by cluster barriers.
//
// Every dot product is a fixed-shape reduction in fp64, so results are
// bit-reproducible and every block sees the same alpha and beta.  fp64 vector
// updates are fused multiply-adds, fp32 ones round the product and the sum.
//
// Termination does not depend on the reductions: the iteration counter grows
// on every pass and the loop ends once it reaches maxit.

#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <type_traits>

#include "internal.cuh"

namespace spmv {

namespace {

constexpr int CG_THREADS = 512;  // two blocks per SM

struct CgState {
    double rho, stop, bb, alpha, beta;
    int32_t iter, maxit, converged, breakdown;
    unsigned done;  // thread blocks that have left their partial of the running dot product
};

// Sum of N partials in shared memory by one whole warp, every lane returning
// it, in one fixed order.  On this GPU an SM issues one fp64 warp instruction
// per 16 cycles and a dependent one waits 64, so sums are made by one warp
// (a shuffle tree in every warp costs as many fp64 instructions per warp) and
// as trees.
template <int N>
__device__ __forceinline__ double warp_sum_shared(const double *v) {
    static_assert(N % 128 == 0, "");
    const int lane = threadIdx.x & 31;
    double a[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
    for (int i = 0; i < N / 128; ++i)
#pragma unroll
        for (int u = 0; u < 4; ++u) a[u] += v[128 * i + 32 * u + lane];
    double t = (a[0] + a[1]) + (a[2] + a[3]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    return t;
}

// fixed-order sum over the block (every block with the same inputs returns
// the same value); result valid in every thread
__device__ double block_sum(double v) {
    __shared__ double s_v[CG_THREADS];
    __shared__ double s_total;
    __syncthreads();  // the last sum's values are read
    s_v[threadIdx.x] = v;
    __syncthreads();
    if (threadIdx.x < 32) {
        const double t = warp_sum_shared<CG_THREADS>(s_v);
        if (threadIdx.x == 0) s_total = t;
    }
    __syncthreads();
    return s_total;
}

// sum of part[0..n) in one fixed order, identical in every block
__device__ double sum_parts(const double *part, int n) {
    double v = 0.0;
    for (int i = threadIdx.x; i < n; i += CG_THREADS) v += part[i];
    return block_sum(v);
}

__device__ __forceinline__ double wide(double v) { return v; }
__device__ __forceinline__ double wide(float v) { return (double)v; }

// a + s*b.  fp64: rounded once, one instruction where a product and a sum are
// two (the vector updates of a large fp64 solve are bound by them, not by HBM).
// fp32: the product and the sum rounded separately, so that the fp64 history
// of r.r stays the one this iteration has always written (fused, it moves in
// the seventh digit; nothing is gained, fp32 instructions are not scarce).
__device__ __forceinline__ double axpy1(double a, double s, double b) { return fma(s, b, a); }
__device__ __forceinline__ float axpy1(float a, float s, float b) { return __fadd_rn(a, __fmul_rn(s, b)); }

template <typename T>
__global__ void __launch_bounds__(CG_THREADS) k_cg_start(int64_t m, const T *__restrict__ r, const T *__restrict__ b,
                                                         T *__restrict__ p, double *part_rr, double *part_bb) {
    double rr = 0.0, bb = 0.0;
    const int64_t stride = (int64_t)gridDim.x * CG_THREADS;
    for (int64_t i = (int64_t)blockIdx.x * CG_THREADS + threadIdx.x; i < m; i += stride) {
        const T ri = r[i];
        const double rw = wide(ri), bw = wide(b[i]);
        p[i] = ri;
        rr = fma(rw, rw, rr);
        bb = fma(bw, bw, bb);
    }
    rr = block_sum(rr);
    bb = block_sum(bb);
    if (threadIdx.x == 0) {
        part_rr[blockIdx.x] = rr;
        part_bb[blockIdx.x] = bb;
    }
}

__global__ void __launch_bounds__(CG_THREADS) k_cg_init(const double *part_rr, const double *part_bb, int nparts,
                                                        CgState *st, double *hist, double tol2, int32_t maxit,
                                                        cudaGraphConditionalHandle cond) {
    const double rr = sum_parts(part_rr, nparts);
    const double bb = sum_parts(part_bb, nparts);
    if (threadIdx.x == 0) {
        const double stop = tol2 * bb;
        st->rho = rr;
        st->done = 0;
        st->alpha = st->beta = 0.0;
        st->stop = stop;
        st->bb = bb;
        st->iter = 0;
        st->maxit = maxit;
        st->converged = rr <= stop;
        st->breakdown = 0;
        hist[0] = rr;
        cudaGraphSetConditional(cond, (maxit > 0 && rr > stop) ? 1u : 0u);
    }
}

// W elements per thread and access: 16-byte accesses where the caller's x is
// 16-byte aligned (the plan's own vectors always are), else one element
template <typename T, int W>
struct Pack {
    T v[W];
};
template <typename T, int W>
__device__ __forceinline__ Pack<T, W> ld_pack(const T *p) {
    Pack<T, W> o;
    if constexpr (W * sizeof(T) == 16) *reinterpret_cast<int4 *>(o.v) = *reinterpret_cast<const int4 *>(p);
    else o.v[0] = *p;
    return o;
}
template <typename T, int W>
__device__ __forceinline__ void st_pack(T *p, const Pack<T, W> &o) {
    if constexpr (W * sizeof(T) == 16) *reinterpret_cast<int4 *>(p) = *reinterpret_cast<const int4 *>(o.v);
    else *p = o.v[0];
}
// f(first) for the packs of [0, m) this thread owns
template <int W, typename F>
__device__ __forceinline__ void for_packs(int64_t m, F f) {
    const int64_t stride = (int64_t)gridDim.x * CG_THREADS, t = (int64_t)blockIdx.x * CG_THREADS + threadIdx.x;
    const int64_t packs = m / W;
#pragma unroll 2
    for (int64_t i = t; i < packs; i += stride) f(i * W);
}

// The calling block leaves its partial sum; the last block to do so gets the
// total, summed over the blocks in block order, and true.
__device__ bool last_block_total(double mine, double *part, unsigned *done, double *total) {
    __shared__ unsigned s_arrived;
    mine = block_sum(mine);
    if (threadIdx.x == 0) {
        part[blockIdx.x] = mine;
        __threadfence();
        s_arrived = atomicAdd(done, 1u);
    }
    __syncthreads();
    if (s_arrived != gridDim.x - 1) return false;
    __threadfence();
    double v = 0.0;
    for (int i = threadIdx.x; i < (int)gridDim.x; i += CG_THREADS) v += __ldcg(part + i);
    *total = block_sum(v);
    if (threadIdx.x == 0) *done = 0u;
    return true;
}

// p.q; the last block forms alpha, or records a breakdown
template <typename T, int W>
__global__ void __launch_bounds__(CG_THREADS) k_cg_dot(int64_t m, const T *p, const T *q, double *part, CgState *st) {
    double pq = 0.0;
    for_packs<W>(m, [&](int64_t i) {
        const Pack<T, W> a = ld_pack<T, W>(p + i), b = ld_pack<T, W>(q + i);
#pragma unroll
        for (int u = 0; u < W; ++u) pq = fma(wide(a.v[u]), wide(b.v[u]), pq);
    });
    if (W > 1 && blockIdx.x == 0 && threadIdx.x < m % W)
        pq = fma(wide(p[m - m % W + threadIdx.x]), wide(q[m - m % W + threadIdx.x]), pq);
    double total;
    if (!last_block_total(pq, part, &st->done, &total) || threadIdx.x != 0) return;
    if (!(total > 0.0)) {  // nothing moves any more
        st->breakdown = 1;
        st->converged = 0;
        st->alpha = 0.0;
    } else {
        st->alpha = st->rho / total;
    }
}

// r -= alpha q, r.r; the last block forms beta and decides whether the loop goes on
template <typename T, int W>
__global__ void __launch_bounds__(CG_THREADS) k_cg_residual(int64_t m, T *r, const T *q, double *part, CgState *st,
                                                            double *hist, cudaGraphConditionalHandle cond) {
    if (st->breakdown) {
        if (blockIdx.x == 0 && threadIdx.x == 0) cudaGraphSetConditional(cond, 0u);
        return;
    }
    const T alpha = (T)st->alpha;
    double rr = 0.0;
    auto one = [&](T ri, T qi) -> T {
        const T v = axpy1(ri, -alpha, qi);
        rr = fma(wide(v), wide(v), rr);
        return v;
    };
    for_packs<W>(m, [&](int64_t i) {
        Pack<T, W> a = ld_pack<T, W>(r + i);
        const Pack<T, W> b = ld_pack<T, W>(q + i);
#pragma unroll
        for (int u = 0; u < W; ++u) a.v[u] = one(a.v[u], b.v[u]);
        st_pack<T, W>(r + i, a);
    });
    if (W > 1 && blockIdx.x == 0 && threadIdx.x < m % W) {
        const int64_t i = m - m % W + threadIdx.x;
        r[i] = one(r[i], q[i]);
    }
    double total;
    if (!last_block_total(rr, part, &st->done, &total) || threadIdx.x != 0) return;
    st->beta = total / st->rho;
    st->rho = total;
    st->iter += 1;
    hist[st->iter] = total;
    st->converged = total <= st->stop;
    cudaGraphSetConditional(cond, (st->iter < st->maxit && total > st->stop) ? 1u : 0u);
}

// x += alpha p, p = r + beta p
template <typename T, int W>
__global__ void __launch_bounds__(CG_THREADS) k_cg_direction(int64_t m, T *x, T *p, const T *r, const CgState *st) {
    if (st->breakdown) return;
    const T alpha = (T)st->alpha, beta = (T)st->beta;
    for_packs<W>(m, [&](int64_t i) {
        Pack<T, W> a = ld_pack<T, W>(x + i), b = ld_pack<T, W>(p + i);
        const Pack<T, W> c = ld_pack<T, W>(r + i);
#pragma unroll
        for (int u = 0; u < W; ++u) {
            a.v[u] = axpy1(a.v[u], alpha, b.v[u]);
            b.v[u] = axpy1(c.v[u], beta, b.v[u]);
        }
        st_pack<T, W>(x + i, a);
        st_pack<T, W>(p + i, b);
    });
    if (W > 1 && blockIdx.x == 0 && threadIdx.x < m % W) {
        const int64_t i = m - m % W + threadIdx.x;
        x[i] = axpy1(x[i], alpha, p[i]);
        p[i] = axpy1(r[i], beta, p[i]);
    }
}

// ---------------------------------------------------------------------------
// Small systems: the whole solve in one thread-block cluster.  CTA c owns rows
// [c << shift, (c + 1) << shift); each thread keeps the x, r and p entries of
// its RPT rows in registers, p is also in the CTA's shared memory, where the
// other CTAs gather it (distributed shared memory), and an iteration is
// three cluster barriers.  The matrix is read from the CSR arrays, a row per
// thread (its slice stays in the SM's L1).  fp64 instructions are scarce (one
// warp instruction per 16 cycles and SM), so one warp per CTA sums the
// threads' partials and forms the scalars.  What bounds an iteration is
// latency: the barriers, the gathers and the dependent fp64 reductions and
// divisions.  200 iterations on the 64 x 64 5-point Laplacian (fp64): 5057 us
// in the graph form with five kernels, 1095 here.  Where a CTA's rows fit in
// its shared memory they are copied there once (27-point, 1000 rows: 8.4 us an
// iteration read in place, 6.9 staged).
// ---------------------------------------------------------------------------
constexpr int CL_THREADS = 512, CL_MAX_CTAS = 16, CL_MAX_RPT = 4;
constexpr int CL_SMEM = 200 * 1024;  // dynamic shared memory of a CTA
constexpr int64_t CL_MAX_ROW = 64, CL_MAX_NNZ = 3 << 17;

__device__ __forceinline__ unsigned cluster_rank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ unsigned cluster_size() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_barrier() {
    __syncwarp();  // the aligned form wants whole warps
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// address of this CTA's shared-memory word in CTA `rank`
__device__ __forceinline__ unsigned cluster_addr(unsigned addr, unsigned rank) {
    unsigned r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ double ld_cluster(unsigned a, double) {
    double v;
    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ float ld_cluster(unsigned a, float) {
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ void st_cluster(unsigned a, double v) {
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}

template <typename V, typename T>
__device__ __forceinline__ T widen(V v) {
    if constexpr (std::is_same<V, __nv_bfloat16>::value) return __bfloat162float(v);
    else return v;
}

template <typename V, typename T, int RPT>
__global__ void __launch_bounds__(CL_THREADS, 1)
k_cg_cluster(int m, int shift, int cap, const int *__restrict__ rowptr, const int *colidx, const V *vals, const T *b,
             T *x, double tol2, int32_t maxit, double *hist, CgState *st) {
    // this CTA's p, then (cap > 0) the values and columns of its rows
    extern __shared__ __align__(16) unsigned char cl_smem[];
    T *sp = reinterpret_cast<T *>(cl_smem);
    __shared__ double red[2][CL_THREADS];                                // threads' partials
    __shared__ double slot[2][2][CL_MAX_CTAS];                           // [phase][sum][CTA]
    __shared__ double s_out[2];
    const int tid = threadIdx.x, lane = tid & 31, nthr = blockDim.x;
    const unsigned rank = cluster_rank(), nc = cluster_size();
    const unsigned sp_addr = (unsigned)__cvta_generic_to_shared(sp);
    const int row0 = (int)(rank << shift), own = 1 << shift;
    int rs[RPT], re[RPT];
    bool have[RPT];
    T xv[RPT], rv[RPT], pv[RPT];
#pragma unroll
    for (int k = 0; k < RPT; ++k) {
        const int l = tid + k * nthr, row = row0 + l;
        have[k] = l < own && row < m;
        rs[k] = have[k] ? __ldg(rowptr + row) : 0;
        re[k] = have[k] ? __ldg(rowptr + row + 1) : 0;
        xv[k] = have[k] ? x[row] : T(0);
        if (l < own) sp[l] = xv[k];
    }
    if (cap > 0) {  // at most cap entries: the rows are copied once
        const int e0 = __ldg(rowptr + (row0 < m ? row0 : m)), e1 = __ldg(rowptr + (row0 + own < m ? row0 + own : m));
        V *sv = reinterpret_cast<V *>(cl_smem + sizeof(T) * (size_t)own);
        int *sc = reinterpret_cast<int *>(sv + cap);
        for (int t = tid; t < e1 - e0; t += nthr) {
            sv[t] = vals[e0 + t];
            sc[t] = colidx[e0 + t];
        }
        vals = sv;
        colidx = sc;
#pragma unroll
        for (int k = 0; k < RPT; ++k) {
            rs[k] -= have[k] ? e0 : 0;
            re[k] -= have[k] ? e0 : 0;
        }
    }
    // sum over the cluster of a (and, with two, of b): the threads' partials
    // in thread order by one warp, the CTAs' in rank order by every CTA's
    // first warp; both in lanes 0 of every CTA's first warp
    auto cluster_sums = [&](int phase, double a, double bsum, bool two, double &ta, double &tb) {
        red[0][tid] = a;
        if (two) red[1][tid] = bsum;
        __syncthreads();
        if (tid < 32) {
            const double u = nthr == CL_THREADS ? warp_sum_shared<CL_THREADS>(red[0]) : warp_sum_shared<CL_THREADS / 2>(red[0]);
            const double w = !two                 ? 0.0
                             : nthr == CL_THREADS ? warp_sum_shared<CL_THREADS>(red[1])
                                                  : warp_sum_shared<CL_THREADS / 2>(red[1]);
            if (lane < (int)nc) {
                const unsigned at = (unsigned)__cvta_generic_to_shared(&slot[phase][0][rank]);
                st_cluster(cluster_addr(at, lane), u);
                if (two) st_cluster(cluster_addr(at + CL_MAX_CTAS * 8, lane), w);
            }
        }
        __syncwarp();
        cluster_barrier();
        ta = tb = 0.0;
        if (tid < 32) {
            ta = lane < (int)nc ? slot[phase][0][lane] : 0.0;
            if (two) tb = lane < (int)nc ? slot[phase][1][lane] : 0.0;
#pragma unroll
            for (int o = CL_MAX_CTAS / 2; o > 0; o >>= 1) {
                ta += __shfl_xor_sync(0xffffffffu, ta, o);
                if (two) tb += __shfl_xor_sync(0xffffffffu, tb, o);
            }
        }
    };
    // row k of A times the vector in the CTAs' shared memory: the columns and
    // values of the next four entries are loaded while these four are gathered
    auto product = [&](int k) -> T {
        T acc = T(0);
        const int last = re[k] - 1;
        int c[4];
        T v[4];
        if (rs[k] <= last) {
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int t = rs[k] + u < last ? rs[k] + u : last;
                c[u] = colidx[t];
                v[u] = widen<V, T>(vals[t]);
            }
        }
        for (int t = rs[k]; t <= last; t += 4) {
            T pj[4], w[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                pj[u] = ld_cluster(cluster_addr(sp_addr + (unsigned)(c[u] & (own - 1)) * (unsigned)sizeof(T),
                                                (unsigned)c[u] >> shift), T(0));
                w[u] = v[u];
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int n = t + 4 + u < last ? t + 4 + u : last;
                c[u] = colidx[n];
                v[u] = widen<V, T>(vals[n]);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (t + u <= last) acc = fma(w[u], pj[u], acc);
        }
        return acc;
    };
    cluster_barrier();  // x_0 is in place
    double rr = 0.0, bb = 0.0;
#pragma unroll
    for (int k = 0; k < RPT; ++k) {
        const T bi = have[k] ? b[row0 + tid + k * nthr] : T(0);
        rv[k] = have[k] ? bi - product(k) : T(0);
        pv[k] = rv[k];
        rr = fma(wide(rv[k]), wide(rv[k]), rr);
        bb = fma(wide(bi), wide(bi), bb);
    }
    double rho, bsum, stop = 0.0;
    cluster_sums(0, rr, bb, true, rho, bsum);  // its barrier ends the reads of x_0
    int32_t iter = 0, converged = 0, breakdown = 0;
    // tid 0 of every CTA holds the scalars and decides alike
    __shared__ int s_go;
    if (tid == 0) {
        stop = tol2 * bsum;
        converged = rho <= stop;
        if (rank == 0) hist[0] = rho;
        s_go = maxit > 0 && rho > stop;
    }
    __syncthreads();
    while (s_go) {
#pragma unroll
        for (int k = 0; k < RPT; ++k)
            if (have[k]) sp[tid + k * nthr] = pv[k];
        cluster_barrier();  // p is in place
        T qv[RPT];
        double pq = 0.0;
#pragma unroll
        for (int k = 0; k < RPT; ++k) {
            qv[k] = have[k] ? product(k) : T(0);
            pq = fma(wide(pv[k]), wide(qv[k]), pq);
        }
        double tot, none;
        cluster_sums(0, pq, 0.0, false, tot, none);
        if (tid == 0) {
            if (!(tot > 0.0)) {
                breakdown = 1;
                converged = 0;
                s_go = 0;
            }
            s_out[0] = rho / tot;
        }
        __syncthreads();
        if (!s_go) break;  // breakdown: nothing moves
        const T alpha = (T)s_out[0];
        rr = 0.0;
#pragma unroll
        for (int k = 0; k < RPT; ++k) {
            rv[k] = axpy1(rv[k], -alpha, qv[k]);
            rr = fma(wide(rv[k]), wide(rv[k]), rr);
            xv[k] = axpy1(xv[k], alpha, pv[k]);
        }
        cluster_sums(1, rr, 0.0, false, tot, none);
        if (tid == 0) {
            s_out[1] = tot / rho;
            rho = tot;
            ++iter;
            if (rank == 0) hist[iter] = rho;
            converged = rho <= stop;
            s_go = iter < maxit && rho > stop;
        }
        __syncthreads();
        const T beta = (T)s_out[1];
#pragma unroll
        for (int k = 0; k < RPT; ++k) pv[k] = axpy1(rv[k], beta, pv[k]);
    }
#pragma unroll
    for (int k = 0; k < RPT; ++k)
        if (have[k]) x[row0 + tid + k * nthr] = xv[k];
    if (rank == 0 && tid == 0) {
        st->rho = rho;
        st->stop = stop;
        st->bb = bsum;
        st->iter = iter;
        st->maxit = maxit;
        st->converged = converged;
        st->breakdown = breakdown;
    }
    cluster_barrier();  // no CTA leaves while another may still reach its shared memory
}

int run_spmv(const spmv_matrix *h, double alpha, const void *x, double beta, void *y, cudaStream_t s) {
    return run_product(h, alpha, x, beta, y, s);
}

}  // namespace

struct CgPlan {
    const void *b = nullptr;
    void *x = nullptr;
    double tol = -1.0;
    int32_t maxit = -1;
    int nparts = 0;
    void *r = nullptr, *p = nullptr, *q = nullptr;
    double *part = nullptr;  // 2 x nparts: the running dot product, b.b
    double *hist = nullptr;  // maxit + 1
    CgState *st = nullptr;
    int ctas = 0, shift = 0, cap = 0;  // cluster form: CTAs (0: graph form), log2 of a CTA's rows, staged entries
    cudaStream_t cs = nullptr;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
};

void free_cg(spmv_matrix *h) {
    CgPlan *c = h->cg;
    if (!c) return;
    if (c->exec) cudaGraphExecDestroy(c->exec);
    if (c->graph) cudaGraphDestroy(c->graph);
    if (c->cs) cudaStreamDestroy(c->cs);
    dev_free(c->r);
    dev_free(c->p);
    dev_free(c->q);
    dev_free(c->part);
    dev_free(c->hist);
    dev_free(c->st);
    delete c;
    h->cg = nullptr;
}

namespace {

template <typename T>
int capture_cg(spmv_matrix *h, CgPlan *c) {
    const int64_t m = h->m;
    const int G = c->nparts;
    T *r = (T *)c->r, *p = (T *)c->p, *q = (T *)c->q;
    const T *b = (const T *)c->b;
    T *x = (T *)c->x;
    double *part = c->part, *part_bb = c->part + G;
    cudaStream_t cs = c->cs;
    constexpr int W = 16 / sizeof(T);
    auto direction = ((uintptr_t)x & 15u) == 0 ? k_cg_direction<T, W> : k_cg_direction<T, 1>;

    SPMV_CUDA_TRY(cudaGraphCreate(&c->graph, 0));
    cudaGraphConditionalHandle cond;
    SPMV_CUDA_TRY(cudaGraphConditionalHandleCreate(&cond, c->graph, 0, cudaGraphCondAssignDefault));

    // prologue: r = b - A x, p = r, rho_0, b.b, loop condition
    SPMV_CUDA_TRY(cudaStreamBeginCaptureToGraph(cs, c->graph, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal));
    int st = SPMV_OK;
    cudaError_t e = cudaMemcpyAsync(r, b, sizeof(T) * m, cudaMemcpyDeviceToDevice, cs);
    if (e != cudaSuccess) st = cuda_status(e, "cudaMemcpyAsync(r <- b)");
    if (st == SPMV_OK) st = run_spmv(h, -1.0, x, 1.0, r, cs);
    if (st == SPMV_OK) {
        k_cg_start<T><<<G, CG_THREADS, 0, cs>>>(m, r, b, p, part, part_bb);
        k_cg_init<<<1, CG_THREADS, 0, cs>>>(part, part_bb, G, c->st, c->hist, c->tol * c->tol, c->maxit, cond);
        e = cudaGetLastError();
        if (e != cudaSuccess) st = cuda_status(e, "CG prologue launch");
    }
    cudaGraphNode_t loop = nullptr;
    if (st == SPMV_OK) {
        cudaStreamCaptureStatus cst;
        const cudaGraphNode_t *deps = nullptr;
        size_t ndeps = 0;
        e = cudaStreamGetCaptureInfo(cs, &cst, nullptr, nullptr, &deps, nullptr, &ndeps);
        if (e != cudaSuccess) st = cuda_status(e, "cudaStreamGetCaptureInfo");
        if (st == SPMV_OK) {
            cudaGraphNodeParams np = {};
            np.type = cudaGraphNodeTypeConditional;
            np.conditional.handle = cond;
            np.conditional.type = cudaGraphCondTypeWhile;
            np.conditional.size = 1;
            e = cudaGraphAddNode(&loop, c->graph, deps, nullptr, ndeps, &np);
            if (e != cudaSuccess) st = cuda_status(e, "cudaGraphAddNode(while)");
            if (st == SPMV_OK) {
                e = cudaStreamUpdateCaptureDependencies(cs, &loop, nullptr, 1, cudaStreamSetCaptureDependencies);
                if (e != cudaSuccess) st = cuda_status(e, "cudaStreamUpdateCaptureDependencies");
            }
            if (st == SPMV_OK) {
                // body: one CG iteration
                cudaGraph_t body = np.conditional.phGraph_out[0];
                cudaStream_t bs = nullptr;
                e = cudaStreamCreateWithFlags(&bs, cudaStreamNonBlocking);
                if (e != cudaSuccess) st = cuda_status(e, "cudaStreamCreate(body)");
                if (st == SPMV_OK) {
                    e = cudaStreamBeginCaptureToGraph(bs, body, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal);
                    if (e != cudaSuccess) st = cuda_status(e, "cudaStreamBeginCaptureToGraph(body)");
                }
                if (st == SPMV_OK) {
                    st = run_spmv(h, 1.0, p, 0.0, q, bs);
                    if (st == SPMV_OK) {
                        k_cg_dot<T, W><<<G, CG_THREADS, 0, bs>>>(m, p, q, part, c->st);
                        k_cg_residual<T, W><<<G, CG_THREADS, 0, bs>>>(m, r, q, part, c->st, c->hist, cond);
                        direction<<<G, CG_THREADS, 0, bs>>>(m, x, p, r, c->st);
                        e = cudaGetLastError();
                        if (e != cudaSuccess) st = cuda_status(e, "CG body launch");
                    }
                    cudaGraph_t bout = nullptr;
                    e = cudaStreamEndCapture(bs, &bout);
                    if (e != cudaSuccess && st == SPMV_OK) st = cuda_status(e, "cudaStreamEndCapture(body)");
                }
                if (bs) cudaStreamDestroy(bs);
            }
        }
    }
    cudaGraph_t out = nullptr;
    e = cudaStreamEndCapture(cs, &out);
    if (e != cudaSuccess && st == SPMV_OK) st = cuda_status(e, "cudaStreamEndCapture");
    if (st != SPMV_OK) return st;
    SPMV_CUDA_TRY(cudaGraphInstantiate(&c->exec, c->graph, 0));
    return SPMV_OK;
}

// The cluster form's kernel for this value type and rows per thread.
template <typename V, typename T>
const void *cluster_kernel(int rpt) {
    return rpt == 1   ? (const void *)k_cg_cluster<V, T, 1>
           : rpt == 2 ? (const void *)k_cg_cluster<V, T, 2>
                      : (const void *)k_cg_cluster<V, T, CL_MAX_RPT>;
}
const void *cluster_kernel(int vt, int rpt) {
    return vt == SPMV_F64   ? cluster_kernel<double, double>(rpt)
           : vt == SPMV_F32 ? cluster_kernel<float, float>(rpt)
                            : cluster_kernel<__nv_bfloat16, float>(rpt);
}

size_t cluster_smem(int vt, int shift, int64_t cap) {
    return vec_size(vt) * ((size_t)1 << shift) + (value_size(vt) + 4) * (size_t)cap;
}

struct ClusterLaunch {
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute attr{};
    const void *kernel = nullptr;
    ClusterLaunch(int vt, int ctas, int shift, int cap, cudaStream_t s) {
        const int own = 1 << shift, threads = own < CL_THREADS ? own : CL_THREADS;
        kernel = cluster_kernel(vt, own / threads);
        cfg.gridDim = dim3((unsigned)ctas);
        cfg.blockDim = dim3((unsigned)threads);
        cfg.dynamicSmemBytes = cluster_smem(vt, shift, cap);
        cfg.stream = s;
        attr.id = cudaLaunchAttributeClusterDimension;
        attr.val.clusterDim.x = (unsigned)ctas;
        attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
        cfg.attrs = &attr;
        cfg.numAttrs = 1;
    }
    ClusterLaunch(const ClusterLaunch &) = delete;
};

// Whether the cluster form takes this system, with how many CTAs of how many
// rows, and whether the rows are staged.  The line: 16 SMs have a tenth of the
// chip's fp64 and L2 rates, the graph form pays about 20 us an iteration for
// its four dependent launches.  Microseconds per iteration, cluster / graph:
// 5-point fp64 1024 rows 5.6 / 19.5, 4096 5.8 / 20.0, 32,700 12.1 / 22.1;
// 27-point fp64 8000 rows (195K entries, staged) 9.8 / 23.6, 13,824 (343K,
// read in place) 18.2 / 23.6, 19,683 (507K) 29.0 / 24.7, fp32 23.6 / 23.4.
// A row is one thread's serial work, hence the limit on its length.  It is
// summed in column order, as the formats with one lane per row sum it, so only
// those take this form: a handle set to another format keeps that format's
// products.
bool cluster_fits(const spmv_matrix *h, int *ctas, int *shift, int *cap) {
    const int fmt = h->cfg.format;
    const bool lane_rows = fmt == SPMV_FMT_ELL || fmt == SPMV_FMT_SELL || (fmt == SPMV_FMT_HYB && h->hyb_nnz == 0) ||
                           (fmt == SPMV_FMT_CSR && h->cfg.threads_per_row == 1 && !csr_uneven(h, 1));
    if (!lane_rows || h->npanels > 0 || h->m > (int64_t)CL_MAX_CTAS * CL_THREADS * CL_MAX_RPT || h->max_row > CL_MAX_ROW ||
        h->nnz > CL_MAX_NNZ)
        return false;
    int sh = 8, n = 1;
    while (((int64_t)CL_MAX_CTAS << sh) < h->m) ++sh;
    while (((int64_t)n << sh) < h->m) n *= 2;
    // the CTA's rows in shared memory where they fit
    int64_t entries = std::min<int64_t>(h->max_row << sh, h->nnz);
    entries = (entries + 7) / 8 * 8;
    if (cluster_smem(h->vt, sh, entries) > CL_SMEM) entries = 0;
    ClusterLaunch L(h->vt, n, sh, (int)entries, nullptr);
    int most = 0;
    if (cudaFuncSetAttribute(L.kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, CL_SMEM) != cudaSuccess ||
        (n > 8 && cudaFuncSetAttribute(L.kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) ||
        cudaOccupancyMaxActiveClusters(&most, L.kernel, &L.cfg) != cudaSuccess || most < 1) {
        cudaGetLastError();  // such a cluster cannot run here
        return false;
    }
    *ctas = n;
    *shift = sh;
    *cap = (int)entries;
    return true;
}

int launch_cluster(const spmv_matrix *h, CgPlan *c, cudaStream_t s) {
    ClusterLaunch L(h->vt, c->ctas, c->shift, c->cap, s);
    int m = (int)h->m, shift = c->shift, cap = c->cap;
    double tol2 = c->tol * c->tol;
    void *args[] = {&m,    &shift, &cap,      (void *)&h->rowptr, (void *)&h->colidx, (void *)&h->vals, &c->b,
                    &c->x, &tol2,  &c->maxit, &c->hist,           &c->st};
    SPMV_CUDA_TRY(cudaLaunchKernelExC(&L.cfg, L.kernel, args));
    return SPMV_OK;
}

int build_plan(spmv_matrix *h, const void *d_b, void *d_x, double tol, int32_t maxit, cudaStream_t s) {
    CgPlan *c = h->cg;
    if (c && c->b == d_b && c->x == d_x && c->tol == tol && c->maxit == maxit) return SPMV_OK;
    free_cg(h);
    c = new (std::nothrow) CgPlan();
    if (!c) {
        set_error("spmv_cg: host allocation failed");
        return SPMV_ERR_OOM;
    }
    h->cg = c;
    c->b = d_b;
    c->x = d_x;
    c->tol = tol;
    c->maxit = maxit;
    // two blocks per SM: their partials and arrivals meet in one word, so no
    // more of them than fill the chip
    c->nparts = (int)std::min<int64_t>(2 * (h->sm_count > 0 ? h->sm_count : 152),
                                       std::max<int64_t>(1, (h->m + 2 * CG_THREADS - 1) / (2 * CG_THREADS)));
    const size_t vb = vec_size(h->vt) * (size_t)h->m;
    // a plan that fails half-built is released, so a later call with the
    // same arguments builds it again instead of reusing it
    auto fail = [&](int st) {
        free_cg(h);
        return st;
    };
    cudaError_t e = cudaSuccess;
    if (cluster_fits(h, &c->ctas, &c->shift, &c->cap)) {
        e = dev_malloc(&c->hist, sizeof(double) * ((size_t)maxit + 1));
        if (e == cudaSuccess) e = dev_malloc(&c->st, sizeof(CgState));
        return e == cudaSuccess ? SPMV_OK : fail(cuda_status(e, "spmv_cg plan"));
    }
    e = dev_malloc(&c->r, vb);
    if (e == cudaSuccess) e = dev_malloc(&c->p, vb);
    if (e == cudaSuccess) e = dev_malloc(&c->q, vb);
    if (e == cudaSuccess) e = dev_malloc(&c->part, sizeof(double) * 2 * c->nparts);
    if (e == cudaSuccess) e = dev_malloc(&c->hist, sizeof(double) * ((size_t)maxit + 1));
    if (e == cudaSuccess) e = dev_malloc(&c->st, sizeof(CgState));
    if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&c->cs, cudaStreamNonBlocking);
    if (e != cudaSuccess) return fail(cuda_status(e, "spmv_cg plan"));
    // one eager product before capture: occupancy and carveout settings of
    // the kernel are resolved outside the capture
    int st = run_spmv(h, 1.0, d_b, 0.0, c->q, s);
    if (st == SPMV_OK) {
        e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) st = cuda_status(e, "spmv_cg plan");
    }
    if (st == SPMV_OK) st = h->vt == SPMV_F64 ? capture_cg<double>(h, c) : capture_cg<float>(h, c);
    if (st != SPMV_OK) return fail(st);
    return SPMV_OK;
}

}  // namespace
}  // namespace spmv

using namespace spmv;

extern "C" int spmv_cg(spmv_handle h, const void *d_b, void *d_x, double tol, int32_t maxit, double *d_rho,
                       spmv_cg_result *out, void *stream) {
    entry_reset();
    if (!h || !out) {
        set_error("spmv_cg: NULL handle or result");
        return SPMV_ERR_INVALID;
    }
    std::memset(out, 0, sizeof *out);
    if (h->m != h->n) {
        set_error("spmv_cg: matrix is %lld x %lld, not square", (long long)h->m, (long long)h->n);
        return SPMV_ERR_INVALID;
    }
    if (!(tol >= 0.0) || !std::isfinite(tol) || maxit < 0 || maxit > SPMV_CG_MAX_ITERATIONS) {
        set_error("spmv_cg: need 0 <= tol < inf and 0 <= maxit <= %d", SPMV_CG_MAX_ITERATIONS);
        return SPMV_ERR_INVALID;
    }
    if (h->m > 0 && (!d_b || !d_x)) {
        set_error("spmv_cg: NULL vector");
        return SPMV_ERR_INVALID;
    }
    cudaStream_t s = (cudaStream_t)stream;
    if (h->m == 0) {
        out->converged = 1;
        if (d_rho) SPMV_CUDA_TRY(cudaMemsetAsync(d_rho, 0, sizeof(double), s));
        return SPMV_OK;
    }
    SPMV_TRY(build_plan(h, d_b, d_x, tol, maxit, s));
    CgPlan *c = h->cg;
    if (c->ctas > 0) SPMV_TRY(launch_cluster(h, c, s));
    else SPMV_CUDA_TRY(cudaGraphLaunch(c->exec, s));
    CgState st;
    SPMV_CUDA_TRY(cudaMemcpyAsync(&st, c->st, sizeof st, cudaMemcpyDeviceToHost, s));
    SPMV_CUDA_TRY(cudaStreamSynchronize(s));
    if (d_rho)
        SPMV_CUDA_TRY(cudaMemcpyAsync(d_rho, c->hist, sizeof(double) * ((size_t)st.iter + 1), cudaMemcpyDeviceToDevice, s));
    out->iterations = st.iter;
    out->converged = st.converged;
    out->breakdown = st.breakdown;
    out->rho0 = 0.0;
    out->rho = st.rho;
    out->bb = st.bb;
    SPMV_CUDA_TRY(cudaMemcpyAsync(&out->rho0, c->hist, sizeof(double), cudaMemcpyDeviceToHost, s));
    SPMV_CUDA_TRY(cudaStreamSynchronize(s));
    return SPMV_OK;
}
