// Krylov solver around the H-FMM apply: restarted GMRES for
//     (sigma I + A) x = b,   A_ij = u_{x_j}(x_i)  (Sec. 2.4),
// the dense system of a second-kind integral equation discretised on the
// plan's points.  Every operator application is one hfmm apply; the Krylov
// vectors stay on the device and are orthogonalised there by two passes of
// classical Gram-Schmidt (as orthogonal as the modified form to rounding; dot
// products accumulated in FP64): one kernel takes all dot products of a pass, one
// subtracts all projections, and for short vectors one cluster does the whole step.
// The host reads one Hessenberg column per Arnoldi
// step and solves the small least-squares problem (Givens rotations).
//
// The modified form took a kernel, a copy and a host round trip per dot product:
// 1600 points, FP64, 14 steps: 28 ms, of which the applies were 2.3 ms (one GB300).
#include <algorithm>
#include <cmath>
#include <complex>
#include <vector>

#include <cooperative_groups.h>

#include "plan.cuh"
#include "split64.cuh"

namespace {

namespace cg = cooperative_groups;

using zc = std::complex<double>;

constexpr int SV_THREADS = 256;
constexpr int SV_BLOCKS = 4 * 152;

template <class T> struct Cx;
template <> struct Cx<cd> {
    static __device__ __forceinline__ double re(cd v) { return v.x; }
    static __device__ __forceinline__ double im(cd v) { return v.y; }
    static __device__ __forceinline__ cd mk(double r, double i) { return cmk(r, i); }
};
template <> struct Cx<cf> {
    static __device__ __forceinline__ double re(cf v) { return v.x; }
    static __device__ __forceinline__ double im(cf v) { return v.y; }
    static __device__ __forceinline__ cf mk(double r, double i) { return cfmk((float)r, (float)i); }
};

// sum over the block, in thread 0
__device__ __forceinline__ double2 sv_block_sum(double sr, double si, double2* red) {
    for (int o = 16; o > 0; o >>= 1) {
        sr += __shfl_down_sync(0xffffffffu, sr, o);
        si += __shfl_down_sync(0xffffffffu, si, o);
    }
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = make_double2(sr, si);
    __syncthreads();
    double2 t = make_double2(0.0, 0.0);
    if (threadIdx.x == 0)
        for (int w = 0; w < SV_THREADS / 32; ++w) { t.x += red[w].x; t.y += red[w].y; }
    return t;
}

// the block that finishes last adds the blocks' partial sums of `cnt` values (part[value][block])
// in block order into out; *ticket is zero between launches
__device__ __forceinline__ bool sv_last_block(unsigned* ticket) {
    __shared__ bool last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        last = atomicAdd(ticket, 1u) == gridDim.x - 1;
        if (last) *ticket = 0;
    }
    __syncthreads();
    if (last) __threadfence();
    return last;
}

__device__ __forceinline__ double2 sv_warp_sum(double sr, double si) {
    for (int o = 16; o > 0; o >>= 1) {
        sr += __shfl_xor_sync(0xffffffffu, sr, o);
        si += __shfl_xor_sync(0xffffffffu, si, o);
    }
    return make_double2(sr, si);
}

__device__ __forceinline__ void sv_add_parts(const double2* part, int cnt, double2* out) {
    const int lane = threadIdx.x & 31;
    for (int i = threadIdx.x >> 5; i < cnt; i += SV_THREADS / 32) {
        double sr = 0.0, si = 0.0;
        for (unsigned k = lane; k < gridDim.x; k += 32) {
            const double2 p = __ldcg(part + (size_t)i * gridDim.x + k);
            sr += p.x;
            si += p.y;
        }
        const double2 s = sv_warp_sum(sr, si);
        if (lane == 0) out[i] = s;
    }
}

// h_i = <v_i, w>, i < cnt (v_i = V + i n); with shift, w += sigma v_{cnt - 1} first (the operator's
// shift).  A block keeps its part of w in shared memory, a warp takes every eighth vector.
template <class T>
__global__ void __launch_bounds__(SV_THREADS) dots_kernel(const T* __restrict__ V, T* __restrict__ w, int64_t n, int chunk,
                                                          int cnt, int shift, double sr, double si,
                                                          double2* __restrict__ part, double2* __restrict__ h,
                                                          unsigned* __restrict__ ticket) {
    extern __shared__ double2 ws[];
    const int lane = threadIdx.x & 31;
    const int64_t lo = (int64_t)blockIdx.x * chunk;
    const int m = (int)(n - lo < chunk ? n - lo : chunk);
    for (int i = threadIdx.x; i < m; i += SV_THREADS) {
        T x = w[lo + i];
        if (shift) {
            const T v = V[(int64_t)(cnt - 1) * n + lo + i];
            const double vr = Cx<T>::re(v), vi = Cx<T>::im(v);
            x = Cx<T>::mk(Cx<T>::re(x) + sr * vr - si * vi, Cx<T>::im(x) + sr * vi + si * vr);
            w[lo + i] = x;
        }
        ws[i] = make_double2(Cx<T>::re(x), Cx<T>::im(x));
    }
    __syncthreads();
    for (int j = threadIdx.x >> 5; j < cnt; j += SV_THREADS / 32) {
        const T* v = V + (int64_t)j * n + lo;
        double tr = 0.0, ti = 0.0;
#pragma unroll 4
        for (int i = lane; i < m; i += 32) {
            const double ar = Cx<T>::re(v[i]), ai = Cx<T>::im(v[i]);
            const double2 b = ws[i];
            tr += ar * b.x + ai * b.y;
            ti += ar * b.y - ai * b.x;
        }
        const double2 t = sv_warp_sum(tr, ti);
        if (lane == 0) part[(size_t)j * gridDim.x + blockIdx.x] = t;
    }
    if (sv_last_block(ticket)) sv_add_parts(part, cnt, h);
}

// w += sgn sum_i c_i v_i, i < cnt; norm: also |w|^2 into *nrm
template <class T>
__global__ void __launch_bounds__(SV_THREADS) combine_kernel(const T* V, const double2* __restrict__ c, int cnt,
                                                             double sgn, T* w, int64_t n, int chunk,
                                                             double2* __restrict__ part, double2* __restrict__ nrm,
                                                             unsigned* __restrict__ ticket) {
    __shared__ double2 red[SV_THREADS / 32];
    const int64_t lo = (int64_t)blockIdx.x * chunk;
    double s = 0.0;
    for (int64_t i = lo + threadIdx.x; i < n && i < lo + chunk; i += SV_THREADS) {
        double wr = 0.0, wi = 0.0;
#pragma unroll 4
        for (int j = 0; j < cnt; ++j) {
            const double2 a = c[j];
            const T v = V[(int64_t)j * n + i];
            const double vr = Cx<T>::re(v), vi = Cx<T>::im(v);
            wr += a.x * vr - a.y * vi;
            wi += a.x * vi + a.y * vr;
        }
        const T x = Cx<T>::mk(Cx<T>::re(w[i]) + sgn * wr, Cx<T>::im(w[i]) + sgn * wi);
        w[i] = x;
        s += Cx<T>::re(x) * Cx<T>::re(x) + Cx<T>::im(x) * Cx<T>::im(x);
    }
    if (!nrm) return;
    const double2 t = sv_block_sum(s, 0.0, red);
    if (threadIdx.x == 0) part[blockIdx.x] = t;
    if (sv_last_block(ticket)) sv_add_parts(part, 1, nrm);
}

// v = w / |w| (v = 0 for |w| = 0); the column h = h1 + h2 and |w|^2 for the host
template <class T>
__global__ void __launch_bounds__(SV_THREADS) normalise_kernel(const T* __restrict__ w, const double2* __restrict__ nrm,
                                                               T* __restrict__ v, int64_t n, int cnt,
                                                               const double2* __restrict__ h1,
                                                               const double2* __restrict__ h2, double2* __restrict__ col) {
    const double d = sqrt(nrm->x), inv = d > 0.0 ? 1.0 / d : 0.0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        v[i] = Cx<T>::mk(inv * Cx<T>::re(w[i]), inv * Cx<T>::im(w[i]));
    if (blockIdx.x == 0)
        for (int i = threadIdx.x; i <= cnt; i += SV_THREADS)
            col[i] = i < cnt ? make_double2(h1[i].x + h2[i].x, h1[i].y + h2[i].y) : *nrm;
}

// A whole Arnoldi step's orthogonalisation in one cluster: shift, two passes of dot products and
// projections, norm, v_{j + 1} and the Hessenberg column, w kept in FP64 in shared memory and
// the CTAs' sums added in rank order.  For vectors of up to CGS_MAX elements: five kernels took 60 us there
// (1600 points), each mostly its start and the two latencies of its reduction; sixteen SMs have
// the FP64 rate for the 16 n (j + 1) FMAs up to a few thousand points.  1600 points, 38 steps a
// solve: 8.95 -> 8.61 ms (7.8 with the applies of today).
constexpr int CGS_CTAS = 16, CGS_THREADS = 512, CGS_WARPS = CGS_THREADS / 32;
constexpr int64_t CGS_MAX = 4096;
constexpr int CGS_MAX_RESTART = 1024;

template <class T>
__global__ void __launch_bounds__(CGS_THREADS) cgs_kernel(const T* __restrict__ V, T* vnext, const T* __restrict__ w,
                                                          int64_t n, int chunk, int cnt, double sr, double si,
                                                          double2* __restrict__ col) {
    extern __shared__ double2 cgs_s[];
    cg::cluster_group cluster = cg::this_cluster();
    double2* ws = cgs_s;                       // [chunk]
    double2* hp = ws + chunk;                  // [2][cnt] this CTA's dot products
    double2* hs = hp + 2 * cnt;                // [cnt] a pass's sums
    double2* ht = hs + cnt;                    // [cnt] both passes'
    double2* red = ht + cnt;                   // [CGS_THREADS]
    double2* nr = red + CGS_THREADS;           // [1]
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, rank = (int)cluster.block_rank();
    const int64_t lo = (int64_t)rank * chunk;
    const int m = (int)(n <= lo ? 0 : n - lo < chunk ? n - lo : chunk);
    for (int i = tid; i < m; i += CGS_THREADS) {
        const T x = w[lo + i], v = V[(int64_t)(cnt - 1) * n + lo + i];
        const double vr = Cx<T>::re(v), vi = Cx<T>::im(v);
        ws[i] = make_double2(Cx<T>::re(x) + sr * vr - si * vi, Cx<T>::im(x) + sr * vi + si * vr);
    }
    __syncthreads();
    const int tiles = (m + 31) / 32, parts = tiles > 0 && tiles < CGS_WARPS ? CGS_WARPS / tiles : 1, at_once = CGS_WARPS / parts;
    for (int pass = 0; pass < 2; ++pass) {
        double2* mine = hp + pass * cnt;
        for (int j = wid; j < cnt; j += CGS_WARPS) {
            const T* v = V + (int64_t)j * n + lo;
            double tr = 0.0, ti = 0.0;
#pragma unroll 4
            for (int i = lane; i < m; i += 32) {
                const double ar = Cx<T>::re(v[i]), ai = Cx<T>::im(v[i]);
                const double2 b = ws[i];
                tr += ar * b.x + ai * b.y;
                ti += ar * b.y - ai * b.x;
            }
            const double2 t = sv_warp_sum(tr, ti);
            if (lane == 0) mine[j] = t;
        }
        cluster.sync();
        for (int j = tid; j < cnt; j += CGS_THREADS) {
            double2 t = make_double2(0.0, 0.0);
#pragma unroll
            for (int r = 0; r < CGS_CTAS; ++r) {
                const double2 o = cluster.map_shared_rank(mine, r)[j];
                t.x += o.x;
                t.y += o.y;
            }
            hs[j] = t;
            ht[j] = pass == 0 ? t : make_double2(ht[j].x + t.x, ht[j].y + t.y);
        }
        __syncthreads();
        // a warp takes 32 elements; where there are fewer such tiles than warps, several share the vectors of one
        for (int t0 = 0; t0 < tiles; t0 += at_once) {
            const int tile = t0 + wid / parts, part = wid % parts, i = tile * 32 + lane;
            const bool live = wid < at_once * parts && i < m;
            double wr = 0.0, wi = 0.0;
            if (live) {
#pragma unroll 4
                for (int j = part; j < cnt; j += parts) {
                    const double2 a = hs[j];
                    const T v = V[(int64_t)j * n + lo + i];
                    const double vr = Cx<T>::re(v), vi = Cx<T>::im(v);
                    wr += a.x * vr - a.y * vi;
                    wi += a.x * vi + a.y * vr;
                }
            }
            red[tid] = make_double2(wr, wi);
            __syncthreads();
            if (live && part == 0) {
                for (int o = 1; o < parts; ++o) {
                    wr += red[tid + 32 * o].x;
                    wi += red[tid + 32 * o].y;
                }
                ws[i] = make_double2(ws[i].x - wr, ws[i].y - wi);
            }
            __syncthreads();
        }
    }
    double s = 0.0;
    for (int i = tid; i < m; i += CGS_THREADS) s += ws[i].x * ws[i].x + ws[i].y * ws[i].y;
    const double2 ss = sv_warp_sum(s, 0.0);
    if (lane == 0) red[wid] = ss;
    __syncthreads();
    if (tid == 0) {
        double2 t = make_double2(0.0, 0.0);
        for (int k = 0; k < CGS_WARPS; ++k) t.x += red[k].x;
        *nr = t;
    }
    cluster.sync();
    double nn = 0.0;
    for (int r = 0; r < CGS_CTAS; ++r) nn += cluster.map_shared_rank(nr, r)->x;
    const double d = sqrt(nn), inv = d > 0.0 ? 1.0 / d : 0.0;
    for (int i = tid; i < m; i += CGS_THREADS) vnext[lo + i] = Cx<T>::mk(inv * ws[i].x, inv * ws[i].y);
    if (rank == 0)
        for (int j = tid; j <= cnt; j += CGS_THREADS) col[j] = j < cnt ? ht[j] : make_double2(nn, 0.0);
    cluster.sync();                            // nobody's shared memory is read any more
}

// y = alpha x + beta y (alpha, beta complex)
template <class T>
__global__ void axpby_kernel(double ar, double ai, const T* __restrict__ x, double br, double bi, T* __restrict__ y,
                             int64_t n) {
    const bool ready = br != 0.0 || bi != 0.0;      // beta = 0: y is only written
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const double xr = Cx<T>::re(x[i]), xi = Cx<T>::im(x[i]);
        const double yr = ready ? Cx<T>::re(y[i]) : 0.0, yi = ready ? Cx<T>::im(y[i]) : 0.0;
        y[i] = Cx<T>::mk(ar * xr - ai * xi + br * yr - bi * yi, ar * xi + ai * xr + br * yi + bi * yr);
    }
}

template <class T>
struct Krylov {
    hfmm_plan_s* P;
    cudaStream_t st;
    int64_t n;
    // device: block partial sums, two passes' dot products, a norm, a column; the column's page-locked copy
    double2 *part, *h1, *h2, *nrm, *col, *host;
    unsigned* ticket;
    int chunk;           // vector elements of a block in the Gram-Schmidt kernels
    bool one_cluster;    // cgs_kernel takes a whole step

    unsigned blocks() const { return (unsigned)((n + chunk - 1) / chunk); }
    hfmm_status read(const double2* d, int cnt) {
        HFMM_CUDA_TRY(cudaMemcpyAsync(host, d, sizeof(double2) * cnt, cudaMemcpyDeviceToHost, st));
        HFMM_CUDA_TRY(cudaStreamSynchronize(st));
        return HFMM_OK;
    }
    // |a|^2
    hfmm_status norm2(T* a, double* out) {
        combine_kernel<T><<<blocks(), SV_THREADS, 0, st>>>(a, h1, 0, 0.0, a, n, chunk, part, nrm, ticket);
        HFMM_CUDA_TRY(cudaGetLastError());
        HFMM_TRY(read(nrm, 1));
        *out = host[0].x;
        return HFMM_OK;
    }
    size_t cgs_smem(int cnt) const {
        return sizeof(double2) * ((size_t)((n + CGS_CTAS - 1) / CGS_CTAS) + 4 * (size_t)cnt + CGS_THREADS + 1);
    }
    // Whether a basis of m vectors is orthogonalised by cgs_kernel: short vectors, and a device (or the part of
    // one that this process has) that can place a cluster of 16 CTAs with their shared memory.
    hfmm_status choose_cgs(int m) {
        one_cluster = false;
        if (n > CGS_MAX || m > CGS_MAX_RESTART) return HFMM_OK;
        HFMM_CUDA_TRY(cudaFuncSetAttribute(cgs_kernel<T>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
        HFMM_CUDA_TRY(cudaFuncSetAttribute(cgs_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, 96 * 1024));
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3(CGS_CTAS);
        cfg.blockDim = dim3(CGS_THREADS);
        cfg.dynamicSmemBytes = cgs_smem(m);
        cudaLaunchAttribute at{};
        at.id = cudaLaunchAttributeClusterDimension;
        at.val.clusterDim.x = CGS_CTAS;
        at.val.clusterDim.y = at.val.clusterDim.z = 1;
        cfg.attrs = &at;
        cfg.numAttrs = 1;
        int clusters = 0;
        one_cluster = cudaOccupancyMaxActiveClusters(&clusters, cgs_kernel<T>, &cfg) == cudaSuccess && clusters > 0;
        cudaGetLastError();
        return HFMM_OK;
    }
    // Arnoldi step: w = (sigma + A) v_j minus its projections on v_0 .. v_j, v_{j + 1} = w / |w|;
    // host[0 .. j] = the Hessenberg column, host[j + 1].x = |w|^2
    hfmm_status arnoldi(zc sigma, T* V, int j, T* w) {
        HFMM_TRY(apply(V + (size_t)j * n, w));
        if (one_cluster) {                                 // the column goes straight to the host's pages
            const int part_n = (int)((n + CGS_CTAS - 1) / CGS_CTAS), cnt = j + 1;
            HFMM_CUDA_TRY(pdl_launch_if(false, cgs_kernel<T>, dim3(CGS_CTAS), dim3(CGS_THREADS), cgs_smem(cnt), st, CGS_CTAS, V,
                                        V + (size_t)(j + 1) * n, w, n, part_n, cnt, sigma.real(), sigma.imag(), host));
            HFMM_CUDA_TRY(cudaStreamSynchronize(st));
            return HFMM_OK;
        }
        const unsigned g = blocks();
        const size_t sm = sizeof(double2) * chunk;
        dots_kernel<T><<<g, SV_THREADS, sm, st>>>(V, w, n, chunk, j + 1, 1, sigma.real(), sigma.imag(), part, h1, ticket);
        combine_kernel<T><<<g, SV_THREADS, 0, st>>>(V, h1, j + 1, -1.0, w, n, chunk, part, nullptr, ticket);
        dots_kernel<T><<<g, SV_THREADS, sm, st>>>(V, w, n, chunk, j + 1, 0, 0.0, 0.0, part, h2, ticket);
        combine_kernel<T><<<g, SV_THREADS, 0, st>>>(V, h2, j + 1, -1.0, w, n, chunk, part, nrm, ticket);
        normalise_kernel<T><<<(unsigned)std::min<int64_t>(SV_BLOCKS, (n + SV_THREADS - 1) / SV_THREADS), SV_THREADS, 0, st>>>(
            w, nrm, V + (size_t)(j + 1) * n, n, j + 1, h1, h2, col);
        HFMM_CUDA_TRY(cudaGetLastError());
        return read(col, j + 2);
    }
    // y = a x + b y
    hfmm_status axpby(zc a, const T* x, zc b, T* y) {
        axpby_kernel<T><<<SV_BLOCKS, SV_THREADS, 0, st>>>(a.real(), a.imag(), x, b.real(), b.imag(), y, n);
        HFMM_CUDA_TRY(cudaGetLastError());
        return HFMM_OK;
    }
    hfmm_status apply(const T* v, T* y) {
        if (P->precision == HFMM_MIXED)
            return apply_mixed(P, 1, (const cf*)v, (cf*)y, HFMM_PART_ALL, false, st);
        return apply_fp64(P, 1, (const cd*)v, (cd*)y, HFMM_PART_ALL, false, st);
    }
    // y = sigma v + A v
    hfmm_status op(zc sigma, const T* v, T* y) {
        HFMM_TRY(apply(v, y));
        return axpby(sigma, v, zc(1.0, 0.0), y);
    }
};

template <class T>
hfmm_status gmres(hfmm_plan_s* P, zc sigma, const T* b, T* x, double tol, int m, int maxit, int* iters,
                  double* relres, cudaStream_t st) {
    const int64_t n = P->n;
    // workspace: m + 1 Krylov vectors and one more, kept by the plan
    const size_t need = sizeof(T) * (size_t)n * (m + 2);
    if (!P->krylov || P->krylov_bytes < need) {
        HFMM_TRY(plan_alloc(P, (void**)&P->krylov, need));
        P->krylov_bytes = need;
    }
    // small arrays: a pass's block sums [m + 1][blocks], its dot products (twice), a norm, a column, the ticket
    // two blocks per SM where the vectors are long enough, at most 2048 elements a block
    const int chunk = (int)std::min<int64_t>(2048, std::max<int64_t>(32, (n + 303) / 304));
    const size_t nblk = (size_t)((n + chunk - 1) / chunk);
    const size_t words = (size_t)(m + 1) * nblk + 3 * (size_t)(m + 2) + 2;
    if (!P->krylov_part || P->krylov_words < words) {
        HFMM_TRY(plan_alloc(P, (void**)&P->krylov_part, sizeof(double2) * words));
        P->krylov_words = words;
    }
    if (!P->krylov_host || P->krylov_host_words < (size_t)m + 2) {
        if (P->krylov_host) cudaFreeHost(P->krylov_host);
        P->krylov_host = nullptr;
        double2* made = nullptr;
        HFMM_CUDA_TRY(cudaMallocHost((void**)&made, sizeof(double2) * ((size_t)m + 2)));
        P->krylov_host = made;
        P->krylov_host_words = (size_t)m + 2;
    }
    double2* small = P->krylov_part;
    Krylov<T> K{P, st, n, small + 3 * (size_t)(m + 2) + 2, small, small + (m + 2), small + 3 * (size_t)(m + 2),
                small + 2 * (size_t)(m + 2), P->krylov_host, (unsigned*)(small + 3 * (size_t)(m + 2) + 1), chunk, false};
    HFMM_TRY(K.choose_cgs(m));
    HFMM_CUDA_TRY(cudaMemsetAsync(K.ticket, 0, sizeof(unsigned), st));
    T* V = (T*)P->krylov;
    T* w = V + (size_t)n * (m + 1);
    auto vec = [&](int j) { return V + (size_t)n * j; };
    double bb;
    HFMM_CUDA_TRY(cudaMemcpyAsync(w, b, sizeof(T) * n, cudaMemcpyDeviceToDevice, st));
    HFMM_TRY(K.norm2(w, &bb));
    const double bnorm = std::sqrt(bb);
    *iters = 0;
    *relres = 0.0;
    if (bnorm == 0.0) {
        HFMM_CUDA_TRY(cudaMemsetAsync(x, 0, sizeof(T) * n, st));
        HFMM_CUDA_TRY(cudaStreamSynchronize(st));
        return HFMM_OK;
    }
    std::vector<zc> H((size_t)(m + 1) * m), g(m + 1), cs(m), sn(m), y(m);
    while (*iters < maxit) {
        // r = b - (sigma x + A x) into V_0
        HFMM_TRY(K.op(sigma, x, vec(0)));
        HFMM_TRY(K.axpby(zc(1.0, 0.0), b, zc(-1.0, 0.0), vec(0)));
        double rr;
        HFMM_TRY(K.norm2(vec(0), &rr));
        const double beta = std::sqrt(rr);
        *relres = beta / bnorm;
        if (*relres <= tol) break;
        HFMM_TRY(K.axpby(zc(1.0 / beta, 0.0), vec(0), zc(0.0, 0.0), vec(0)));
        std::fill(g.begin(), g.end(), zc(0.0, 0.0));
        g[0] = beta;
        int j = 0;
        for (; j < m && *iters < maxit; ++j) {
            ++*iters;
            HFMM_TRY(K.arnoldi(sigma, V, j, w));
            for (int i = 0; i <= j; ++i) H[(size_t)i * m + j] = zc(K.host[i].x, K.host[i].y);
            const double hn = std::sqrt(K.host[j + 1].x);
            H[(size_t)(j + 1) * m + j] = hn;
            // Givens rotations: apply the previous ones to column j, make a new one
            for (int i = 0; i < j; ++i) {
                const zc a = H[(size_t)i * m + j], c = H[(size_t)(i + 1) * m + j];
                H[(size_t)i * m + j] = std::conj(cs[i]) * a + std::conj(sn[i]) * c;
                H[(size_t)(i + 1) * m + j] = -sn[i] * a + cs[i] * c;
            }
            const zc a = H[(size_t)j * m + j];
            const double den = std::sqrt(std::norm(a) + hn * hn);
            cs[j] = den > 0.0 ? a / den : zc(1.0, 0.0);
            sn[j] = den > 0.0 ? zc(hn / den, 0.0) : zc(0.0, 0.0);
            H[(size_t)j * m + j] = den;
            H[(size_t)(j + 1) * m + j] = 0.0;
            g[j + 1] = -sn[j] * g[j];
            g[j] = std::conj(cs[j]) * g[j];
            *relres = std::abs(g[j + 1]) / bnorm;
            if (*relres <= tol || hn == 0.0) { ++j; break; }
        }
        // y = H(0:j, 0:j)^-1 g(0:j); x += V y
        for (int i = j - 1; i >= 0; --i) {
            zc s = g[i];
            for (int k = i + 1; k < j; ++k) s -= H[(size_t)i * m + k] * y[k];
            y[i] = s / H[(size_t)i * m + i];
        }
        for (int i = 0; i < j; ++i) K.host[i] = make_double2(y[i].real(), y[i].imag());
        HFMM_CUDA_TRY(cudaMemcpyAsync(K.col, K.host, sizeof(double2) * j, cudaMemcpyHostToDevice, st));
        combine_kernel<T><<<K.blocks(), SV_THREADS, 0, st>>>(V, K.col, j, 1.0, x, n, chunk, K.part, nullptr, K.ticket);
        HFMM_CUDA_TRY(cudaGetLastError());
        if (*relres <= tol) break;
    }
    // the true residual of the returned x
    HFMM_TRY(K.op(sigma, x, w));
    HFMM_TRY(K.axpby(zc(1.0, 0.0), b, zc(-1.0, 0.0), w));
    double rr;
    HFMM_TRY(K.norm2(w, &rr));
    *relres = std::sqrt(rr) / bnorm;
    return HFMM_OK;
}

}  // namespace

extern "C" hfmm_status hfmm_solve(hfmm_plan_t P, const double* sigma, const void* b, void* x, double tol,
                                  int32_t restart, int32_t maxit, int32_t* iters, double* relres, void* stream) {
    if (!P || !sigma || !b || !x || !iters || !relres) {
        hfmm_set_error("hfmm_solve: null argument");
        return HFMM_ERR_INVALID_ARG;
    }
    if (!(tol > 0.0) || restart < 1 || restart > 1000 || maxit < 1) {
        hfmm_set_error("hfmm_solve: need tol > 0, 1 <= restart <= 1000, maxit >= 1");
        return HFMM_ERR_INVALID_ARG;
    }
    for (const void* p : {b, (const void*)x}) {
        cudaPointerAttributes a;
        const bool dev = cudaPointerGetAttributes(&a, p) == cudaSuccess && a.type == cudaMemoryTypeDevice;
        cudaGetLastError();
        if (!dev) {
            hfmm_set_error("hfmm_solve: b and x must be device buffers");
            return HFMM_ERR_INVALID_ARG;
        }
    }
    const zc s(sigma[0], sigma[1]);
    cudaStream_t st = (cudaStream_t)stream;
    int it = 0;
    double rr = 0.0;
    hfmm_status status = P->precision == HFMM_MIXED
                             ? gmres<cf>(P, s, (const cf*)b, (cf*)x, tol, restart, maxit, &it, &rr, st)
                             : gmres<cd>(P, s, (const cd*)b, (cd*)x, tol, restart, maxit, &it, &rr, st);
    *iters = it;
    *relres = rr;
    if (status != HFMM_OK) return status;
    if (rr > tol) {
        hfmm_set_error("hfmm_solve: relative residual %.3g after %d iterations (tol %.3g)", rr, it, tol);
        return HFMM_ERR_NUMERICS;
    }
    return HFMM_OK;
}
