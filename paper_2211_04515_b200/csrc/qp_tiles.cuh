// Pieces of the streaming cooperative kernels (one block of 512 threads per SM): block reductions and the walk over a
// tensor's tiles.
#pragma once

#include "qp_internal.cuh"

constexpr int SS_THREADS = 512;                   // 128 registers a thread; 768 and 1024 threads spill and were slower
constexpr int SS_WARPS = SS_THREADS / 32;
constexpr int SS_TILE = 1024;                     // elements of a warp tile: 32 per lane
constexpr int SS_MERGE = 5;                       // block partials per lane that are in flight in a merge

// Reduction of N values at once; OPS: 0 sum, 1 min, 2 max.  Lane 0 gets the results.
template <int... OPS>
__device__ __forceinline__ void ss_warp_reduce(double (&v)[sizeof...(OPS)])
{
    constexpr int N = sizeof...(OPS);
    constexpr int ops[N] = {OPS...};
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int j = 0; j < N; ++j) {
            const double t = __shfl_down_sync(0xFFFFFFFFu, v[j], o);
            v[j] = ops[j] == 0 ? v[j] + t : (ops[j] == 1 ? fmin(v[j], t) : fmax(v[j], t));
        }
}

// The same over the block; every thread gets the results, merged in warp order (the same bits in every block).
// sh: SS_WARPS * N doubles.
template <int... OPS>
__device__ __forceinline__ void ss_reduce(double (&v)[sizeof...(OPS)], double* sh)
{
    constexpr int N = sizeof...(OPS);
    constexpr int ops[N] = {OPS...};
    ss_warp_reduce<OPS...>(v);
    __syncthreads();
    if ((threadIdx.x & 31) == 0)
#pragma unroll
        for (int j = 0; j < N; ++j) sh[(threadIdx.x >> 5) * N + j] = v[j];
    __syncthreads();
#pragma unroll
    for (int j = 0; j < N; ++j) {
        double r = sh[j];
        for (int w = 1; w < SS_WARPS; ++w) {
            const double t = sh[w * N + j];
            r = ops[j] == 0 ? r + t : (ops[j] == 1 ? fmin(r, t) : fmax(r, t));
        }
        v[j] = r;
    }
}

// ---- streaming.  A warp works on tiles of N 16-byte vectors per lane, held in registers; a vector's registers are
// reloaded from the warp's next tile as soon as its elements have been taken out, so the loads of a whole tile are
// in flight all the time without a second set of registers or moves between the two.
template <typename T, int N>
struct SsStream {
    static constexpr int EPV = qp_span<T>::EPV, ELEMS = N * 32 * EPV;
    // tiles first, first + step, ... below ntiles (REVERSE: from the last one); f.begin() / f.pair(a, b, i) / f.end()
    // for every tile, by all lanes together; i = 0, 1, ... numbers the pairs of a tile
    template <bool REVERSE, typename F>
    static __device__ __forceinline__ void run(const T* x, uint64_t ntiles, uint64_t first, uint64_t step, int lane, F& f)
    {
        if (first >= ntiles) return;
        const uint64_t m = (ntiles - first + step - 1) / step;
        const uint4* p = reinterpret_cast<const uint4*>(x + (first + (REVERSE ? m - 1 : 0) * step) * ELEMS) + lane;
        const int64_t stride = (REVERSE ? -1 : 1) * (int64_t)(step * (ELEMS / EPV));
        uint4 v[N];
#pragma unroll
        for (int j = 0; j < N; ++j) v[j] = __ldg(p + j * 32);
        for (uint64_t i = 1; i <= m; ++i) {
            const bool more = i < m;
            if (more) p += stride;
            f.begin();
#pragma unroll
            for (int j = 0; j < N; ++j) {
                const uint4 w = v[j];
                if (more) v[j] = __ldg(p + j * 32);
                const unsigned u[4] = {w.x, w.y, w.z, w.w};
                if constexpr (sizeof(T) == 4) {
                    f.pair(__uint_as_float(u[0]), __uint_as_float(u[1]), 2 * j);
                    f.pair(__uint_as_float(u[2]), __uint_as_float(u[3]), 2 * j + 1);
                } else {
#pragma unroll
                    for (int h = 0; h < 4; ++h)
                        f.pair(__uint_as_float(u[h] << 16), __uint_as_float(u[h] & 0xFFFF0000u), 4 * j + h);
                }
            }
            f.end();
        }
    }
};
template <typename T, int ELEMS> using SsTiles = SsStream<T, ELEMS / 32 / qp_span<T>::EPV>;


// ---- launches whose blocks wait for one another: a cooperative grid, or one thread-block cluster
constexpr unsigned QP_CLUSTER_BLOCKS = 16;        // the largest cluster (above 8: by attribute, where the device has the SMs)

// One cluster while every warp of it has at most one tile; the search with 2 bits at 2^17, 2^18 and 3 * 2^17 elements takes 23,
// 24.7 and 28.8 us in a cluster, 26.7, 28.1 and 28.8 in a grid, at 2^20 35 and 28.8.
constexpr uint64_t QP_CLUSTER_MAX_N = (uint64_t)QP_CLUSTER_BLOCKS * SS_WARPS * SS_TILE;

inline cudaLaunchConfig_t qp_cluster_config(cudaLaunchAttribute* at, unsigned G, unsigned threads, size_t bytes, cudaStream_t s)
{
    at->id = cudaLaunchAttributeClusterDimension;
    at->val.clusterDim.x = G;
    at->val.clusterDim.y = at->val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(G);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = bytes;
    cfg.stream = s;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cfg;
}

// whether the device can hold `kernel` as a cluster of every size up to QP_CLUSTER_BLOCKS (the largest one tells)
inline int qp_cluster_fits(const void* kernel, unsigned threads, size_t bytes)
{
    cudaLaunchAttribute at;
    const cudaLaunchConfig_t cfg = qp_cluster_config(&at, QP_CLUSTER_BLOCKS, threads, bytes, nullptr);
    int clusters = 0;
    const bool ok = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
                    cudaOccupancyMaxActiveClusters(&clusters, kernel, &cfg) == cudaSuccess && clusters >= 1;
    if (!ok) cudaGetLastError();
    return ok ? 1 : 0;
}

// (the tests that make a barrier's wait run out have the counting barrier)
inline int qp_cluster_wanted(const qp_ctx* ctx, int fits, uint64_t n)
{
    return fits && n <= QP_CLUSTER_MAX_N && ctx->bar_extra == 0;
}

inline cudaError_t qp_launch_together(void* kernel, unsigned G, unsigned threads, void** params, size_t bytes, int cluster, cudaStream_t s)
{
    if (!cluster) return cudaLaunchCooperativeKernel(kernel, dim3(G), dim3(threads), params, bytes, s);
    cudaLaunchAttribute at;
    const cudaLaunchConfig_t cfg = qp_cluster_config(&at, G, threads, bytes, s);
    return cudaLaunchKernelExC(&cfg, kernel, params);
}
