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

// Two values at once over a warp, in one shuffle more than one takes: lanes 0..15 get a's result, lanes 16..31 b's.
__device__ __forceinline__ double ss_pair_sum(double a, double b)
{
    const bool upper = (threadIdx.x & 16) != 0;
    double v = upper ? b : a;
    v += __shfl_xor_sync(0xFFFFFFFFu, upper ? a : b, 16);
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    return v;
}
__device__ __forceinline__ float ss_pair_min(float a, float b)
{
    const bool upper = (threadIdx.x & 16) != 0;
    float v = upper ? b : a;
    v = fminf(v, __shfl_xor_sync(0xFFFFFFFFu, upper ? a : b, 16));
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) v = fminf(v, __shfl_xor_sync(0xFFFFFFFFu, v, o));
    return v;
}

// Two sums, a smallest and a largest value and a count over the block, for the lanes of warp 0 (the warps' results in a fixed
// order); the other warps have stored theirs and are behind the block barrier.  RANGE: lo and hi are wanted.
struct SsBlock { double sum[2 * SS_WARPS]; float least[2 * SS_WARPS]; unsigned count[SS_WARPS]; };
struct SsParts { double a, b; float lo, hi; unsigned count; };
template <bool RANGE>
__device__ __forceinline__ SsParts ss_block_parts(SsParts v, SsBlock& sh)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __syncwarp();                                             // (lanes that have parted take a shuffle one after another)
    const double s = ss_pair_sum(v.a, v.b);
    float l = 0.f;
    if (RANGE) l = ss_pair_min(v.lo, -v.hi);
    const unsigned c = __reduce_add_sync(0xFFFFFFFFu, v.count);
    if ((lane & 15) == 0) {
        sh.sum[lane + warp] = s;
        if (RANGE) sh.least[lane + warp] = l;
        if (lane == 0) sh.count[warp] = c;
    }
    static_assert(SS_WARPS == 16, "a lane per warp's sum and half");
    __syncthreads();
    if (warp == 0) {
        double t = sh.sum[lane];
        float m = RANGE ? sh.least[lane] : 0.f;
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) {
            t += __shfl_xor_sync(0xFFFFFFFFu, t, o);
            if (RANGE) m = fminf(m, __shfl_xor_sync(0xFFFFFFFFu, m, o));
        }
        v.a = __shfl_sync(0xFFFFFFFFu, t, 0);
        v.b = __shfl_sync(0xFFFFFFFFu, t, 16);
        if (RANGE) {
            v.lo = __shfl_sync(0xFFFFFFFFu, m, 0);
            v.hi = -__shfl_sync(0xFFFFFFFFu, m, 16);
        }
        v.count = __reduce_add_sync(0xFFFFFFFFu, lane < SS_WARPS ? sh.count[lane] : 0u);
    }
    return v;
}

// Block partials: rows of 16 bytes per block.  All blocks read all of them at the same time, so what counts is how few sectors of
// L2 a merge asks for: with a partial's five doubles 64 bytes apart from the next block's, the slowest of 148 blocks had the sums of
// phase A 6 us after the fastest; with two rows of 16 bytes it is within 1 us.  One warp, SS_MERGE blocks per lane in flight;
// take(u): the ROWS vectors of a block, in order of its number per lane.
__device__ __forceinline__ uint4 ss_row(double a, double b)
{
    const unsigned long long u = (unsigned long long)__double_as_longlong(a), v = (unsigned long long)__double_as_longlong(b);
    return make_uint4((unsigned)u, (unsigned)(u >> 32), (unsigned)v, (unsigned)(v >> 32));
}
__device__ __forceinline__ double ss_row_first(const uint4& r) { return __hiloint2double((int)r.y, (int)r.x); }
__device__ __forceinline__ double ss_row_second(const uint4& r) { return __hiloint2double((int)r.w, (int)r.z); }
// In a cluster the rows go into every block's shared memory instead, rows[r][block]: by warp 0, a lane per block, before the
// cluster's barrier; behind it lane b < G has block b's.
typedef uint4 SsRows[16];                                     // of as many blocks as a cluster has at most
__device__ __forceinline__ void ss_push(SsRows& row, unsigned G, const uint4& v)
{
    const unsigned lane = threadIdx.x & 31;
    if (lane < G) {
        unsigned at;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(at) : "r"((unsigned)__cvta_generic_to_shared(&row[blockIdx.x])), "r"(lane));
        asm volatile("st.shared::cluster.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(at), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
    }
    __syncwarp();
}
template <int ROWS, typename F>
__device__ __forceinline__ void ss_merge_pushed(const SsRows* rows, unsigned G, F&& take)
{
    const unsigned b = threadIdx.x & 31;
    if (b < G) {
        uint4 p[ROWS];
#pragma unroll
        for (int r = 0; r < ROWS; ++r) p[r] = rows[r][b];
        take(p);
    }
}
template <int ROWS, typename F>
__device__ __forceinline__ void ss_merge(const uint4* part, unsigned G, F&& take)
{
    for (unsigned b0 = threadIdx.x & 31; b0 < G; b0 += 32 * SS_MERGE) {
        uint4 p[SS_MERGE][ROWS];
#pragma unroll
        for (int u = 0; u < SS_MERGE; ++u)
#pragma unroll
            for (int r = 0; r < ROWS; ++r)
                if (b0 + 32 * u < G) p[u][r] = __ldcg(part + (size_t)r * G + b0 + 32 * u);
#pragma unroll
        for (int u = 0; u < SS_MERGE; ++u)
            if (b0 + 32 * u < G) take(p[u]);
    }
}

// A warp's first tile; the others follow `step` tiles apart.  Up to 32 tiles a warp, warp w of block b starts with tile w G + b, so that
// the last tiles are spread over the blocks (closed-form sender, 27 M bf16 elements at 6 bits: 38.6 us, 39.8 with a block's warps side
// by side; 51 M fp32 at 3 bits 84.2 and 85.5); beyond that the last tiles count for less than the 64 KB that a block's warps
// read side by side (90 M fp32 at 8 bits: 146 us spread, 141.8 side by side; 268 M: 392 and 386).
__device__ __forceinline__ uint64_t ss_first_tile(uint64_t ntiles, uint64_t step)
{
    const unsigned w = threadIdx.x >> 5;
    return ntiles <= 32 * step ? w * gridDim.x + blockIdx.x : blockIdx.x * SS_WARPS + w;
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


// The elements behind the last whole tile, for the last block: loaded once, up to two per thread, and kept for all passes.  (As loads in
// every pass, after its own, they were the longest chain of a small tensor's.)
struct SsTail {
    float v[2];
    int m;
    template <typename T>
    __device__ __forceinline__ void load(const T* x, uint64_t tail0, uint64_t n, bool mine)
    {
        static_assert(SS_TILE <= 2 * SS_THREADS, "two per thread");
        m = 0;
        v[0] = v[1] = 0.f;
        const uint64_t i = tail0 + threadIdx.x;
        if (mine && i < n) {
            v[0] = qp_load_one(x + i);
            m = 1;
            if (i + SS_THREADS < n) { v[1] = qp_load_one(x + i + SS_THREADS); m = 2; }
        }
    }
    template <typename F>
    __device__ __forceinline__ void each(F&& f) const
    {
        if (m > 0) f(v[0]);
        if (m > 1) f(v[1]);
        __syncwarp();
    }
};

// ---- launches whose blocks wait for one another: a cooperative grid, or one thread-block cluster
constexpr unsigned QP_CLUSTER_BLOCKS = 16;        // the largest cluster (above 8: by attribute, where the device has the SMs)

// One cluster while every warp of it has at most one tile.  The search sender with 2 bits at 2^17, 2^18, 3 * 2^17 and 2^20 fp32 elements
// takes 19.6, 20.9, 23.0 and 31.2 us in a cluster, 22.6, 22.9, 23.0 and 23.0 in a grid; the closed form at 8 bits 10.6, 10.6, 11.6 and
// 16.1, and 12.7 in a grid.
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

// Blocks of such a launch: a tile per warp.  (In a cluster a block per tile, up to 16, gains on the passes what it loses on the
// barriers: one image at 8 bits the same, with the search at 2 bits 20.1 us against 19.0.)
inline unsigned qp_together_blocks(const qp_ctx* ctx, int cluster, uint64_t ntiles)
{
    const uint64_t most = cluster ? QP_CLUSTER_BLOCKS : (uint64_t)ctx->sm_count, want = (ntiles + SS_WARPS - 1) / SS_WARPS;
    return (unsigned)(want < most ? want : most);
}

inline cudaError_t qp_launch_together(void* kernel, unsigned G, unsigned threads, void** params, size_t bytes, int cluster, cudaStream_t s)
{
    if (!cluster) return cudaLaunchCooperativeKernel(kernel, dim3(G), dim3(threads), params, bytes, s);
    cudaLaunchAttribute at;
    const cudaLaunchConfig_t cfg = qp_cluster_config(&at, G, threads, bytes, s);
    return cudaLaunchKernelExC(&cfg, kernel, params);
}
