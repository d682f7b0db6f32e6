// a6: unpack + dequantize, the receiver's side (paper Sec. 3).  y_i = fma(code_i, scale, lo).
//
// HBM-bound and write-dominated: bits/8 bytes read, 4 (or 2) bytes written per element.
//
// Fast path, bits 1..8: the mirror image of the packer.  A warp owns 1024 elements
// (= 32*bits packed words).  Lane l fetches its `bits` words (widest aligned vector for
// bits 1,2,4,8; 128-byte coalesced through shared memory otherwise), cuts them into the 8
// "quads" (4 codes each) of its 32 consecutive elements, and the quads cross the warp
// through a chunk-swizzled 1 KB staging buffer so that lane l then expands quad j*32+l and
// stores 16-byte vectors that are fully coalesced across the warp.  The last, partial tile is a guarded
// iteration of the same loop, and an output that is not aligned takes element stores: one launch.
//
// HOST: the receiver on host buffers.  The kernel reads the packed words from page-locked memory and writes the elements to
// the work buffer and to page-locked memory, so both directions of the link are busy at once and the two copies around the
// kernel, 4 us each and in series with it, are gone.  What bounds it: the link, 49 GB/s of stores (a copy engine's 55).  One image
// at 8 bits: 19 us against 35 (bf16 14.5 / 26), 1.2 M elements 111 / 126 (bf16 65 / 84), 4.2 M 389 / 391 (230 / 246).
#include <cuda.h>

#include "qp_internal.cuh"

namespace {

constexpr int TILE = 1024;
constexpr int WARPS = QP_THREADS / 32;

struct DQ { float lo, scale; };

__device__ __forceinline__ DQ load_dq(const qp_qparams_t* __restrict__ d_qp, const qp_qparams_t& h_qp, int bits,
                                      unsigned* status)
{
    DQ q;
    if (d_qp) {
        q.lo = __ldg(&d_qp->lo); q.scale = __ldg(&d_qp->scale);
        if (blockIdx.x == 0 && threadIdx.x == 0 && __ldg(&d_qp->bits) != bits) atomicOr(status, QP_DEV_BITS_MISMATCH);
    } else {
        q.lo = h_qp.lo; q.scale = h_qp.scale;
    }
    return q;
}

__device__ __forceinline__ int swz(int p) { return ((((p >> 2) ^ ((p >> 5) & 1)) << 2) | (p & 3)); }

// integer code (< 2^23) to float without a conversion instruction: 2^23 + c, minus 2^23
__device__ __forceinline__ float code_to_float(unsigned c) { return __fsub_rn(__uint_as_float(0x4B000000u | c), 8388608.0f); }

__device__ __forceinline__ float dequant(unsigned c, const DQ& q) { return fmaf(code_to_float(c), q.scale, q.lo); }

__device__ __forceinline__ void store_out(float* y, uint64_t i4, const float (&v)[4])
{
    __stcs(reinterpret_cast<float4*>(y) + i4, make_float4(v[0], v[1], v[2], v[3]));
}
__device__ __forceinline__ void store_out(unsigned short* y, uint64_t i4, const float (&v)[4])
{
    uint2 o;
    o.x = (unsigned)qp_f32_to_bf16(v[0]) | ((unsigned)qp_f32_to_bf16(v[1]) << 16);
    o.y = (unsigned)qp_f32_to_bf16(v[2]) | ((unsigned)qp_f32_to_bf16(v[3]) << 16);
    __stcs(reinterpret_cast<uint2*>(y) + i4, o);
}
__device__ __forceinline__ void store_one(float* y, uint64_t i, float v) { y[i] = v; }
__device__ __forceinline__ void store_one(unsigned short* y, uint64_t i, float v) { y[i] = qp_f32_to_bf16(v); }

// One tile; unless it has all its elements (ALL: the caller knows that it has), its words are read up to nwords and its elements written up to n.  VEC: y
// is aligned for 4-element stores; otherwise the elements are stored one by one.
template <int BITS, typename TO, bool VEC, bool HOST, bool ALL = false>
__device__ __forceinline__ void unpack_tile(const uint32_t* __restrict__ in, uint64_t n, uint64_t nwords, uint64_t tile, int lane,
                                            const DQ& q, uint32_t* sw, TO* __restrict__ y, uint32_t* __restrict__ work,
                                            TO* __restrict__ y_host)
{
    constexpr unsigned MASK = (1u << BITS) - 1u;
    constexpr int QB = 4 * BITS;
    constexpr unsigned QMASK = QB >= 32 ? 0xFFFFFFFFu : ((1u << (QB & 31)) - 1u);
    const uint32_t* it = in + tile * (32 * BITS);
    uint32_t* wk = HOST ? work + tile * (32 * BITS) : nullptr;
    bool full = (tile + 1) * TILE <= n;                           // warp-uniform
    if (ALL) full = true;
    uint32_t w[BITS];
    if (full && BITS == 8) {
        const uint4 a = __ldg(reinterpret_cast<const uint4*>(it + lane * 8));
        const uint4 b = __ldg(reinterpret_cast<const uint4*>(it + lane * 8) + 1);
        w[0] = a.x; w[1 % BITS] = a.y; w[2 % BITS] = a.z; w[3 % BITS] = a.w;
        w[4 % BITS] = b.x; w[5 % BITS] = b.y; w[6 % BITS] = b.z; w[7 % BITS] = b.w;
        if constexpr (HOST) {
            *reinterpret_cast<uint4*>(wk + lane * 8) = a;
            *(reinterpret_cast<uint4*>(wk + lane * 8) + 1) = b;
        }
    } else if (full && BITS == 4) {
        const uint4 a = __ldg(reinterpret_cast<const uint4*>(it + lane * 4));
        w[0] = a.x; w[1 % BITS] = a.y; w[2 % BITS] = a.z; w[3 % BITS] = a.w;
        if constexpr (HOST) *reinterpret_cast<uint4*>(wk + lane * 4) = a;
    } else if (full && BITS == 2) {
        const uint2 a = __ldg(reinterpret_cast<const uint2*>(it + lane * 2));
        w[0] = a.x; w[1 % BITS] = a.y;
        if constexpr (HOST) *reinterpret_cast<uint2*>(wk + lane * 2) = a;
    } else {
        const int room = ALL ? 32 * BITS : (int)min((uint64_t)(32 * BITS), nwords - tile * (32 * BITS));
#pragma unroll
        for (int m = 0; m < BITS; ++m) {
            const uint32_t v = m * 32 + lane < room ? __ldg(it + m * 32 + lane) : 0u;
            sw[m * 32 + lane] = v;
            if (HOST && m * 32 + lane < room) wk[m * 32 + lane] = v;
        }
        __syncwarp();
#pragma unroll
        for (int m = 0; m < BITS; ++m) w[m] = sw[lane * BITS + m];
        __syncwarp();
    }
    uint32_t qd[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const int bit = QB * k, word = bit >> 5, sh = bit & 31;
        uint32_t v = w[word] >> sh;
        if (sh + QB > 32) v |= w[(word + 1) % BITS] << (32 - sh);
        qd[k] = v & QMASK;
    }
    *reinterpret_cast<uint4*>(&sw[swz(8 * lane)]) = make_uint4(qd[0], qd[1], qd[2], qd[3]);
    *reinterpret_cast<uint4*>(&sw[swz(8 * lane + 4)]) = make_uint4(qd[4], qd[5], qd[6], qd[7]);
    __syncwarp();
    uint32_t mine[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) mine[j] = sw[swz(j * 32 + lane)];
    const int have = full ? TILE : (int)(n - tile * TILE);
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        float v[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) v[i] = dequant((mine[j] >> (BITS * i)) & MASK, q);
        const int k = (j * 32 + lane) * 4;
        if (VEC && (full || k + 4 <= have)) {
            store_out(y, tile * (TILE / 4) + j * 32 + lane, v);
            if constexpr (HOST) store_out(y_host, tile * (TILE / 4) + j * 32 + lane, v);
        } else {
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (k + i < have) {
                    store_one(y, tile * TILE + k + i, v[i]);
                    if constexpr (HOST) store_one(y_host, tile * TILE + k + i, v[i]);
                }
        }
    }
    __syncwarp();
}

// ntiles counts the last, partial tile too.  In the loop's body where a warp writes 4 KB a tile (fp32: 1 to 3 % faster at 2^26 elements
// and more), behind the loop where it writes 2 KB and the loop is bound by its instructions (bf16: 2^26 elements at 4 bits 51.3 us, 57.4
// with the partial tile's tests in the loop; 2^28 at 8 bits 169 and 191).
template <int BITS, typename TO, bool VEC, bool HOST = false>
__global__ void __launch_bounds__(QP_THREADS) unpack_kernel(const uint32_t* __restrict__ in, uint64_t n, uint64_t nwords,
                                                            uint64_t ntiles, const qp_qparams_t* __restrict__ d_qp,
                                                            qp_qparams_t h_qp, TO* __restrict__ y,
                                                            unsigned* __restrict__ status, uint32_t* __restrict__ work = nullptr,
                                                            TO* __restrict__ y_host = nullptr)
{
    __shared__ __align__(16) uint32_t stage[WARPS][256];
    const DQ q = load_dq(d_qp, h_qp, BITS, status);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t* sw = stage[warp];
    const unsigned warps = blockDim.x >> 5;
    const uint64_t wstride = (uint64_t)gridDim.x * warps;
    uint64_t tile = (uint64_t)blockIdx.x * warps + warp;
    if constexpr (sizeof(TO) == 2) {
        for (const uint64_t whole = n / TILE; tile < whole; tile += wstride)
            unpack_tile<BITS, TO, VEC, HOST, true>(in, n, nwords, tile, lane, q, sw, y, work, y_host);
        if (tile < ntiles) unpack_tile<BITS, TO, VEC, HOST>(in, n, nwords, tile, lane, q, sw, y, work, y_host);
    } else {
        for (; tile < ntiles; tile += wstride) unpack_tile<BITS, TO, VEC, HOST>(in, n, nwords, tile, lane, q, sw, y, work, y_host);
    }
}

// bits = 16: thread t expands one 16-byte vector of 8 codes.
template <typename TO, bool ALIGNED>
__global__ void __launch_bounds__(QP_THREADS) unpack16_kernel(const uint4* __restrict__ in, uint64_t n,
                                                              const qp_qparams_t* __restrict__ d_qp, qp_qparams_t h_qp,
                                                              TO* __restrict__ y, unsigned* __restrict__ status)
{
    const DQ q = load_dq(d_qp, h_qp, 16, status);
    const uint64_t nvec = (n + 7) / 8;
    const uint64_t stride = (uint64_t)gridDim.x * QP_THREADS;
    for (uint64_t v = (uint64_t)blockIdx.x * QP_THREADS + threadIdx.x; v < nvec; v += stride) {
        const uint4 a = __ldg(in + v);
        const unsigned c[8] = {a.x & 0xFFFFu, a.x >> 16, a.y & 0xFFFFu, a.y >> 16,
                               a.z & 0xFFFFu, a.z >> 16, a.w & 0xFFFFu, a.w >> 16};
        float f[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) f[i] = dequant(c[i], q);
        const uint64_t e0 = v * 8;
        if (ALIGNED && e0 + 8 <= n) {
            const float lo4[4] = {f[0], f[1], f[2], f[3]}, hi4[4] = {f[4], f[5], f[6], f[7]};
            store_out(y, v * 2, lo4);
            store_out(y, v * 2 + 1, hi4);
        } else {
#pragma unroll
            for (int i = 0; i < 8; ++i)
                if (e0 + i < n) store_one(y, e0 + i, f[i]);
        }
    }
}

template <typename TO>
int32_t unpack_typed(qp_ctx* ctx, const void* d_packed, uint64_t n, int bits, const qp_qparams_t* d_qp,
                     const qp_qparams_t& h_qp, TO* y, cudaStream_t s)
{
    const bool aligned = ((uintptr_t)y & 15u) == 0;
    if (bits == 16) {
        const uint64_t nvec = (n + 7) / 8;
        uint64_t want = (nvec + QP_THREADS - 1) / QP_THREADS;
        const uint64_t cap = (uint64_t)ctx->sm_count * 64;
        const int blocks = (int)(want > cap ? cap : want);
        ctx->launches += 1;
        if (aligned)
            unpack16_kernel<TO, true><<<blocks, QP_THREADS, 0, s>>>(static_cast<const uint4*>(d_packed), n, d_qp, h_qp, y, ctx->d_status);
        else
            unpack16_kernel<TO, false><<<blocks, QP_THREADS, 0, s>>>(static_cast<const uint4*>(d_packed), n, d_qp, h_qp, y, ctx->d_status);
        return qp_check_launch(ctx, "qp_unpack_dequantize");
    }
    const uint32_t* in = static_cast<const uint32_t*>(d_packed);
    const uint64_t nwords = qp_packed_bytes(n, bits) / 4, ntiles = (n + TILE - 1) / TILE;
    const qp_grid_shape g = qp_tile_grid(ctx, ntiles, WARPS);
    ctx->launches += 1;
#define QP_UNPACK_CASE(B)                                                                                                    \
    case B:                                                                                                                  \
        if (aligned) unpack_kernel<B, TO, true><<<g.blocks, g.threads, 0, s>>>(in, n, nwords, ntiles, d_qp, h_qp, y, ctx->d_status); \
        else unpack_kernel<B, TO, false><<<g.blocks, g.threads, 0, s>>>(in, n, nwords, ntiles, d_qp, h_qp, y, ctx->d_status);        \
        break;
    switch (bits) {
        QP_UNPACK_CASE(1) QP_UNPACK_CASE(2) QP_UNPACK_CASE(3) QP_UNPACK_CASE(4)
        QP_UNPACK_CASE(5) QP_UNPACK_CASE(6) QP_UNPACK_CASE(7) QP_UNPACK_CASE(8)
    }
#undef QP_UNPACK_CASE
    return qp_check_launch(ctx, "qp_unpack_dequantize");
}

template <typename TO>
int32_t unpack_host_typed(qp_ctx* ctx, const uint32_t* in, uint64_t n, int bits, const qp_qparams_t& h_qp, uint32_t* work, TO* y,
                          TO* y_host, cudaStream_t s)
{
    const uint64_t nwords = qp_packed_bytes(n, bits) / 4, ntiles = (n + TILE - 1) / TILE;
    const qp_grid_shape g = qp_tile_grid(ctx, ntiles, WARPS);
    ctx->launches += 1;
#define QP_UNPACK_CASE(B)                                                                                                      \
    case B:                                                                                                                    \
        unpack_kernel<B, TO, true, true>                                                                                       \
            <<<g.blocks, g.threads, 0, s>>>(in, n, nwords, ntiles, nullptr, h_qp, y, ctx->d_status, work, y_host);             \
        break;
    switch (bits) {
        QP_UNPACK_CASE(1) QP_UNPACK_CASE(2) QP_UNPACK_CASE(3) QP_UNPACK_CASE(4)
        QP_UNPACK_CASE(5) QP_UNPACK_CASE(6) QP_UNPACK_CASE(7) QP_UNPACK_CASE(8)
    }
#undef QP_UNPACK_CASE
    return qp_check_launch(ctx, "qp_receiver_host");
}

// The device's address of [p, p + bytes) inside one allocation or registration of page-locked host memory, or NULL.  (The
// runtime's attributes say nothing of its extent: two registrations with unlocked pages between them look alike at both ends.)
void* mapped(const void* p, uint64_t bytes)
{
    using Get = CUresult (*)(unsigned, CUpointer_attribute*, void**, CUdeviceptr);
    static const Get get = [] {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult r;
        if (cudaGetDriverEntryPoint("cuPointerGetAttributes", &f, cudaEnableDefault, &r) != cudaSuccess || r != cudaDriverEntryPointSuccess) {
            cudaGetLastError();
            f = nullptr;
        }
        return reinterpret_cast<Get>(f);
    }();
    unsigned type = 0;
    CUdeviceptr at = 0, start = 0;
    size_t size = 0;
    CUpointer_attribute what[] = {CU_POINTER_ATTRIBUTE_MEMORY_TYPE, CU_POINTER_ATTRIBUTE_DEVICE_POINTER,
                                  CU_POINTER_ATTRIBUTE_RANGE_START_ADDR, CU_POINTER_ATTRIBUTE_RANGE_SIZE};
    void* into[] = {&type, &at, &start, &size};
    if (!get || get(4, what, into, (CUdeviceptr)(uintptr_t)p) != CUDA_SUCCESS) return nullptr;
    const bool ok = type == CU_MEMORYTYPE_HOST && at && at >= start && bytes <= size && at - start <= size - bytes;
    return ok ? reinterpret_cast<void*>((uintptr_t)at) : nullptr;
}

bool apart(const void* a, uint64_t na, const void* b, uint64_t nb)
{
    return (uintptr_t)a + na <= (uintptr_t)b || (uintptr_t)b + nb <= (uintptr_t)a;
}

}  // namespace

// The receiver on page-locked, 16-byte aligned buffers in one launch, its status in *rc; false where it does not apply: copy
// engines move more than 16 MB of elements as fast or faster (their rate is the better one, and the copies' latencies no longer
// show).
bool qp_launch_unpack_host(qp_ctx* ctx, const void* h_packed, uint64_t n, int bits, const qp_qparams_t& h_qp, void* d_packed,
                           void* d_y, void* h_y, int out_dtype, cudaStream_t s, int32_t* rc)
{
    const uint64_t esz = out_dtype == QP_F32 ? 4 : 2;
    if (n == 0 || bits > 8 || h_qp.bits != bits || n * esz > 16ull << 20 ||
        (((uintptr_t)h_packed | (uintptr_t)d_packed | (uintptr_t)d_y | (uintptr_t)h_y) & 15u))
        return false;
    const void* in = mapped(h_packed, qp_packed_bytes(n, bits));
    void* out = in ? mapped(h_y, n * esz) : nullptr;
    if (!out) return false;
    // the kernel reads and writes at the same time, the copies one after the other: buffers that overlap are theirs
    const uint64_t np = qp_packed_bytes(n, bits), ny = n * esz;
    if (!apart(in, np, out, ny) || !apart(in, np, d_packed, np) || !apart(in, np, d_y, ny) || !apart(out, ny, d_packed, np) ||
        !apart(out, ny, d_y, ny))
        return false;
    if (out_dtype == QP_F32)
        *rc = unpack_host_typed<float>(ctx, static_cast<const uint32_t*>(in), n, bits, h_qp, static_cast<uint32_t*>(d_packed),
                                       static_cast<float*>(d_y), static_cast<float*>(out), s);
    else
        *rc = unpack_host_typed<unsigned short>(ctx, static_cast<const uint32_t*>(in), n, bits, h_qp, static_cast<uint32_t*>(d_packed),
                                                static_cast<unsigned short*>(d_y), static_cast<unsigned short*>(out), s);
    return true;
}

int32_t qp_launch_unpack(qp_ctx* ctx, const void* d_packed, uint64_t n, int bits, const qp_qparams_t* d_qp,
                         qp_qparams_t h_qp, void* d_y, int out_dtype, cudaStream_t s)
{
    if (out_dtype == QP_F32) return unpack_typed<float>(ctx, d_packed, n, bits, d_qp, h_qp, static_cast<float*>(d_y), s);
    return unpack_typed<unsigned short>(ctx, d_packed, n, bits, d_qp, h_qp, static_cast<unsigned short*>(d_y), s);
}
