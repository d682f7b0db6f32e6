// a5: clamp + uniform quantize + bit-pack (paper Sec. 3: uniform quantization of the clipped
// activation; the packed layout is this library's: element i owns stream bits
// [i*bits, (i+1)*bits), LSB first).
//
// HBM-bound: 4 (or 2) bytes read and bits/8 bytes written per element.
//
// Fast path, bits 1..8.  A warp owns a tile of 1024 consecutive elements, which is exactly
// 32*bits output words.  Loads are fully coalesced 16-byte vectors (lane l takes vector
// j*32+l, all of them issued before first use).  Each group of 4 consecutive elements is
// quantized to a "quad" of 4*bits bits; quads cross the warp through 1 KB of shared memory
// (chunk-swizzled, conflict-free both ways) so that every lane ends up with the 8 quads of
// 32 consecutive elements = `bits` whole 32-bit words, which it stores as the widest aligned
// vector (bits 1,2,4,8) or, for the other widths, through shared memory again so that global
// stores are 128-byte coalesced.
//
// bits = 16: one uint16 per element, plain vectorised map.
// The last, partial tile and the pad words are guarded iterations of the same loop, and an input that
// is not 16-byte aligned takes the same kernel with element loads: one launch for every shape.
#include "qp_packtile.cuh"

namespace {

constexpr int TILE = QP_TILE;
constexpr int WARPS = QP_THREADS / 32;

struct QP4 { float lo, hi, inv; unsigned mask; };

__device__ __forceinline__ QP4 load_qp(const qp_qparams_t* __restrict__ d_qp, const qp_qparams_t& h_qp, int bits,
                                       unsigned* status)
{
    QP4 q;
    if (d_qp) {
        q.lo = __ldg(&d_qp->lo); q.hi = __ldg(&d_qp->hi); q.inv = __ldg(&d_qp->inv_scale);
        if (blockIdx.x == 0 && threadIdx.x == 0 && __ldg(&d_qp->bits) != bits) atomicOr(status, QP_DEV_BITS_MISMATCH);
    } else {
        q.lo = h_qp.lo; q.hi = h_qp.hi; q.inv = h_qp.inv_scale;
    }
    q.mask = (bits >= 32) ? 0xFFFFFFFFu : ((1u << bits) - 1u);
    return q;
}

// ntiles counts the last, partial tile too: in the loop's body for fp32, behind the loop for bf16, whose loop is bound by its
// instructions (2^27 elements at 1, 3 and 6 bits: 47.2, 49.6 and 55.4 us, with the partial tile's tests in it 51.3, 54.6 and 59.5).
template <int BITS, typename T, bool VEC>
__global__ void __launch_bounds__(QP_THREADS) pack_kernel(const T* __restrict__ x, uint64_t n, uint64_t ntiles,
                                                          const qp_qparams_t* __restrict__ d_qp, qp_qparams_t h_qp,
                                                          uint32_t* __restrict__ out, uint64_t nwords,
                                                          unsigned* __restrict__ status, int reverse)
{
    __shared__ __align__(16) uint32_t stage[WARPS][256];
    const QP4 q = load_qp(d_qp, h_qp, BITS, status);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned warps = blockDim.x >> 5;
    const uint64_t wstride = (uint64_t)gridDim.x * warps;
    uint64_t it = (uint64_t)blockIdx.x * warps + warp;
    // `reverse`: the grid walks the tensor from its end (the tiles are the same), for a call that
    // follows a pass which ended there and left that part of x in L2
    if constexpr (sizeof(T) == 2) {
        const uint64_t whole = n / TILE;
        for (; it < whole; it += wstride)
            qp_pack_tile<BITS, T, VEC, true>(x, n, reverse ? whole - 1 - it : it, lane, q.lo, q.hi, q.inv, out, nwords, stage[warp]);
        if (it < ntiles) qp_pack_tile<BITS, T, VEC>(x, n, it, lane, q.lo, q.hi, q.inv, out, nwords, stage[warp]);
    } else {
        for (; it < ntiles; it += wstride)
            qp_pack_tile<BITS, T, VEC>(x, n, reverse ? ntiles - 1 - it : it, lane, q.lo, q.hi, q.inv, out, nwords, stage[warp]);
    }
}

// bits = 16: thread t converts the 8 elements [8t, 8t+8) to one 16-byte vector of uint16 codes.
template <typename T, bool ALIGNED>
__global__ void __launch_bounds__(QP_THREADS) pack16_kernel(const T* __restrict__ x, uint64_t n,
                                                            const qp_qparams_t* __restrict__ d_qp, qp_qparams_t h_qp,
                                                            uint4* __restrict__ out, uint64_t nvec_out,
                                                            unsigned* __restrict__ status)
{
    const QP4 q = load_qp(d_qp, h_qp, 16, status);
    const uint64_t stride = (uint64_t)gridDim.x * QP_THREADS;
    for (uint64_t v = (uint64_t)blockIdx.x * QP_THREADS + threadIdx.x; v < nvec_out; v += stride) {
        float e[8];
        const uint64_t e0 = v * 8;
        if (ALIGNED && e0 + 8 <= n) {
            if constexpr (sizeof(T) == 4) {
                float a[4], b[4];
                qp_load_vec(x + e0, a);
                qp_load_vec(x + e0 + 4, b);
#pragma unroll
                for (int i = 0; i < 4; ++i) { e[i] = a[i]; e[4 + i] = b[i]; }
            } else {
                qp_load_vec(x + e0, e);
            }
        } else {
#pragma unroll
            for (int i = 0; i < 8; ++i) e[i] = (e0 + i < n) ? qp_load_one(x + e0 + i) : __int_as_float(0x7FC00000);
        }
        unsigned c[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) c[i] = (e0 + i < n) ? qp_code(e[i], q.lo, q.hi, q.inv, q.mask) : 0u;
        out[v] = make_uint4(c[0] | (c[1] << 16), c[2] | (c[3] << 16), c[4] | (c[5] << 16), c[6] | (c[7] << 16));
    }
}

template <typename T>
int32_t pack_typed(qp_ctx* ctx, const T* x, uint64_t n, int bits, const qp_qparams_t* d_qp, const qp_qparams_t& h_qp,
                   void* d_packed, cudaStream_t s)
{
    const bool aligned = ((uintptr_t)x & 15u) == 0;
    if (bits == 16) {
        const uint64_t nvec_out = qp_packed_bytes(n, 16) / 16;
        uint64_t want = (nvec_out + QP_THREADS - 1) / QP_THREADS;
        const uint64_t cap = (uint64_t)ctx->sm_count * 64;
        const int blocks = (int)(want > cap ? cap : want);
        ctx->launches += 1;
        if (aligned)
            pack16_kernel<T, true><<<blocks, QP_THREADS, 0, s>>>(x, n, d_qp, h_qp, static_cast<uint4*>(d_packed), nvec_out, ctx->d_status);
        else
            pack16_kernel<T, false><<<blocks, QP_THREADS, 0, s>>>(x, n, d_qp, h_qp, static_cast<uint4*>(d_packed), nvec_out, ctx->d_status);
        return qp_check_launch(ctx, "qp_quantize_pack");
    }
    const uint64_t nwords = qp_packed_bytes(n, bits) / 4;
    const uint64_t ntiles = (n + TILE - 1) / TILE;
    uint32_t* out = static_cast<uint32_t*>(d_packed);
    // a hint, not a dependency: start where the last pass over this tensor stopped
    const int reverse = (ctx->last_x == static_cast<const void*>(x) && ctx->last_x_end) ? 1 : 0;
    ctx->last_x = x;
    ctx->last_x_end = reverse ? 0 : 1;
    const qp_grid_shape g = qp_tile_grid(ctx, ntiles, WARPS);
    ctx->launches += 1;
#define QP_PACK_CASE(B)                                                                                                        \
    case B:                                                                                                                    \
        if (aligned) pack_kernel<B, T, true><<<g.blocks, g.threads, 0, s>>>(x, n, ntiles, d_qp, h_qp, out, nwords, ctx->d_status, reverse); \
        else pack_kernel<B, T, false><<<g.blocks, g.threads, 0, s>>>(x, n, ntiles, d_qp, h_qp, out, nwords, ctx->d_status, reverse);        \
        break;
    switch (bits) {
        QP_PACK_CASE(1) QP_PACK_CASE(2) QP_PACK_CASE(3) QP_PACK_CASE(4)
        QP_PACK_CASE(5) QP_PACK_CASE(6) QP_PACK_CASE(7) QP_PACK_CASE(8)
    }
#undef QP_PACK_CASE
    return qp_check_launch(ctx, "qp_quantize_pack");
}

}  // namespace

int32_t qp_launch_pack(qp_ctx* ctx, const void* d_x, int dtype, uint64_t n, int bits, const qp_qparams_t* d_qp,
                       qp_qparams_t h_qp, void* d_packed, cudaStream_t s)
{
    if (dtype == QP_F32) return pack_typed<float>(ctx, static_cast<const float*>(d_x), n, bits, d_qp, h_qp, d_packed, s);
    return pack_typed<unsigned short>(ctx, static_cast<const unsigned short*>(d_x), n, bits, d_qp, h_qp, d_packed, s);
}
