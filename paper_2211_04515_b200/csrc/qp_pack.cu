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
#include "qp_internal.cuh"

namespace {

constexpr int TILE = 1024;                 // elements per warp tile
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

// physical word of quad p in a warp's 256-word staging buffer: 16-byte chunk index XOR bit 3
__device__ __forceinline__ int swz(int p) { return ((((p >> 2) ^ ((p >> 5) & 1)) << 2) | (p & 3)); }

template <int BITS>
__device__ __forceinline__ unsigned quad_of(const float* e, const QP4& q)
{
    unsigned r = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) r |= qp_code(e[i], q.lo, q.hi, q.inv, q.mask) << (BITS * i);
    return r;
}

// ntiles counts the last, partial tile too: its missing elements are NaN (code 0) and its words are
// written up to nwords, pad words included.  VEC: x is 16-byte aligned.  Otherwise every lane loads the
// elements of its vectors one by one (the four loads of a vector touch the same lines, so they hit L1).
template <int BITS, typename T, bool VEC>
__global__ void __launch_bounds__(QP_THREADS) pack_kernel(const T* __restrict__ x, uint64_t n, uint64_t ntiles,
                                                          const qp_qparams_t* __restrict__ d_qp, qp_qparams_t h_qp,
                                                          uint32_t* __restrict__ out, uint64_t nwords,
                                                          unsigned* __restrict__ status, int reverse)
{
    constexpr int EPV = qp_span<T>::EPV;          // 4 (f32) or 8 (bf16) elements per 16-byte vector
    constexpr int NLOAD = TILE / (32 * EPV);      // 8 or 4 vector loads per lane
    __shared__ __align__(16) uint32_t stage[WARPS][256];
    const QP4 q = load_qp(d_qp, h_qp, BITS, status);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t* sw = stage[warp];
    const unsigned warps = blockDim.x >> 5;
    const uint64_t wstride = (uint64_t)gridDim.x * warps;

    // `reverse`: the grid walks the tensor from its end (the tiles are the same), for a call that
    // follows a pass which ended there and left that part of x in L2
    for (uint64_t it = (uint64_t)blockIdx.x * warps + warp; it < ntiles; it += wstride) {
        const uint64_t tile = reverse ? ntiles - 1 - it : it;
        const T* xt = x + tile * TILE;
        const bool full = (tile + 1) * TILE <= n;                 // warp-uniform
        float e[NLOAD][EPV];
        if (full) {
#pragma unroll
            for (int j = 0; j < NLOAD; ++j) {
                if constexpr (VEC) {
                    qp_load_vec(xt + (j * 32 + lane) * EPV, e[j]);
                } else {
#pragma unroll
                    for (int i = 0; i < EPV; ++i) e[j][i] = qp_load_one(xt + (j * 32 + lane) * EPV + i);
                }
            }
        } else {
            const int have = (int)(n - tile * TILE);
#pragma unroll
            for (int j = 0; j < NLOAD; ++j)
#pragma unroll
                for (int i = 0; i < EPV; ++i) {
                    const int k = (j * 32 + lane) * EPV + i;
                    e[j][i] = k < have ? qp_load_one(xt + k) : __int_as_float(0x7FC00000);
                }
        }
#pragma unroll
        for (int j = 0; j < NLOAD; ++j) {
            if constexpr (EPV == 4) {
                sw[swz(j * 32 + lane)] = quad_of<BITS>(e[j], q);
            } else {
                uint2 two;
                two.x = quad_of<BITS>(e[j], q);
                two.y = quad_of<BITS>(e[j] + 4, q);
                *reinterpret_cast<uint2*>(&sw[swz(2 * (j * 32 + lane))]) = two;
            }
        }
        __syncwarp();
        const uint4 a = *reinterpret_cast<const uint4*>(&sw[swz(8 * lane)]);
        const uint4 b = *reinterpret_cast<const uint4*>(&sw[swz(8 * lane + 4)]);
        const uint32_t qd[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
        uint32_t w[BITS];
#pragma unroll
        for (int m = 0; m < BITS; ++m) w[m] = 0u;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            constexpr int QB = 4 * BITS;
            const int bit = QB * k, word = bit >> 5, sh = bit & 31;
            w[word] |= qd[k] << sh;
            if (sh + QB > 32) w[(word + 1) % BITS] |= qd[k] >> (32 - sh);
        }
        uint32_t* ot = out + tile * (32 * BITS);
        if (full && BITS == 8) {
            uint4* o = reinterpret_cast<uint4*>(ot + lane * 8);
            o[0] = make_uint4(w[0], w[1 % BITS], w[2 % BITS], w[3 % BITS]);
            o[1] = make_uint4(w[4 % BITS], w[5 % BITS], w[6 % BITS], w[7 % BITS]);
        } else if (full && BITS == 4) {
            *reinterpret_cast<uint4*>(ot + lane * 4) = make_uint4(w[0], w[1 % BITS], w[2 % BITS], w[3 % BITS]);
        } else if (full && BITS == 2) {
            *reinterpret_cast<uint2*>(ot + lane * 2) = make_uint2(w[0], w[1 % BITS]);
        } else {
            __syncwarp();
#pragma unroll
            for (int m = 0; m < BITS; ++m) sw[lane * BITS + m] = w[m];
            __syncwarp();
            const int room = (int)min((uint64_t)(32 * BITS), nwords - tile * (32 * BITS));
#pragma unroll
            for (int m = 0; m < BITS; ++m)
                if (m * 32 + lane < room) ot[m * 32 + lane] = sw[m * 32 + lane];
        }
        __syncwarp();
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
