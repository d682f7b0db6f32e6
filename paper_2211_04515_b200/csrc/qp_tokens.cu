// Token-wise variant of the path (a variant of this library: the paper, Sec. 3, uses one clip range
// per tensor).  The tensor is [tokens, channels], row-major; a token is a row of `channels`
// contiguous elements (one position of a ViT sequence) and gets the statistics, clip range and
// quantizer that the per-tensor functions give for its row alone.  Bit-width and packed layout
// are shared, so the receiver needs the `tokens` quantizers (24 bytes each) with the stream.
//
//   tok_stats_kernel    (rows that do not suit tok_rows_kernel) a warp per token: the row is read once from HBM (sums, min, max), the mean
//                       comes out of a warp reduction, and the second pass over the row (deviations)
//                       finds it in L1; fp32 partials per lane folded into fp64, fixed shuffle order
//   tok_pack_kernel     the per-tensor packer's warp tile (1024 elements = 32 * bits words, coalesced
//                       16-byte loads, quads across the warp through swizzled shared memory) with the
//                       quantizer looked up per 16-byte vector: a vector never straddles two tokens
//                       when `channels` is a multiple of the vector's elements, and a lane's vectors
//                       are 128 elements apart, so the token index moves on by a compare instead of
//                       a division
//   tok_unpack_kernel   the mirror image
//   tok_rows_kernel     the same statistics from rows in shared memory and, in the sender, clip, quantize and
//                       pack of the row as well
//   tok_*_scalar        any shape and alignment: a thread per 32 elements, token by division
#include "qp_packtile.cuh"

QP_CK_UNIT

namespace {

constexpr int TILE = 1024;
constexpr int WARPS = QP_THREADS / 32;

// ---------------------------------------------------------------------------- statistics

template <typename T, bool VEC>
__global__ void __launch_bounds__(QP_THREADS) tok_stats_kernel(const T* __restrict__ x, uint64_t tokens, uint32_t C,
                                                               qp_stats_t* __restrict__ out, unsigned* __restrict__ status)
{
    constexpr int EPV = qp_span<T>::EPV;
    const int lane = threadIdx.x & 31;
    const uint64_t wstride = (uint64_t)gridDim.x * WARPS;
    const float inf = __int_as_float(0x7F800000);
    bool any_bad = false;
    for (uint64_t t = (uint64_t)blockIdx.x * WARPS + (threadIdx.x >> 5); t < tokens; t += wstride) {
        const T* row = x + t * C;
        double s = 0.0, sa = 0.0;
        float mn = inf, mx = -inf;
        unsigned bad = 0;
        auto first = [&](float v) {
            if (qp_is_finite(v)) { s += (double)v; sa += (double)fabsf(v); mn = fminf(mn, v); mx = fmaxf(mx, v); }
            else ++bad;
        };
        if (VEC) {
            for (uint32_t v0 = lane; v0 < C / EPV; v0 += 32) {
                float e[EPV];
                qp_load_vec(row + (size_t)v0 * EPV, e);
                float ps = 0.f, psa = 0.f;
#pragma unroll
                for (int i = 0; i < EPV; ++i) { ps += e[i]; psa += fabsf(e[i]); mn = fminf(mn, e[i]); mx = fmaxf(mx, e[i]); }
                if (psa < inf) { s += (double)ps; sa += (double)psa; }
                else {                                       // a NaN or Inf among them (min/max may hold it: redone below)
                    mn = inf; mx = -inf; bad = 0xFFFFFFFFu;
                }
            }
            if (__any_sync(0xFFFFFFFFu, bad == 0xFFFFFFFFu)) {   // rare: the whole row again, element by element
                s = 0.0; sa = 0.0; mn = inf; mx = -inf; bad = 0;
                for (uint32_t i = lane; i < C; i += 32) first(qp_load_one(row + i));
            }
        } else {
            for (uint32_t i = lane; i < C; i += 32) first(qp_load_one(row + i));
        }
        for (int o = 16; o > 0; o >>= 1) {                   // fixed order: bit-reproducible
            s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
            sa += __shfl_xor_sync(0xFFFFFFFFu, sa, o);
            mn = fminf(mn, __shfl_xor_sync(0xFFFFFFFFu, mn, o));
            mx = fmaxf(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, o));
            bad += __shfl_xor_sync(0xFFFFFFFFu, bad, o);
        }
        const unsigned nf = C - bad;
        const double mean = nf ? s / (double)nf : 0.0;
        const float m_hi = (float)mean, m_lo = (float)(mean - (double)m_hi);   // the mean as an unevaluated fp32 pair
        double sd = 0.0, sv = 0.0;
        auto second = [&](float v, float& d1, float& d2) {
            if (qp_is_finite(v)) {
                const float d = __fsub_rn(__fsub_rn(v, m_hi), m_lo);
                d1 += fabsf(d);
                d2 = fmaf(d, d, d2);
            }
        };
        if (VEC) {
            for (uint32_t v0 = lane; v0 < C / EPV; v0 += 32) {
                float e[EPV];
                qp_load_vec(row + (size_t)v0 * EPV, e);
                float d1 = 0.f, d2 = 0.f;
#pragma unroll
                for (int i = 0; i < EPV; ++i) second(e[i], d1, d2);
                sd += (double)d1;
                sv += (double)d2;
            }
        } else {
            for (uint32_t i = lane; i < C; i += 32) {
                float d1 = 0.f, d2 = 0.f;
                second(qp_load_one(row + i), d1, d2);
                sd += (double)d1;
                sv += (double)d2;
            }
        }
        for (int o = 16; o > 0; o >>= 1) {
            sd += __shfl_xor_sync(0xFFFFFFFFu, sd, o);
            sv += __shfl_xor_sync(0xFFFFFFFFu, sv, o);
        }
        if (lane == 0) {
            qp_stats_t st;
            st.n = C;
            st.nonfinite = bad;
            st.mean = mean;
            st.mean_abs = nf ? sa / (double)nf : 0.0;
            st.mad = nf ? sd / (double)nf : 0.0;
            st.var = nf ? sv / (double)nf : 0.0;
            st.min = nf ? (double)mn : 0.0;
            st.max = nf ? (double)mx : 0.0;
            st.hist_peak = 0;
            st.hist_bins = 0;
            st.reserved = 0;
            out[t] = st;
        }
        any_bad |= bad != 0;
    }
    if (any_bad && lane == 0) atomicOr(status, QP_DEV_NONFINITE);
}

__global__ void __launch_bounds__(128) tok_clip_kernel(const qp_stats_t* __restrict__ st, uint64_t tokens, int bits, int method,
                                                       int dist, int bmode, double F, qp_qparams_t* __restrict__ qp_out,
                                                       unsigned* __restrict__ status)
{
    const uint64_t t = (uint64_t)blockIdx.x * 128 + threadIdx.x;
    if (t >= tokens) return;
    double lo, hi;
    qp_clip_ends(st[t], method, dist, bmode, bits, F, lo, hi);
    qp_qparams_t q;
    const int rc = qp_fill_qparams(lo, hi, bits, &q);
    qp_out[t] = q;
    if (rc == QP_WARN_DEGENERATE) atomicOr(status, QP_DEV_DEGENERATE);
}

// ---------------------------------------------------------------------------- quantize + pack

// token and position inside it of element `el`; then moved on by `step` elements at a time
struct TokCursor {
    uint64_t tok;
    uint32_t rem, C;
    __device__ __forceinline__ TokCursor(uint64_t el, uint32_t channels) : tok(el / channels), rem((uint32_t)(el % channels)), C(channels) {}
    __device__ __forceinline__ void advance(uint32_t step)
    {
        rem += step;
        while (rem >= C) { rem -= C; ++tok; }
    }
};

// Fast path: x 16-byte aligned, channels a multiple of the vector's elements (a vector lies in one token).
template <int BITS, typename T>
__global__ void __launch_bounds__(QP_THREADS) tok_pack_kernel(const T* __restrict__ x, uint64_t ntiles, uint32_t C,
                                                              const qp_qparams_t* __restrict__ d_qp,
                                                              uint32_t* __restrict__ out, unsigned* __restrict__ status)
{
    constexpr int EPV = qp_span<T>::EPV;
    constexpr int NLOAD = TILE / (32 * EPV);
    __shared__ __align__(16) uint32_t stage[WARPS][256];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t* sw = stage[warp];
    const uint64_t wstride = (uint64_t)gridDim.x * WARPS;
    bool mismatch = false;
    for (uint64_t tile = (uint64_t)blockIdx.x * WARPS + warp; tile < ntiles; tile += wstride) {
        const T* xt = x + tile * TILE;
        float e[NLOAD][EPV];
#pragma unroll
        for (int j = 0; j < NLOAD; ++j) qp_load_vec(xt + (j * 32 + lane) * EPV, e[j]);
        TokCursor cur(tile * TILE + (uint64_t)lane * EPV, C);
#pragma unroll
        for (int j = 0; j < NLOAD; ++j) {
            const qp_qparams_t* q = d_qp + cur.tok;
            const float lo = __ldg(&q->lo), hi = __ldg(&q->hi), inv = __ldg(&q->inv_scale);
            mismatch |= __ldg(&q->bits) != BITS;
            unsigned quads[EPV / 4];
#pragma unroll
            for (int h = 0; h < EPV / 4; ++h) {
                quads[h] = qp_quad<BITS>(e[j] + 4 * h, lo, hi, inv);
            }
            if constexpr (EPV == 4) sw[qp_swz(j * 32 + lane)] = quads[0];
            else *reinterpret_cast<uint2*>(&sw[qp_swz(2 * (j * 32 + lane))]) = make_uint2(quads[0], quads[1]);
            cur.advance(32 * EPV);
        }
        __syncwarp();
        uint32_t w[BITS];
        qp_quads_to_words<BITS>(sw, lane, w);
        uint32_t* ot = out + tile * (32 * BITS);
        __syncwarp();
#pragma unroll
        for (int m = 0; m < BITS; ++m) sw[lane * BITS + m] = w[m];
        __syncwarp();
#pragma unroll
        for (int m = 0; m < BITS; ++m) ot[m * 32 + lane] = sw[m * 32 + lane];
        __syncwarp();
    }
    if (mismatch) atomicOr(status, QP_DEV_BITS_MISMATCH);
}

// Any shape: thread t packs elements [first + 32t, first + 32t + 32) that exist into `bits` words (16 bits:
// 16 words) and writes those below nwords.
template <typename T>
__global__ void __launch_bounds__(QP_THREADS) tok_pack_scalar(const T* __restrict__ x, uint64_t first, uint64_t n, uint32_t C,
                                                              int bits, const qp_qparams_t* __restrict__ d_qp,
                                                              uint32_t* __restrict__ out, uint64_t nwords,
                                                              unsigned* __restrict__ status)
{
    const uint64_t t = (uint64_t)blockIdx.x * QP_THREADS + threadIdx.x;
    const uint64_t w0 = t * (uint64_t)bits;
    if (w0 >= nwords) return;
    const unsigned mask = (1u << bits) - 1u;
    uint32_t w[16];
#pragma unroll
    for (int m = 0; m < 16; ++m) w[m] = 0u;
    const uint64_t e0 = first + t * 32;
    bool mismatch = false;
    if (e0 < n) {
        TokCursor cur(e0, C);
        for (int i = 0; i < 32 && e0 + i < n; ++i) {
            const qp_qparams_t* q = d_qp + cur.tok;
            mismatch |= __ldg(&q->bits) != bits;
            const unsigned c = qp_code(qp_load_one(x + e0 + i), __ldg(&q->lo), __ldg(&q->hi), __ldg(&q->inv_scale), mask);
            const int bit = i * bits, word = bit >> 5, sh = bit & 31;
            w[word] |= c << sh;
            if (sh + bits > 32) w[word + 1] |= c >> (32 - sh);
            cur.advance(1);
        }
    }
    for (int m = 0; m < bits; ++m)
        if (w0 + m < nwords) out[w0 + m] = w[m];
    if (mismatch) atomicOr(status, QP_DEV_BITS_MISMATCH);
}

// ---------------------------------------------------------------------------- unpack + dequantize

__device__ __forceinline__ float tok_code_to_float(unsigned c) { return __fsub_rn(__uint_as_float(0x4B000000u | c), 8388608.0f); }

__device__ __forceinline__ void tok_store4(float* y, uint64_t el, const float (&v)[4])
{
    __stcs(reinterpret_cast<float4*>(y + el), make_float4(v[0], v[1], v[2], v[3]));
}
__device__ __forceinline__ void tok_store4(unsigned short* y, uint64_t el, const float (&v)[4])
{
    uint2 o;
    o.x = (unsigned)qp_f32_to_bf16(v[0]) | ((unsigned)qp_f32_to_bf16(v[1]) << 16);
    o.y = (unsigned)qp_f32_to_bf16(v[2]) | ((unsigned)qp_f32_to_bf16(v[3]) << 16);
    __stcs(reinterpret_cast<uint2*>(y + el), o);
}
__device__ __forceinline__ void tok_store1(float* y, uint64_t el, float v) { y[el] = v; }
__device__ __forceinline__ void tok_store1(unsigned short* y, uint64_t el, float v) { y[el] = qp_f32_to_bf16(v); }

// Fast path: y aligned for 4-element stores, channels a multiple of 4.
template <int BITS, typename TO>
__global__ void __launch_bounds__(QP_THREADS) tok_unpack_kernel(const uint32_t* __restrict__ in, uint64_t ntiles, uint32_t C,
                                                                const qp_qparams_t* __restrict__ d_qp, TO* __restrict__ y,
                                                                unsigned* __restrict__ status)
{
    __shared__ __align__(16) uint32_t stage[WARPS][256];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t* sw = stage[warp];
    const uint64_t wstride = (uint64_t)gridDim.x * WARPS;
    constexpr unsigned MASK = (1u << BITS) - 1u;
    constexpr int QB = 4 * BITS;
    constexpr unsigned QMASK = QB >= 32 ? 0xFFFFFFFFu : ((1u << (QB & 31)) - 1u);
    bool mismatch = false;
    for (uint64_t tile = (uint64_t)blockIdx.x * WARPS + warp; tile < ntiles; tile += wstride) {
        const uint32_t* it = in + tile * (32 * BITS);
        uint32_t w[BITS];
#pragma unroll
        for (int m = 0; m < BITS; ++m) sw[m * 32 + lane] = __ldg(it + m * 32 + lane);
        __syncwarp();
#pragma unroll
        for (int m = 0; m < BITS; ++m) w[m] = sw[lane * BITS + m];
        __syncwarp();
        uint32_t qd[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int bit = QB * k, word = bit >> 5, sh = bit & 31;
            uint32_t v = w[word] >> sh;
            if (sh + QB > 32) v |= w[(word + 1) % BITS] << (32 - sh);
            qd[k] = v & QMASK;
        }
        *reinterpret_cast<uint4*>(&sw[qp_swz(8 * lane)]) = make_uint4(qd[0], qd[1], qd[2], qd[3]);
        *reinterpret_cast<uint4*>(&sw[qp_swz(8 * lane + 4)]) = make_uint4(qd[4], qd[5], qd[6], qd[7]);
        __syncwarp();
        uint32_t mine[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) mine[j] = sw[qp_swz(j * 32 + lane)];
        TokCursor cur(tile * TILE + (uint64_t)lane * 4, C);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const qp_qparams_t* q = d_qp + cur.tok;
            const float lo = __ldg(&q->lo), scale = __ldg(&q->scale);
            mismatch |= __ldg(&q->bits) != BITS;
            float v[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) v[i] = fmaf(tok_code_to_float((mine[j] >> (BITS * i)) & MASK), scale, lo);
            tok_store4(y, tile * TILE + (uint64_t)(j * 32 + lane) * 4, v);
            cur.advance(128);
        }
        __syncwarp();
    }
    if (mismatch) atomicOr(status, QP_DEV_BITS_MISMATCH);
}

template <typename TO>
__global__ void __launch_bounds__(QP_THREADS) tok_unpack_scalar(const uint32_t* __restrict__ in, uint64_t first, uint64_t n,
                                                                uint32_t C, int bits, const qp_qparams_t* __restrict__ d_qp,
                                                                TO* __restrict__ y, unsigned* __restrict__ status)
{
    const uint64_t t = (uint64_t)blockIdx.x * QP_THREADS + threadIdx.x;
    const uint64_t e0 = first + t * 32;
    if (e0 >= n) return;
    const uint32_t* wp = in + t * (uint64_t)bits;          // `in` already points at the word of element `first`
    const unsigned mask = (1u << bits) - 1u;
    const int cnt = (int)((n - e0) < 32 ? (n - e0) : 32);
    const int nw = (cnt * bits + 31) >> 5;
    uint32_t w[17];
#pragma unroll
    for (int m = 0; m < 17; ++m) w[m] = 0u;
    for (int m = 0; m < nw; ++m) w[m] = __ldg(wp + m);
    TokCursor cur(e0, C);
    bool mismatch = false;
    for (int i = 0; i < cnt; ++i) {
        const qp_qparams_t* q = d_qp + cur.tok;
        mismatch |= __ldg(&q->bits) != bits;
        const int bit = i * bits, word = bit >> 5, sh = bit & 31;
        uint32_t c = w[word] >> sh;
        if (sh + bits > 32) c |= w[word + 1] << (32 - sh);
        tok_store1(y, e0 + i, fmaf(tok_code_to_float(c & mask), __ldg(&q->scale), __ldg(&q->lo)));
        cur.advance(1);
    }
    if (mismatch) atomicOr(status, QP_DEV_BITS_MISMATCH);
}

// ---------------------------------------------------------------------------- rows in shared memory
//
// A warp takes a token, copies its row into its own piece of shared memory (asynchronous 16-byte copies)
// and does everything to it from there: statistics and, in the sender, clip, quantize and pack as well.
// The row is read from HBM once and the packed words written once: the sender is bound by those bytes (161 MB
// for the ViT-Huge tensor at 8 bits, 24.7 us at the copy peak), where the three kernels read the tensor twice
// and took 76 us (statistics 49, clip 2.5, pack 24.5).  The row is not kept in registers: with 128 of
// them only 16 warps fit an SM and the chains of one token do not overlap enough with the others'
// (53 us).  What a token costs beside its elements is kept small by giving the lanes different work: the two
// sums of a pass reduce together (half a warp each), and the quotients of the statistics and of the
// quantizer are one division with another numerator in every lane.

// s0 and s1 summed over the warp, both results in every lane; fixed order
__device__ __forceinline__ void tok_reduce2(double& s0, double& s1, int lane)
{
    const bool upper = (lane & 16) != 0;
    double v = upper ? s1 : s0;
    v += __shfl_xor_sync(0xFFFFFFFFu, upper ? s0 : s1, 16);
    for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    s0 = __shfl_sync(0xFFFFFFFFu, v, 0);
    s1 = __shfl_sync(0xFFFFFFFFu, v, 16);
}

// 8 consecutive-vector elements of the row as four pairs: vectors v and v + 32 of fp32, vector v of bf16
template <typename T>
__device__ __forceinline__ void tok_lds8(const T* row, int v, qp_f2 (&p)[4])
{
    if constexpr (sizeof(T) == 4) {
        const ulonglong2 a = *reinterpret_cast<const ulonglong2*>(row + v * 4);
        const ulonglong2 b = *reinterpret_cast<const ulonglong2*>(row + (v + 32) * 4);
        p[0] = a.x; p[1] = a.y; p[2] = b.x; p[3] = b.y;
    } else {
        const uint4 r = *reinterpret_cast<const uint4*>(row + v * 8);
        const unsigned w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) p[i] = qp_pack2(__uint_as_float(w[i] << 16), __uint_as_float(w[i] & 0xFFFF0000u));
    }
}

// a 16-byte vector of the row as floats
template <typename T>
__device__ __forceinline__ void tok_widen(const uint4& r, float (&e)[qp_span<T>::EPV])
{
    const unsigned w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        if constexpr (sizeof(T) == 4) {
            e[i] = __uint_as_float(w[i]);
        } else {
            e[2 * i] = __uint_as_float(w[i] << 16);
            e[2 * i + 1] = __uint_as_float(w[i] & 0xFFFF0000u);
        }
    }
}
template <typename T>
__device__ __forceinline__ void tok_lds(const T* p, float (&e)[qp_span<T>::EPV])
{
    tok_widen<T>(*reinterpret_cast<const uint4*>(p), e);
}

// sum of 8 magnitudes as a tree, and of 8 values: no longer chain of roundings than a run of four
__device__ __forceinline__ float tok_abs8(const qp_f2 (&p)[4])
{
    float a[4], b[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) qp_unpack2(p[i], a[i], b[i]);
    return ((fabsf(a[0]) + fabsf(a[1])) + (fabsf(a[2]) + fabsf(a[3]))) + ((fabsf(b[0]) + fabsf(b[1])) + (fabsf(b[2]) + fabsf(b[3])));
}
__device__ __forceinline__ float tok_sum8(const qp_f2 (&p)[4])
{
    float a, b;
    qp_unpack2(qp_add2(qp_add2(p[0], p[1]), qp_add2(p[2], p[3])), a, b);
    return a + b;
}

// statistics of the row in shared memory (nvec whole vectors), the same in every lane; true if it holds
// non-finite values.  The loops over whole groups of 32 lanes x 8 elements are uniform; what is left of the
// row (less than one such group) is padded: with copies of nothing (zero) for the sums, and skipped in the
// deviations by an infinite value.
template <typename T>
__device__ __forceinline__ bool tok_row_stats(const T* row, int nvec, uint32_t C, int lane, qp_stats_t& st)
{
    constexpr int EPV = qp_span<T>::EPV;
    constexpr int STEP = 8 / EPV * 32;                        // vectors of one round: 64 (fp32), 32 (bf16)
    const float inf = __int_as_float(0x7F800000);
    // first moments: fp32 over 8 elements, then fp64
    double s = 0.0, sa = 0.0;
    float mn = inf, mx = -inf;
    unsigned bad = 0u;
    bool odd = false;                                         // a NaN or Inf (or an fp32 overflow) in this lane
    auto tail8 = [&](int v0, float missing, qp_f2 (&p)[4]) {  // the last, partial round
        float e[8];
#pragma unroll
        for (int h = 0; h < 8 / EPV; ++h) {
            const int v = v0 + h * 32 + lane;
            float a[EPV];
            if (v < nvec) tok_lds<T>(row + QP_CK(v, nvec) * EPV, a);
#pragma unroll
            for (int i = 0; i < EPV; ++i) e[h * EPV + i] = v < nvec ? a[i] : missing;
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) p[i] = qp_pack2(e[2 * i], e[2 * i + 1]);
    };
    auto moments = [&](const qp_f2 (&p)[4]) {
        const float psa = tok_abs8(p);
        s += (double)tok_sum8(p);
        sa += (double)psa;
        odd |= !(psa < inf);
    };
    const int whole = nvec / STEP * STEP;
#pragma unroll 2
    for (int v0 = 0; v0 < whole; v0 += STEP) {
        qp_f2 p[4];
        tok_lds8<T>(row, QP_CK(v0 + lane, nvec - (STEP - 32)), p);
        moments(p);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            float a, b;
            qp_unpack2(p[i], a, b);
            mn = qp_min3(mn, a, b);
            mx = qp_max3(mx, a, b);
        }
    }
    if (whole < nvec) {
        qp_f2 p[4];
        tail8(whole, 0.f, p);
        moments(p);
#pragma unroll
        for (int h = 0; h < 8 / EPV; ++h)
            if (whole + h * 32 + lane < nvec) {
                float a[EPV];
                tok_lds<T>(row + (whole + h * 32 + lane) * EPV, a);
#pragma unroll
                for (int i = 0; i < EPV; i += 2) { mn = qp_min3(mn, a[i], a[i + 1]); mx = qp_max3(mx, a[i], a[i + 1]); }
            }
    }
    const bool guard = __any_sync(0xFFFFFFFFu, odd);
    if (guard) {                                              // rare: the row again, element by element
        s = 0.0; sa = 0.0; mn = inf; mx = -inf;
        for (int v = lane; v < nvec; v += 32) {
            float e[EPV];
            tok_lds<T>(row + v * EPV, e);
#pragma unroll
            for (int i = 0; i < EPV; ++i) {
                if (qp_is_finite(e[i])) {
                    s += (double)e[i];
                    sa += (double)fabsf(e[i]);
                    mn = fminf(mn, e[i]);
                    mx = fmaxf(mx, e[i]);
                } else {
                    ++bad;
                }
            }
        }
        bad = __reduce_add_sync(0xFFFFFFFFu, bad);
    }
    tok_reduce2(s, sa, lane);
    {
        const bool upper = (lane & 16) != 0;                  // min of x in one half, min of -x in the other
        float v = upper ? -mx : mn;
        v = fminf(v, __shfl_xor_sync(0xFFFFFFFFu, upper ? mn : -mx, 16));
        for (int o = 8; o > 0; o >>= 1) v = fminf(v, __shfl_xor_sync(0xFFFFFFFFu, v, o));
        mn = __shfl_sync(0xFFFFFFFFu, v, 0);
        mx = -__shfl_sync(0xFFFFFFFFu, v, 16);
    }
    const unsigned nf = C - bad;
    const double mean = nf ? s / (double)nf : 0.0;
    const float m_hi = (float)mean, m_lo = (float)(mean - (double)m_hi);   // the mean as an unevaluated fp32 pair

    // deviations
    double sd = 0.0, sv = 0.0;
    const qp_f2 nhi = qp_pack2(-m_hi, -m_hi), nlo = qp_pack2(-m_lo, -m_lo);
    auto deviations = [&](const qp_f2 (&p)[4], bool check) {
        qp_f2 d[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) d[i] = qp_add2(qp_add2(p[i], nhi), nlo);
        if (check) {                                          // uniform: non-finite values, or elements that do not exist
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                float a, b, da, db;
                qp_unpack2(p[i], a, b);
                qp_unpack2(d[i], da, db);
                d[i] = qp_pack2(qp_is_finite(a) ? da : 0.f, qp_is_finite(b) ? db : 0.f);
            }
        }
        sd += (double)tok_abs8(d);
        qp_f2 q2 = qp_fma2(d[0], d[0], 0ull);
#pragma unroll
        for (int i = 1; i < 4; ++i) q2 = qp_fma2(d[i], d[i], q2);
        float qa, qb;
        qp_unpack2(q2, qa, qb);
        sv += (double)(qa + qb);
    };
#pragma unroll 2
    for (int v0 = 0; v0 < whole; v0 += STEP) {
        qp_f2 p[4];
        tok_lds8<T>(row, QP_CK(v0 + lane, nvec - (STEP - 32)), p);
        deviations(p, guard);
    }
    if (whole < nvec) {
        qp_f2 p[4];
        tail8(whole, inf, p);
        deviations(p, true);
    }
    tok_reduce2(sd, sv, lane);

    const double q = (lane == 0 ? sa : lane == 1 ? sd : sv) / (double)(nf ? nf : 1u);   // the three means in three lanes
    st.n = C;
    st.nonfinite = bad;
    st.mean = mean;
    st.mean_abs = nf ? __shfl_sync(0xFFFFFFFFu, q, 0) : 0.0;
    st.mad = nf ? __shfl_sync(0xFFFFFFFFu, q, 1) : 0.0;
    st.var = nf ? __shfl_sync(0xFFFFFFFFu, q, 2) : 0.0;
    st.min = nf ? (double)mn : 0.0;
    st.max = nf ? (double)mx : 0.0;
    st.hist_peak = 0;
    st.hist_bins = 0;
    st.reserved = 0;
    return bad != 0u;
}

constexpr int TR_WARPS = 8;                                   // warps per block
// Blocks per SM, 48 registers a thread: a row is a chain of waits, and 72 % of the issue slots were taken with four.  fp32 of 25216 x 1280
// at 4 and 8 bits 41.3 -> 39.0 and 37.2 -> 36.3 us, 16000 x 2048 at 8 bits 41.1 -> 35.3, 40000 x 192 bf16 at 4 bits 28.4 -> 26.7; six
// (40 registers) are slower again (39.2, 37.1, 37.0).
constexpr int TR_BLOCKS = 5;
// Statistics of rows so long that shared memory has no room for five blocks keep 64 registers: 12608 rows of 2048, 2560 and 3072 fp32
// channels 22.4, 31.3 and 34.1 us with 48, 21.5, 30.1 and 33.5 with 64 (no bound: 21.3, 29.5 and 33.3, but 18.0 at 1600 against
// 16.9).  The sender's gain or lose 1 to 3 % by width and type, on both sides of nothing.
constexpr int TR_LONG_BLOCKS = 4;
constexpr size_t TR_SM_BYTES = 228 * 1024;                    // shared memory of an SM, of which a block takes 1 KB more than it asks for
// Rounds of 32 vectors that the staged widths load before they store.  One, two and four of them, 12608 rows of 1280 fp32 at 5 bits:
// 21.9, 20.6 and 20.8 us, 2560 bf16 at 6: 32.9, 31.8 and 31.5, 2560 fp32 at 4: 43.1, 41.1 and 41.1 (quads in a room of their own, four
// blocks an SM: 22.2, 32.9 and 41.1).
constexpr int TR_ROUNDS = 4;

// bytes of shared memory a warp needs for a row (a multiple of 16).  The sender's quads, a byte per element, take the
// place of the elements that they were made of, its words that of the elements behind.
__host__ __device__ constexpr size_t tok_row_bytes(uint32_t C, size_t esz) { return (size_t)C * esz; }

// BITS = 0: statistics only (any row of whole vectors).  BITS = 1..8: the whole sender, rows of whole
// 32-element groups (a row is then whole words).
template <int BITS, typename T, int BLOCKS>
__global__ void __launch_bounds__(TR_WARPS * 32, BLOCKS) tok_rows_kernel(const T* __restrict__ x, uint64_t tokens, uint32_t C, int method,
                                                                 int bmode, double F, uint32_t* __restrict__ out,
                                                                 uint64_t nwords, qp_qparams_t* __restrict__ qp_out,
                                                                 qp_stats_t* __restrict__ st_out, unsigned* __restrict__ status)
{
    extern __shared__ __align__(16) unsigned char raw[];
    constexpr int EPV = qp_span<T>::EPV;
    const int lane = threadIdx.x & 31;
    T* row = reinterpret_cast<T*>(raw + (threadIdx.x >> 5) * tok_row_bytes(C, sizeof(T)));
    const int nvec = (int)(C / EPV);
    unsigned raise = 0u;
    const uint64_t wstride = (uint64_t)gridDim.x * TR_WARPS;
    for (uint64_t t = (uint64_t)blockIdx.x * TR_WARPS + (threadIdx.x >> 5); t < tokens; t += wstride) {
        const T* src = x + t * C;
        auto fetch = [&](int v) {
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(row + QP_CK(v, nvec) * EPV)),
                         "l"(src + (size_t)v * EPV)
                         : "memory");
        };
#pragma unroll 4
        for (int v0 = 0; v0 < (nvec & ~31); v0 += 32) fetch(v0 + lane);
        if ((nvec & ~31) + lane < nvec) fetch((nvec & ~31) + lane);
        asm volatile("cp.async.commit_group;" ::: "memory");
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncwarp();

        qp_stats_t st;
        if (tok_row_stats<T>(row, nvec, C, lane, st)) raise |= QP_DEV_NONFINITE;
        if (lane == 0) st_out[t] = st;
        if constexpr (BITS > 0) {
            constexpr unsigned mask = (1u << BITS) - 1u;
            uint32_t* sw = reinterpret_cast<uint32_t*>(row);
            const int groups = (int)(C / 32);
            double lo_d, hi_d;
            qp_clip_ends(st, method, QP_DIST_LAPLACE, bmode, BITS, F, lo_d, hi_d);
            qp_qparams_t q;
            q.lo = (float)lo_d;
            q.hi = (float)hi_d;
            q.bits = BITS;
            q.flags = (!(q.hi > q.lo) || !(q.lo - q.lo == 0.f) || !(q.hi - q.hi == 0.f)) ? 1 : 0;
            q.scale = q.inv_scale = 0.f;
            if (q.flags) {
                raise |= QP_DEV_DEGENERATE;
            } else {                                         // scale and its reciprocal in two lanes
                const double range = (double)q.hi - (double)q.lo, levels_m1 = (double)mask;
                const double num = lane == 0 ? range : levels_m1, den = lane == 0 ? levels_m1 : range;
                const float v = (float)(num / den);
                q.scale = __shfl_sync(0xFFFFFFFFu, v, 0);
                q.inv_scale = __shfl_sync(0xFFFFFFFFu, v, 1);
            }
            if (lane == 0) qp_out[t] = q;
            uint32_t* orow = out + t * (uint64_t)(groups * BITS);
            constexpr bool STAGED = BITS != 8 && !(BITS == 4 && EPV == 8);
            auto load = [&](int v) { return *reinterpret_cast<const uint4*>(row + QP_CK(v, nvec) * EPV); };
            auto quantize = [&](int v, const uint4& r) {     // vector v: its quads to the output (8 bits: a quad is a word) or to `sw`
                float e[EPV];
                tok_widen<T>(r, e);
                if constexpr (EPV == 4) {
                    const unsigned qd = qp_quad<BITS>(e, q.lo, q.hi, q.inv_scale);
                    if constexpr (BITS == 8) orow[v] = qd;
                    else sw[QP_CK(qp_swz(v), (int)(C / 4))] = qd;
                } else {
                    const uint2 qd = make_uint2(qp_quad<BITS>(e, q.lo, q.hi, q.inv_scale),
                                                qp_quad<BITS>(e + 4, q.lo, q.hi, q.inv_scale));
                    if constexpr (BITS == 8) reinterpret_cast<uint2*>(orow)[v] = qd;
                    else if constexpr (BITS == 4) orow[v] = qd.x | (qd.y << 16);
                    else *reinterpret_cast<uint2*>(&sw[QP_CK(qp_swz(2 * v), (int)(C / 4) - 1)]) = qd;
                }
            };
            const int whole = nvec & ~31;
            if constexpr (STAGED) {
                // A round of 32 vectors leaves its quads where vectors of that round and of earlier ones were, which other lanes have
                // read: all lanes load, then all store.
                int v0 = 0;
                for (; v0 + 32 * TR_ROUNDS <= whole; v0 += 32 * TR_ROUNDS) {
                    uint4 r[TR_ROUNDS];
#pragma unroll
                    for (int u = 0; u < TR_ROUNDS; ++u) r[u] = load(v0 + 32 * u + lane);
                    __syncwarp();
#pragma unroll
                    for (int u = 0; u < TR_ROUNDS; ++u) quantize(v0 + 32 * u + lane, r[u]);
                }
                for (; v0 < nvec; v0 += 32) {
                    const bool mine = v0 + lane < nvec;
                    uint4 r = make_uint4(0u, 0u, 0u, 0u);
                    if (mine) r = load(v0 + lane);
                    __syncwarp();
                    if (mine) quantize(v0 + lane, r);
                }
            } else {
#pragma unroll 4
                for (int v0 = 0; v0 < whole; v0 += 32) quantize(v0 + lane, load(v0 + lane));
                if (whole + lane < nvec) quantize(whole + lane, load(whole + lane));
            }
            if constexpr (STAGED) {
                // quads across the warp: 32 elements = BITS words per lane
                __syncwarp();
                uint32_t* words = sw + C / 4;                 // behind the quads
                for (int g = lane; g < groups; g += 32) {
                    uint32_t w[BITS];
                    qp_quads_to_words<BITS>(sw, QP_CK(g, groups), w);
                    if constexpr (BITS == 4) {               // 4, 2, 1: a lane's words are one aligned vector
                        *reinterpret_cast<uint4*>(orow + g * 4) = make_uint4(w[0], w[1], w[2], w[3]);
                    } else if constexpr (BITS == 2) {
                        *reinterpret_cast<uint2*>(orow + g * 2) = make_uint2(w[0], w[1]);
                    } else if constexpr (BITS == 1) {
                        orow[g] = w[0];
                    } else {
#pragma unroll
                        for (int m = 0; m < BITS; ++m) words[QP_CK(g * BITS + m, (int)(C / 4))] = w[m];
                    }
                }
                if constexpr (BITS != 4 && BITS != 2 && BITS != 1) {
                    __syncwarp();
                    for (int i = lane; i < groups * BITS; i += 32) orow[i] = words[QP_CK(i, (int)(C / 4))];
                }
            }
            if (t == tokens - 1) {                           // pad words
                const uint64_t end = tokens * (uint64_t)(groups * BITS);
                if (lane < (int)(nwords - end)) out[end + lane] = 0u;
            }
        }
        __syncwarp();                                        // the row may be overwritten
    }
    if (raise && lane == 0) atomicOr(status, raise);
}

// ---------------------------------------------------------------------------- host side

int32_t tok_check(qp_ctx* ctx, uint64_t tokens, uint32_t channels)
{
    if (channels < 1) return qp_fail(ctx, QP_ERR_INVALID_ARG, "channels must be at least 1");
    if (tokens >= (1ull << 40) / channels) return qp_fail(ctx, QP_ERR_INVALID_ARG, "tensor too large");
    return QP_OK;
}

unsigned tok_grid(qp_ctx* ctx, uint64_t warps_wanted)
{
    const uint64_t want = (warps_wanted + WARPS - 1) / WARPS;
    const uint64_t cap = (uint64_t)ctx->sm_count * 64;
    return (unsigned)(want < 1 ? 1 : (want < cap ? want : cap));
}

template <typename T>
int32_t pack_tokens_typed(qp_ctx* ctx, const T* x, uint64_t n, uint32_t C, int bits, const qp_qparams_t* d_qp, void* d_packed,
                          cudaStream_t s)
{
    constexpr int EPV = qp_span<T>::EPV;
    uint32_t* out = static_cast<uint32_t*>(d_packed);
    const bool fast = bits <= 8 && C % EPV == 0 && ((uintptr_t)x & 15u) == 0;
    const uint64_t ntiles = fast ? n / TILE : 0;
    if (ntiles) {
        const unsigned blocks = tok_grid(ctx, ntiles);
        ctx->launches += 1;
#define QP_TOK_PACK(B) case B: tok_pack_kernel<B, T><<<blocks, QP_THREADS, 0, s>>>(x, ntiles, C, d_qp, out, ctx->d_status); break;
        switch (bits) {
            QP_TOK_PACK(1) QP_TOK_PACK(2) QP_TOK_PACK(3) QP_TOK_PACK(4) QP_TOK_PACK(5) QP_TOK_PACK(6) QP_TOK_PACK(7) QP_TOK_PACK(8)
        }
#undef QP_TOK_PACK
    }
    const uint64_t done_words = ntiles * 32 * (uint64_t)bits;
    const uint64_t total_words = qp_packed_bytes(n, bits) / 4;
    if (total_words > done_words) {
        const uint64_t nwords = total_words - done_words;
        const uint64_t threads = (nwords + bits - 1) / bits;
        const uint64_t blocks = (threads + QP_THREADS - 1) / QP_THREADS;
        ctx->launches += 1;
        tok_pack_scalar<T><<<(unsigned)blocks, QP_THREADS, 0, s>>>(x, ntiles * TILE, n, C, bits, d_qp, out + done_words, nwords,
                                                                    ctx->d_status);
    }
    return qp_check_launch(ctx, "qp_quantize_pack_tokens");
}

template <typename TO>
int32_t unpack_tokens_typed(qp_ctx* ctx, const void* d_packed, uint64_t n, uint32_t C, int bits, const qp_qparams_t* d_qp, TO* y,
                            cudaStream_t s)
{
    const uint32_t* in = static_cast<const uint32_t*>(d_packed);
    const bool fast = bits <= 8 && C % 4 == 0 && ((uintptr_t)y & (4 * sizeof(TO) - 1)) == 0;
    const uint64_t ntiles = fast ? n / TILE : 0;
    if (ntiles) {
        const unsigned blocks = tok_grid(ctx, ntiles);
        ctx->launches += 1;
#define QP_TOK_UNPACK(B) case B: tok_unpack_kernel<B, TO><<<blocks, QP_THREADS, 0, s>>>(in, ntiles, C, d_qp, y, ctx->d_status); break;
        switch (bits) {
            QP_TOK_UNPACK(1) QP_TOK_UNPACK(2) QP_TOK_UNPACK(3) QP_TOK_UNPACK(4) QP_TOK_UNPACK(5) QP_TOK_UNPACK(6) QP_TOK_UNPACK(7)
            QP_TOK_UNPACK(8)
        }
#undef QP_TOK_UNPACK
    }
    const uint64_t first = ntiles * TILE;
    if (n > first) {
        const uint64_t threads = (n - first + 31) / 32;
        const uint64_t blocks = (threads + QP_THREADS - 1) / QP_THREADS;
        ctx->launches += 1;
        tok_unpack_scalar<TO><<<(unsigned)blocks, QP_THREADS, 0, s>>>(in + ntiles * 32 * (uint64_t)bits, first, n, C, bits, d_qp, y,
                                                                      ctx->d_status);
    }
    return qp_check_launch(ctx, "qp_unpack_dequantize_tokens");
}

// Rows go through shared memory where a row fits: TR_WARPS of them in the 48 KB every block may have would
// stop at 1536 fp32 channels; blocks ask for more, up to what leaves two blocks (16 warps) per SM.  The sender's rows stop
// a byte per element earlier, at 2848 fp32 and 4768 bf16 channels: quads had room of their own when that line was measured.
constexpr size_t TR_SMEM_MAX = 112 * 1024;
bool tok_rows_apply(const void* x, int dtype, uint32_t C, bool sender)
{
    if (!x || (dtype != QP_F32 && dtype != QP_BF16)) return false;
    const size_t esz = dtype == QP_F32 ? 4 : 2;
    return C >= 32 && C % (sender ? 32 : 16 / esz) == 0 && ((uintptr_t)x & 15u) == 0 &&
           (tok_row_bytes(C, esz) + (sender ? C : 0)) * TR_WARPS <= TR_SMEM_MAX;
}

template <int BITS, typename T>
int32_t launch_rows(qp_ctx* ctx, const T* x, uint64_t tokens, uint32_t C, int method, int bmode, uint32_t* out,
                    qp_qparams_t* d_qp, qp_stats_t* d_stats, cudaStream_t s)
{
    const size_t smem = tok_row_bytes(C, sizeof(T)) * TR_WARPS;
    const bool five = TR_BLOCKS * (smem + 1024) <= TR_SM_BYTES;
    const auto kernel = five ? tok_rows_kernel<BITS, T, TR_BLOCKS> : tok_rows_kernel<BITS, T, BITS == 0 ? TR_LONG_BLOCKS : TR_BLOCKS>;
    if (smem > 48 * 1024 && cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TR_SMEM_MAX) != cudaSuccess)
        return qp_check_launch(ctx, "token rows (shared memory)");
    const uint64_t want = (tokens + TR_WARPS - 1) / TR_WARPS, cap = (uint64_t)ctx->sm_count * 64;
    kernel<<<(unsigned)(want < cap ? want : cap), TR_WARPS * 32, smem, s>>>(
        x, tokens, C, method, bmode, BITS > 0 ? qp_host_aciq_F(BITS, QP_DIST_LAPLACE) : 0.0, out,
        BITS > 0 ? qp_packed_bytes(tokens * C, BITS) / 4 : 0, d_qp, d_stats, ctx->d_status);
    ctx->launches += 1;
    return qp_check_launch(ctx, "token rows");
}

template <typename T>
int32_t sender_tokens_typed(qp_ctx* ctx, const T* x, uint64_t tokens, uint32_t C, int bits, int method, int bmode, void* d_packed,
                            qp_qparams_t* d_qp, qp_stats_t* d_stats, cudaStream_t s)
{
    uint32_t* out = static_cast<uint32_t*>(d_packed);
    switch (bits) {
        case 1: return launch_rows<1>(ctx, x, tokens, C, method, bmode, out, d_qp, d_stats, s);
        case 2: return launch_rows<2>(ctx, x, tokens, C, method, bmode, out, d_qp, d_stats, s);
        case 3: return launch_rows<3>(ctx, x, tokens, C, method, bmode, out, d_qp, d_stats, s);
        case 4: return launch_rows<4>(ctx, x, tokens, C, method, bmode, out, d_qp, d_stats, s);
        case 5: return launch_rows<5>(ctx, x, tokens, C, method, bmode, out, d_qp, d_stats, s);
        case 6: return launch_rows<6>(ctx, x, tokens, C, method, bmode, out, d_qp, d_stats, s);
        case 7: return launch_rows<7>(ctx, x, tokens, C, method, bmode, out, d_qp, d_stats, s);
        default: return launch_rows<8>(ctx, x, tokens, C, method, bmode, out, d_qp, d_stats, s);
    }
}

}  // namespace

extern "C" int32_t qp_stats_tokens(qp_ctx* ctx, const void* d_x, int dtype, uint64_t tokens, uint32_t channels,
                                   qp_stats_t* d_out, void* stream)
{
    if (!ctx) return QP_ERR_INVALID_ARG;
    if (dtype != QP_F32 && dtype != QP_BF16) return qp_fail(ctx, QP_ERR_UNSUPPORTED_DTYPE, "dtype must be QP_F32 or QP_BF16");
    int32_t rc = tok_check(ctx, tokens, channels);
    if (rc) return rc;
    if ((tokens > 0 && (!d_x || !d_out))) return qp_fail(ctx, QP_ERR_INVALID_ARG, "null pointer");
    if (((uintptr_t)d_x & (dtype == QP_F32 ? 3u : 1u)) || ((uintptr_t)d_out & 7u))
        return qp_fail(ctx, QP_ERR_ALIGNMENT, "tensor or d_out not aligned");
    if (tokens == 0) return QP_OK;
    qp_device_guard guard(ctx->device);
    if (!guard.ok) return qp_fail(ctx, QP_ERR_CUDA, "cannot select device");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (tok_rows_apply(d_x, dtype, channels, false)) {
        if (dtype == QP_F32)
            return launch_rows<0>(ctx, static_cast<const float*>(d_x), tokens, channels, 0, 0, nullptr, nullptr, d_out, s);
        return launch_rows<0>(ctx, static_cast<const unsigned short*>(d_x), tokens, channels, 0, 0, nullptr, nullptr, d_out, s);
    }
    const unsigned blocks = tok_grid(ctx, tokens);
    const bool aligned = ((uintptr_t)d_x & 15u) == 0;
    if (dtype == QP_F32) {
        const float* x = static_cast<const float*>(d_x);
        if (aligned && channels % 4 == 0) tok_stats_kernel<float, true><<<blocks, QP_THREADS, 0, s>>>(x, tokens, channels, d_out, ctx->d_status);
        else tok_stats_kernel<float, false><<<blocks, QP_THREADS, 0, s>>>(x, tokens, channels, d_out, ctx->d_status);
    } else {
        const unsigned short* x = static_cast<const unsigned short*>(d_x);
        if (aligned && channels % 8 == 0) tok_stats_kernel<unsigned short, true><<<blocks, QP_THREADS, 0, s>>>(x, tokens, channels, d_out, ctx->d_status);
        else tok_stats_kernel<unsigned short, false><<<blocks, QP_THREADS, 0, s>>>(x, tokens, channels, d_out, ctx->d_status);
    }
    ctx->launches += 1;
    return qp_check_launch(ctx, "qp_stats_tokens");
}

extern "C" int32_t qp_clip_qparams_tokens_device(qp_ctx* ctx, const qp_stats_t* d_stats, uint64_t tokens, int bits, int method,
                                                 int dist, int bmode, qp_qparams_t* d_qp_out, void* stream)
{
    if (!ctx) return QP_ERR_INVALID_ARG;
    if (tokens >= (1ull << 40)) return qp_fail(ctx, QP_ERR_INVALID_ARG, "too many tokens");
    if (tokens > 0 && (!d_stats || !d_qp_out)) return qp_fail(ctx, QP_ERR_INVALID_ARG, "null pointer");
    if (!qp_bits_ok(bits)) return qp_fail(ctx, QP_ERR_UNSUPPORTED_BITS, "bits must be 1..8 or 16");
    if (!qp_clip_method_closed_form(method))
        return qp_fail(ctx, QP_ERR_INVALID_ARG, "method must be ACIQ (| INTERSECT) or MINMAX, optionally | MIDRISE");
    if ((dist != QP_DIST_LAPLACE && dist != QP_DIST_GAUSS) || (bmode != QP_B_MAD && bmode != QP_B_MEAN_ABS))
        return qp_fail(ctx, QP_ERR_INVALID_ARG, "dist/bmode");
    if (tokens == 0) return QP_OK;
    qp_device_guard guard(ctx->device);
    if (!guard.ok) return qp_fail(ctx, QP_ERR_CUDA, "cannot select device");
    tok_clip_kernel<<<(unsigned)((tokens + 127) / 128), 128, 0, static_cast<cudaStream_t>(stream)>>>(
        d_stats, tokens, bits, method, dist, bmode, qp_host_aciq_F(bits, dist), d_qp_out, ctx->d_status);
    ctx->launches += 1;
    return qp_check_launch(ctx, "qp_clip_qparams_tokens_device");
}

extern "C" int32_t qp_quantize_pack_tokens(qp_ctx* ctx, const void* d_x, int dtype, uint64_t tokens, uint32_t channels, int bits,
                                           const qp_qparams_t* d_qp, void* d_packed, uint64_t packed_capacity, void* stream)
{
    if (!ctx) return QP_ERR_INVALID_ARG;
    if (dtype != QP_F32 && dtype != QP_BF16) return qp_fail(ctx, QP_ERR_UNSUPPORTED_DTYPE, "dtype must be QP_F32 or QP_BF16");
    int32_t rc = tok_check(ctx, tokens, channels);
    if (rc) return rc;
    if (!qp_bits_ok(bits)) return qp_fail(ctx, QP_ERR_UNSUPPORTED_BITS, "bits must be 1..8 or 16");
    const uint64_t n = tokens * channels;
    const uint64_t need = qp_packed_bytes(n, bits);
    if (packed_capacity < need) return qp_fail(ctx, QP_ERR_BUFFER_TOO_SMALL, "packed_capacity < qp_packed_bytes(n, bits)");
    if (n > 0 && (!d_qp || !d_x || !d_packed)) return qp_fail(ctx, QP_ERR_INVALID_ARG, "null pointer");
    if (((uintptr_t)d_x & (dtype == QP_F32 ? 3u : 1u)) || ((uintptr_t)d_packed & 15u) || ((uintptr_t)d_qp & 3u))
        return qp_fail(ctx, QP_ERR_ALIGNMENT, "tensor, d_packed (16 bytes) or d_qp not aligned");
    if (n == 0) return QP_OK;
    qp_device_guard guard(ctx->device);
    if (!guard.ok) return qp_fail(ctx, QP_ERR_CUDA, "cannot select device");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (dtype == QP_F32) return pack_tokens_typed<float>(ctx, static_cast<const float*>(d_x), n, channels, bits, d_qp, d_packed, s);
    return pack_tokens_typed<unsigned short>(ctx, static_cast<const unsigned short*>(d_x), n, channels, bits, d_qp, d_packed, s);
}

extern "C" int32_t qp_unpack_dequantize_tokens(qp_ctx* ctx, const void* d_packed, uint64_t tokens, uint32_t channels, int bits,
                                               const qp_qparams_t* d_qp, void* d_y, int out_dtype, void* stream)
{
    if (!ctx) return QP_ERR_INVALID_ARG;
    if (out_dtype != QP_F32 && out_dtype != QP_BF16) return qp_fail(ctx, QP_ERR_UNSUPPORTED_DTYPE, "out_dtype");
    int32_t rc = tok_check(ctx, tokens, channels);
    if (rc) return rc;
    if (!qp_bits_ok(bits)) return qp_fail(ctx, QP_ERR_UNSUPPORTED_BITS, "bits must be 1..8 or 16");
    const uint64_t n = tokens * channels;
    if (n > 0 && (!d_qp || !d_packed || !d_y)) return qp_fail(ctx, QP_ERR_INVALID_ARG, "null pointer");
    if (((uintptr_t)d_packed & 15u) || ((uintptr_t)d_qp & 3u) || ((uintptr_t)d_y & (out_dtype == QP_F32 ? 3u : 1u)))
        return qp_fail(ctx, QP_ERR_ALIGNMENT, "d_packed (16 bytes), d_qp or d_y not aligned");
    if (n == 0) return QP_OK;
    qp_device_guard guard(ctx->device);
    if (!guard.ok) return qp_fail(ctx, QP_ERR_CUDA, "cannot select device");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (out_dtype == QP_F32) return unpack_tokens_typed<float>(ctx, d_packed, n, channels, bits, d_qp, static_cast<float*>(d_y), s);
    return unpack_tokens_typed<unsigned short>(ctx, d_packed, n, channels, bits, d_qp, static_cast<unsigned short*>(d_y), s);
}

// The token-wise sender in one call: statistics -> per-token clip -> quantize+pack, nothing read back to the
// host.  d_stats_work: device memory for `tokens` statistics (80 bytes each), the caller's.
extern "C" int32_t qp_sender_tokens_device(qp_ctx* ctx, const void* d_x, int dtype, uint64_t tokens, uint32_t channels, int bits,
                                           int method, int bmode, void* d_packed, uint64_t packed_capacity,
                                           qp_qparams_t* d_qp_out, qp_stats_t* d_stats_work, void* stream)
{
    if (!ctx) return QP_ERR_INVALID_ARG;
    if (tokens > 0 && (!d_qp_out || !d_stats_work)) return qp_fail(ctx, QP_ERR_INVALID_ARG, "null d_qp_out / d_stats_work");
    int32_t rc;
    if (tokens > 0 && bits >= 1 && bits <= 8 && qp_clip_method_closed_form(method) &&
        (bmode == QP_B_MAD || bmode == QP_B_MEAN_ABS) && tok_rows_apply(d_x, dtype, channels, true)) {
        // the checks of the three calls that this one launch does not get to otherwise
        rc = tok_check(ctx, tokens, channels);
        if (rc) return rc;
        if (packed_capacity < qp_packed_bytes(tokens * channels, bits))
            return qp_fail(ctx, QP_ERR_BUFFER_TOO_SMALL, "packed_capacity < qp_packed_bytes(n, bits)");
        if (!d_packed) return qp_fail(ctx, QP_ERR_INVALID_ARG, "null pointer");
        if (((uintptr_t)d_packed & 15u) || ((uintptr_t)d_qp_out & 3u) || ((uintptr_t)d_stats_work & 7u))
            return qp_fail(ctx, QP_ERR_ALIGNMENT, "d_packed (16 bytes), d_qp_out or d_stats_work not aligned");
        qp_device_guard guard(ctx->device);
        if (!guard.ok) return qp_fail(ctx, QP_ERR_CUDA, "cannot select device");
        cudaStream_t s = static_cast<cudaStream_t>(stream);
        if (dtype == QP_F32)
            return sender_tokens_typed<float>(ctx, static_cast<const float*>(d_x), tokens, channels, bits, method, bmode, d_packed,
                                              d_qp_out, d_stats_work, s);
        return sender_tokens_typed<unsigned short>(ctx, static_cast<const unsigned short*>(d_x), tokens, channels, bits, method,
                                                   bmode, d_packed, d_qp_out, d_stats_work, s);
    }
    rc = qp_stats_tokens(ctx, d_x, dtype, tokens, channels, d_stats_work, stream);
    if (rc < 0) return rc;
    rc = qp_clip_qparams_tokens_device(ctx, d_stats_work, tokens, bits, method, QP_DIST_LAPLACE, bmode, d_qp_out, stream);
    if (rc < 0) return rc;
    return qp_quantize_pack_tokens(ctx, d_x, dtype, tokens, channels, bits, d_qp_out, d_packed, packed_capacity, stream);
}
