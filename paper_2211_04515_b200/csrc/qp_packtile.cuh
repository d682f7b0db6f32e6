// The packer's warp tile, shared by the pack kernel and by the kernels that pack at their end.
//
// A warp owns a tile of 1024 consecutive elements = 32 * BITS output words: coalesced 16-byte loads (lane l takes
// vectors l, l + 32, ..., all issued first), four codes to a quad, quads across the warp through 1 KB of shared
// memory (chunk-swizzled, conflict-free both ways), so that a lane owns the words of 32 consecutive elements.
#pragma once

#include "qp_internal.cuh"

constexpr int QP_TILE = 1024;              // elements per warp tile

// physical word of quad p in a warp's 256-word staging buffer: 16-byte chunk index XOR bit 3
__device__ __forceinline__ int qp_swz(int p) { return ((((p >> 2) ^ ((p >> 5) & 1)) << 2) | (p & 3)); }

// the words of 32 consecutive elements from their 8 quads, the g-th eight in the swizzled buffer
template <int BITS>
__device__ __forceinline__ void qp_quads_to_words(const uint32_t* sw, int g, uint32_t (&w)[BITS])
{
    const uint4 a = *reinterpret_cast<const uint4*>(&sw[qp_swz(8 * g)]);
    const uint4 b = *reinterpret_cast<const uint4*>(&sw[qp_swz(8 * g + 4)]);
    const uint32_t qd[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
    for (int m = 0; m < BITS; ++m) w[m] = 0u;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        constexpr int QB = 4 * BITS;
        const int bit = QB * k, word = bit >> 5, sh = bit & 31;
        w[word] |= qd[k] << sh;
        if (sh + QB > 32) w[(word + 1) % BITS] |= qd[k] >> (32 - sh);
    }
}

// A partial tile's elements: whole vectors as such (VEC), the others one by one, NaN for those that are missing.
template <typename T, bool VEC>
__device__ __forceinline__ void qp_load_part(const T* __restrict__ xt, int have, int lane, float (&e)[QP_TILE / (32 * qp_span<T>::EPV)][qp_span<T>::EPV])
{
    constexpr int EPV = qp_span<T>::EPV;
#pragma unroll
    for (int j = 0; j < QP_TILE / (32 * EPV); ++j) {
        const int k = (j * 32 + lane) * EPV;
        if (VEC && k + EPV <= have) {
            qp_load_vec(xt + k, e[j]);
        } else {
#pragma unroll
            for (int i = 0; i < EPV; ++i) e[j][i] = k + i < have ? qp_load_one(xt + k + i) : __int_as_float(0x7FC00000);
        }
    }
}

// Packs tile `tile` of x (n elements; the last tile may be partial: its missing elements are NaN, code 0) into `out`,
// of which nwords exist (pad words included).  VEC: x is 16-byte aligned; otherwise every lane loads the
// elements of its vectors one by one (the loads of a vector touch the same lines, so they hit L1).
// sw: 256 words of shared memory of this warp.  ALL: the caller knows that the tile has all its elements.
template <int BITS, typename T, bool VEC, bool ALL = false>
__device__ __forceinline__ void qp_pack_tile(const T* __restrict__ x, uint64_t n, uint64_t tile, int lane, float lo, float hi,
                                             float inv, uint32_t* __restrict__ out, uint64_t nwords, uint32_t* sw)
{
    constexpr int EPV = qp_span<T>::EPV;          // 4 (f32) or 8 (bf16) elements per 16-byte vector
    constexpr int NLOAD = QP_TILE / (32 * EPV);   // 8 or 4 vector loads per lane
    const T* xt = x + tile * QP_TILE;
    bool full = (tile + 1) * QP_TILE <= n;                       // warp-uniform
    if (ALL) full = true;
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
        qp_load_part<T, VEC>(xt, (int)(n - tile * QP_TILE), lane, e);
    }
    uint32_t* ot = out + tile * (32 * BITS);
    if constexpr (BITS == 8 || (BITS == 4 && EPV == 8)) {         // a vector's quads are whole words: straight to the output
        if (full) {
#pragma unroll
            for (int j = 0; j < NLOAD; ++j) {
                const int v = j * 32 + lane;
                const unsigned a = qp_quad<BITS>(e[j], lo, hi, inv);
                if constexpr (EPV == 4) {
                    ot[v] = a;
                } else {
                    const unsigned b = qp_quad<BITS>(e[j] + 4, lo, hi, inv);
                    if constexpr (BITS == 8) reinterpret_cast<uint2*>(ot)[v] = make_uint2(a, b);
                    else ot[v] = a | (b << 16);
                }
            }
            return;
        }
    }
#pragma unroll
    for (int j = 0; j < NLOAD; ++j) {
        if constexpr (EPV == 4) {
            sw[qp_swz(j * 32 + lane)] = qp_quad<BITS>(e[j], lo, hi, inv);
        } else {
            uint2 two;
            two.x = qp_quad<BITS>(e[j], lo, hi, inv);
            two.y = qp_quad<BITS>(e[j] + 4, lo, hi, inv);
            *reinterpret_cast<uint2*>(&sw[qp_swz(2 * (j * 32 + lane))]) = two;
        }
    }
    __syncwarp();
    uint32_t w[BITS];
    qp_quads_to_words<BITS>(sw, lane, w);
    if (full && BITS == 4) {
        *reinterpret_cast<uint4*>(ot + lane * 4) = make_uint4(w[0], w[1 % BITS], w[2 % BITS], w[3 % BITS]);
    } else if (full && BITS == 2) {
        *reinterpret_cast<uint2*>(ot + lane * 2) = make_uint2(w[0], w[1 % BITS]);
    } else {
        __syncwarp();
#pragma unroll
        for (int m = 0; m < BITS; ++m) sw[lane * BITS + m] = w[m];
        __syncwarp();
        const int room = ALL ? 32 * BITS : (int)min((uint64_t)(32 * BITS), nwords - tile * (32 * BITS));
#pragma unroll
        for (int m = 0; m < BITS; ++m)
            if (m * 32 + lane < room) ot[m * 32 + lane] = sw[m * 32 + lane];
    }
    __syncwarp();
}
// The same at 16 bits, where a vector's codes are whole words.  x is 16-byte aligned.
template <typename T>
__device__ __forceinline__ void qp_pack_tile16(const T* __restrict__ x, uint64_t n, uint64_t tile, int lane, float lo, float hi,
                                               float inv, uint32_t* __restrict__ out, uint64_t nwords)
{
    constexpr int EPV = qp_span<T>::EPV, NLOAD = QP_TILE / (32 * EPV);
    const T* xt = x + tile * QP_TILE;
    const bool full = (tile + 1) * QP_TILE <= n;                 // warp-uniform
    const int have = full ? QP_TILE : (int)(n - tile * QP_TILE);
    float e[NLOAD][EPV];
    if (full) {
#pragma unroll
        for (int j = 0; j < NLOAD; ++j) qp_load_vec(xt + (j * 32 + lane) * EPV, e[j]);
    } else {
        qp_load_part<T, true>(xt, have, lane, e);
    }
    uint32_t* ot = out + tile * (QP_TILE / 2);
    const uint64_t room = nwords - tile * (QP_TILE / 2);          // whole vectors: the stream is padded to 16 bytes
#pragma unroll
    for (int j = 0; j < NLOAD; ++j) {
        const int v = j * 32 + lane;
        unsigned w[EPV / 2];
#pragma unroll
        for (int i = 0; i < EPV; i += 2) {
            unsigned a = qp_code(e[j][i], lo, hi, inv, 0xFFFFu), b = qp_code(e[j][i + 1], lo, hi, inv, 0xFFFFu);
            if (!full) {
                a = v * EPV + i < have ? a : 0u;
                b = v * EPV + i + 1 < have ? b : 0u;
            }
            w[i / 2] = a | (b << 16);
        }
        if ((uint64_t)v * (EPV / 2) < room) {
            if constexpr (EPV == 4) reinterpret_cast<uint2*>(ot)[v] = make_uint2(w[0], w[1]);
            else reinterpret_cast<uint4*>(ot)[v] = make_uint4(w[0], w[1], w[2], w[3]);
        }
    }
}
