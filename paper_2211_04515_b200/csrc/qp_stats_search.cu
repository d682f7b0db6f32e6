// Statistics and directed search (paper Sec. 3, Eq. 1) of a large tensor, and in the sender the packing as well, in
// one cooperative launch (one block per SM).
//
//   phase A   sum x, sum |x|, min, max, non-finite count
//   barrier   grid-wide; every block merges the block partials in index order (the same bits everywhere)
//   phase B   sum |x - mean|, sum (x - mean)^2, histogram over [min, max]
//   barrier   every block: statistics, histogram peak -> b_R, the candidates
//   phase C   one pass that gathers, per interval between the candidates' decision thresholds, the count and
//             the sum of the elements; every block stores its row of interval sums
//   barrier   every block adds up a slice of the intervals over all rows
//   exit      block 0 turns the interval sums into the error of every candidate, picks the first minimum and writes
//             the quantizer; in the sender the other blocks wait for it and all pack
//
// Phase C needs no table of thresholds (qp_affine.cuh).  Its tables hold a replica per lane (per two lanes at 4 bits), so a
// warp's atomics meet neither the same counter nor the same bank.  They are emptied into 64-bit sums before they can
// wrap.  Integer sums: the result does not depend on the order.  Tensors whose clip ends are coarse against the quantization
// step take the "hard" form below, with the exact thresholds.
//
// What bounds it, by time stamps that the blocks took (each figure from the last block before it to its own last block; the
// stamps lengthen the launch): on 129 MB (fp32, 2 bits) phase A 25 us, the read from DRAM; barrier and merge 9; B 20 and C 23, the
// read, most of which L2 still holds, and the instructions (A and B 19 per element together, C 19, at 4 bits 35; one shared
// atomic in B, two in C); between them barrier, merge and candidates 5; rows, barrier and slices 6; block 0's scoring and
// pick 9, its result read back 1; packing 21: 119 in all.  On 39 MB at 4 bits, which L2 holds: A 9, then 9, B 6, 5, C 15, 7, 9, 1 and
// the packing 6: 67.  The calls take 114 and 64 us without the stamps, launch included; two kernels for the statistics, five for the
// search and one for the packing took 171 and 107.
#include <type_traits>

#include "qp_affine.cuh"
#include "qp_gridbar.cuh"
#include "qp_packtile.cuh"
#include "qp_tiles.cuh"

QP_CK_UNIT

namespace {

constexpr unsigned SS_UNIT_BITS = 19;             // offsets are counted in cell / 2^19
constexpr int SS_MAX_HIST = 4096;
constexpr size_t SS_TABLE_BYTES = 2 * SS_SUMS_AT; // dynamic shared memory: interval tables (counts, then sums), the exit's arrays
constexpr size_t SS_HIST_BYTES = 16512;           // and the histogram behind them (room for 4096 bins and one more)
constexpr size_t SS_DYN_BYTES = SS_TABLE_BYTES + SS_HIST_BYTES;

struct SsArgs {
    const void* x;
    uint64_t n, ntiles;                           // ntiles: whole tiles
    int nb, bits, steps, bmode, promised;
    double F;
    const qp_stats_t* st_in;                      // search only: the caller's statistics
    qp_stats_t* st_out;
    qp_ds_result_t* ds_out;
    qp_qparams_t* qp_out;
    double* curve;
    float4* cand;
    int* valid;
    qp_ds_setup* setup;
    double* part;                                 // [grid][8]
    unsigned long long* hist;                     // [nb], zero at entry and at exit
    ulonglong2* rows;                             // [grid][intervals] count, sum
    ulonglong2* tot;                              // [intervals]
    unsigned* bar;                                // [0] arrivals, [1] blocks that have left; zero at entry and at exit
    unsigned* status;
    unsigned spin_limit, bar_extra;
    int cluster;                                   // the grid is one thread-block cluster
    int hist_shift;                               // log2 of the lane replicas of a histogram bin
    int rep_shift;                                // log2 of the lane replicas of an interval
    int flush_tiles;                              // tiles per warp after which the interval tables are emptied
    uint32_t* packed;                             // sender: the packed stream
    uint64_t nwords;
};

// ---- phase A
struct SsMoments {
    double s, sa, bad;
    float mn, mx;
    unsigned odd;                                             // tiles with a non-finite value (or an fp32 overflow)
    qp_f2 s2[2];
    float a4[4], lo, hi;
    __device__ __forceinline__ void clear()
    {
        s = sa = bad = 0.0;
        mn = __int_as_float(0x7F800000);
        mx = -mn;
        odd = 0u;
    }
    __device__ __forceinline__ void one(float v)              // element by element: skips and counts NaN / Inf
    {
        if (qp_is_finite(v)) {
            s += (double)v;
            sa += (double)fabsf(v);
            mn = fminf(mn, v);
            mx = fmaxf(mx, v);
        } else {
            bad += 1.0;
        }
    }
    __device__ __forceinline__ void begin()
    {
        s2[0] = s2[1] = 0ull;
        a4[0] = a4[1] = a4[2] = a4[3] = 0.f;
        lo = mn;
        hi = mx;
    }
    __device__ __forceinline__ void pair(float a, float b, int i)
    {
        s2[i & 1] = qp_add2(s2[i & 1], qp_pack2(a, b));
        a4[(2 * i) & 3] += fabsf(a);
        a4[(2 * i + 1) & 3] += fabsf(b);
        lo = qp_min3(lo, a, b);
        hi = qp_max3(hi, a, b);
    }
    __device__ __forceinline__ void end()
    {
        const float psa = (a4[0] + a4[1]) + (a4[2] + a4[3]);
        if (psa < __int_as_float(0x7F800000)) {               // every element finite
            float sx, sy;
            qp_unpack2(qp_add2(s2[0], s2[1]), sx, sy);
            s += (double)(sx + sy);
            sa += (double)psa;
            mn = lo;
            mx = hi;
        } else {
            ++odd;
        }
    }
};

// ---- phase B: deviations and histogram.  bin = floor((x - min) * inv_w) in fp32, each operation rounded on its
// own; x = max may come out as bin nb, which is counted with the last one.  The floor is taken by adding 2^23
// rounding down; the bin number then sits in the low bits, and one multiply-add makes the address.  Positions are in
// [0, nb] where the range of the tensor and its reciprocal are finite in fp32 and the statistics are this tensor's.
// CARE 1 (the caller's statistics) keeps the bin's number in range, CARE 2 (non-finite elements, or such a range) clamps the
// position: NaN, of 0 * inf, to bin 0, what overflows to the last one.
// The deviations are taken about m, the mean in fp32 (one rounding per element, none where x and m are of a size), and
// moved to the mean itself by the counts of the two sides: sum |x - mean| = sum |x - m| - dm (N_up - N_down).  Their
// sums are taken in fp64: the search subtracts nearly all of sum y^2 again, and the conversion and fp64 pipes are idle here.
struct SsDeviations {
    float m, mn, inv_w;
    unsigned nb, hist_mul, hist_base;                         // byte address of a bin's counter = bits * hist_mul + hist_base
    double sd[2], sv[2];
    unsigned below;                                           // elements below m
    qp_f2 nm, nmn;
    template <int CARE>
    __device__ __forceinline__ void count(float pos, float x) const
    {
        if (CARE == 2) pos = fminf(fmaxf(pos, 0.f), (float)nb);
        unsigned bin = __float_as_uint(__fadd_rd(pos, SS_MAGIC)) - SS_ONE;
        if (CARE == 1) bin = min(bin, nb);
        const unsigned addr = (QP_CK(bin, nb + 1) + SS_ONE) * hist_mul + hist_base;
        if (CARE < 2 || qp_is_finite(x)) asm volatile("red.shared.add.u32 [%0], 1;" ::"r"(addr) : "memory");
    }
    __device__ __forceinline__ void begin() {}
    template <int CARE>
    __device__ __forceinline__ void take(float a, float b, int)
    {
        float da, db, pa, pb;
        const qp_f2 p = qp_pack2(a, b);
        qp_unpack2(qp_add2(p, nm), da, db);
        if (CARE == 2) {
            da = qp_is_finite(a) ? da : 0.f;
            db = qp_is_finite(b) ? db : 0.f;
        }
        const double xa = (double)da, xb = (double)db;
        sv[0] = fma(xa, xa, sv[0]);
        sv[1] = fma(xb, xb, sv[1]);
        sd[0] += fabs(xa);
        sd[1] += fabs(xb);
        below += __float_as_uint(da) >> 31;
        below += __float_as_uint(db) >> 31;
        qp_unpack2(qp_add2(p, nmn), pa, pb);
        count<CARE>(__fmul_rn(pa, inv_w), a);
        count<CARE>(__fmul_rn(pb, inv_w), b);
    }
    __device__ __forceinline__ void end() {}
    __device__ __forceinline__ void one(float v)
    {
        if (!qp_is_finite(v)) return;
        const double d = (double)__fsub_rn(v, m);
        below += d < 0.0;
        sd[0] += fabs(d);
        sv[0] = fma(d, d, sv[0]);
        count<2>(__fmul_rn(__fsub_rn(v, mn), inv_w), v);
    }
};
template <int CARE>
struct SsDeviationsOf {                                       // the stream's view of it
    SsDeviations& d;
    __device__ __forceinline__ void begin() { d.begin(); }
    __device__ __forceinline__ void pair(float a, float b, int i) { d.take<CARE>(a, b, i); }
    __device__ __forceinline__ void end() { d.end(); }
};

// The guarded pass, out of line: inlined, its code moves the compiler's schedule of the ordinary pass (128-image search sender
// 117.8 us inlined, 113.1 as a call; 64 images at 4 bits 62.9 and 62.1).
template <typename T>
__device__ __noinline__ void ss_guarded_deviations(const T* x, uint64_t ntiles, uint64_t first, uint64_t step, int lane, SsDeviations& d)
{
    SsDeviationsOf<2> f = {d};
    SsTiles<T, SS_TILE>::template run<true>(x, ntiles, first, step, lane, f);
}

template <int HH, bool GUARD>
struct SsCounter {
    const SsPlan<HH>& p;
    const SsTable& tb;
    __device__ __forceinline__ void begin() {}
    __device__ __forceinline__ void pair(float a, float b, int)
    {
        if (!GUARD || qp_is_finite(a)) ss_count<HH>(p, tb, a);
        if (!GUARD || qp_is_finite(b)) ss_count<HH>(p, tb, b);
    }
    __device__ __forceinline__ void end() {}
};

// The interval tables' contents go to this block's row (FIRST: set, otherwise added); AGAIN: and the tables back to
// zero.  A thread takes four replicas of an interval (one 16-byte read of each table, consecutive threads consecutive
// vectors).
template <bool AGAIN>
__device__ __forceinline__ void ss_flush(unsigned char* raw, int ni, int rs, ulonglong2* row, bool first)
{
    const int ts = rs - 2;                                    // log2 of the threads per interval; rs is 2 at least
    uint4* cnt = reinterpret_cast<uint4*>(raw);
    uint4* sum = cnt + SS_SUMS_AT / 16;
    const int units = 2 * ni << ts;
    for (int u0 = threadIdx.x & ~31; u0 < units; u0 += SS_THREADS) {
        const int u = u0 + (threadIdx.x & 31);
        unsigned long long cn = 0, cd = 0;
        if (u < units) {
            const uint4 c = cnt[u], d = sum[u];
            cn = (unsigned long long)c.x + c.y + ((unsigned long long)c.z + c.w);
            cd = (unsigned long long)d.x + d.y + ((unsigned long long)d.z + d.w);
            if (AGAIN) cnt[u] = sum[u] = make_uint4(0u, 0u, 0u, 0u);
        }
        for (int o = 1; o < (1 << ts); o <<= 1) {
            cn += __shfl_xor_sync(0xFFFFFFFFu, cn, o);
            cd += __shfl_xor_sync(0xFFFFFFFFu, cd, o);
        }
        if (u < units && (u & ((1 << ts) - 1)) == 0) {
            ulonglong2* at = row + (u >> ts);
            if (!first) { const ulonglong2 old = *at; cn += old.x; cd += old.y; }
            *at = make_ulonglong2(cn, cd);
        }
    }
}

// After the barrier behind the rows: this block's slice of the intervals, added up over all rows.  A warp takes every
// SS_WARPS-th row (32 consecutive intervals per read), the warps' sums meet in shared memory.  Integers: any order.
__device__ __forceinline__ void ss_slices(const SsArgs& a, int count, unsigned char* raw)
{
    ulonglong2* sh = reinterpret_cast<ulonglong2*>(raw);      // [SS_WARPS][32]
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int G = (int)gridDim.x, per = (count + G - 1) / G;
    const int e0 = blockIdx.x * per, e1 = min(e0 + per, count);
    for (int e = e0; e < e1; e += 32) {
        const int i = e + lane;
        unsigned long long n = 0, s = 0;
        if (i < e1)
#pragma unroll 5
            for (int b = warp; b < G; b += SS_WARPS) {
                const ulonglong2 v = __ldcg(a.rows + (size_t)b * count + i);
                n += v.x;
                s += v.y;
            }
        sh[warp * 32 + lane] = make_ulonglong2(n, s);
        __syncthreads();
        if (warp == 0 && i < e1) {
            for (int w = 1; w < SS_WARPS; ++w) { n += sh[w * 32 + lane].x; s += sh[w * 32 + lane].y; }
            a.tot[i] = make_ulonglong2(n, s);
        }
        __syncthreads();
    }
}

// The same for all intervals by one block, for the few rows of a cluster; the block barrier at the end makes them the
// block's to read.
__device__ __forceinline__ void ss_all_slices(const SsArgs& a, int count)
{
    const int G = (int)gridDim.x;
    for (int i = threadIdx.x; i < count; i += SS_THREADS) {
        unsigned long long n = 0, s = 0;
#pragma unroll 8
        for (int b = 0; b < G; ++b) {
            const ulonglong2 v = __ldcg(a.rows + (size_t)b * count + i);
            n += v.x;
            s += v.y;
        }
        a.tot[i] = make_ulonglong2(n, s);
    }
    __syncthreads();
}

// Exclusive prefix sums of n[0..len), s[0..len) (n[len], s[len]: the totals), by `threads` threads (a multiple of
// 32) of which this is number t; sh: 2 * threads / 32 doubles.  Block barriers inside: called by all threads.
__device__ inline void ss_scan(double* n, double* s, int len, int t, int threads, double* sh)
{
    const int per = (len + threads - 1) / threads;
    const int i0 = min(t * per, len), i1 = min(i0 + per, len);
    double a = 0.0, b = 0.0;
    for (int i = i0; i < i1; ++i) { a += n[i]; b += s[i]; }
    double pa = a, pb = b;                                    // inclusive over the warp
    for (int o = 1; o < 32; o <<= 1) {
        const double ta = __shfl_up_sync(0xFFFFFFFFu, pa, o), tb = __shfl_up_sync(0xFFFFFFFFu, pb, o);
        if ((t & 31) >= o) { pa += ta; pb += tb; }
    }
    if ((t & 31) == 31) { sh[2 * (t >> 5)] = pa; sh[2 * (t >> 5) + 1] = pb; }
    __syncthreads();
    double xa = pa - a, xb = pb - b;
    for (int w = 0; w < (t >> 5); ++w) { xa += sh[2 * w]; xb += sh[2 * w + 1]; }
    for (int i = i0; i < i1; ++i) {
        const double vn = n[i], vs = s[i];
        n[i] = xa; s[i] = xb;
        xa += vn; xb += vs;
    }
    if (t == threads - 1) { n[len] = xa; s[len] = xb; }
    __syncthreads();
}

// Block-wide: the error of every candidate is in s_curve[0..ncand); first minimum wins.
__device__ inline void ss_pick(const SsArgs& a, int ncand, const double* s_curve, const float4* s_cand, const int* s_valid,
                               const qp_ds_setup& setup)
{
    if (threadIdx.x >= 32) {
        for (int k = threadIdx.x - 32; k < ncand; k += SS_THREADS - 32) {
            a.curve[k] = s_curve[k];
            a.cand[k] = s_cand[k];
            a.valid[k] = s_valid[k];
        }
        return;
    }
    double bv = __longlong_as_double(0x7FF0000000000000ll);
    int bk = 1 << 30;
    for (int k = threadIdx.x; k < ncand; k += 32)
        if (s_curve[k] < bv) { bv = s_curve[k]; bk = k; }
    for (int o = 16; o > 0; o >>= 1) {
        const double ov = __shfl_down_sync(0xFFFFFFFFu, bv, o);
        const int ok = __shfl_down_sync(0xFFFFFFFFu, bk, o);
        if (ov < bv || (ov == bv && ok < bk)) { bv = ov; bk = ok; }
    }
    if (threadIdx.x == 0) {
        const int best = bk < ncand ? bk : 0;                 // (every error infinite or NaN: keep b_E)
        qp_ds_write_result(best, s_curve, setup, a.steps, a.nb, a.bits, s_cand[best], a.ds_out, a.qp_out, a.status);
        *a.setup = setup;
    }
}

// Block 0, after its arrival: where the boundaries of every candidate lie among the intervals (in shared memory), while
// the other blocks are still on their way.  s_cell[i]: grid cell of interval i; pos[k][i]: first interval of
// code i of a side, i = 0..HH; pos[k][HH + 1] = ni.
template <int HH>
__device__ inline void ss_places(const SsPlan<HH>& p, int ncand, int ni, int* s_edge, unsigned char* s_cell, int* pos)
{
    constexpr int C = HH + 1;
    for (int g = threadIdx.x; g <= SS_GRID; g += SS_THREADS) s_edge[g] = ss_cell_start(p, g);
    const bool flat = !(p.inv_e > 0.f);                       // no width at all: everything has the first code of its side
    for (int w = threadIdx.x; w < ncand * (C + 1); w += SS_THREADS) {
        const int k = w / (C + 1), b = w - k * (C + 1);       // boundary b = 1..HH of candidate k
        pos[w] = QP_CK(b == 0 ? 0 : (b > HH || flat) ? ni : ss_place(p, k, b), ni + 1);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < ni; i += SS_THREADS) {      // cell of an interval: the last one that starts at or before it
        int lo = 0, hi = SS_GRID;
        while (lo < hi) { const int mid = (lo + hi + 1) >> 1; if (s_edge[mid] <= i) lo = mid; else hi = mid - 1; }
        s_cell[i] = (unsigned char)lo;
    }
}

// Block 0, when the totals are complete: interval totals -> error of every candidate.
//   sum over one side and code of (|y| - level)^2 = sum y^2 + N level^2 - 2 level sum |y|,
// sum y^2 of all elements from the statistics, N and sum |y| as differences of prefix sums over the intervals.
template <int HH>
__device__ inline void ss_finish(const SsArgs& a, const SsPlan<HH>& p, const qp_stats_t& st, int ncand, int ni, const unsigned char* s_cell,
                                 const int* pos, const float4* s_cand, const int* s_valid, double* s_curve, double* sh, double* PN)
{
    constexpr int C = HH + 1, C2 = 2 * C;                     // codes of a side, of both: 2, 4, 8, 16
    double* PS = PN + 2 * (ni + 1);                           // PN, PS: [2][ni + 1] counts and sums of |y|, then their prefix sums
    for (int e0 = threadIdx.x; e0 < 2 * ni; e0 += 4 * SS_THREADS) {
        ulonglong2 t[4];
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (e0 + j * SS_THREADS < 2 * ni) t[j] = __ldcg(a.tot + e0 + j * SS_THREADS);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int e = e0 + j * SS_THREADS;
            if (e >= 2 * ni) break;
            const int side = e >= ni, i = e - side * ni;
            const double n = (double)t[j].x, ref = (double)s_cell[i] * p.w, s1 = p.u * (double)t[j].y;
            PN[side * (ni + 1) + i] = n;
            PS[side * (ni + 1) + i] = s1 + n * ref;
        }
    }
    __syncthreads();
    {
        const int side = threadIdx.x >= SS_THREADS / 2;
        ss_scan(PN + side * (ni + 1), PS + side * (ni + 1), ni, threadIdx.x - side * (SS_THREADS / 2), SS_THREADS / 2,
                sh + side * SS_WARPS);
    }
    const double nf = (double)(st.n - st.nonfinite), dm = st.mean - (double)p.m;
    const double s_abs = nf * st.mad + dm * (PN[ni] - PN[2 * ni + 1]);        // sum |y|, sum y: the sides are half sum and half difference
    const double s_sq = nf * (st.var + dm * dm);
    const double s_up = 0.5 * (s_abs + nf * dm), s_down = 0.5 * (s_abs - nf * dm);
    // a candidate's codes in C2 neighbouring lanes, added up by a fixed tree
#pragma unroll 4
    for (int w0 = threadIdx.x & ~31; w0 < ncand * C2; w0 += SS_THREADS) {
        const int w = w0 + (threadIdx.x & 31), k = w / C2, side = (w / C) & 1, i = w % C;
        double v = 0.0;
        if (k < ncand && s_valid[k]) {
            const int p0 = pos[k * (C + 1) + i], p1 = pos[k * (C + 1) + i + 1];
            const double* N = PN + side * (ni + 1);
            const double* S = PS + side * (ni + 1);
            const double s_side = side ? s_down : s_up;
            const double cn = N[p1] - N[p0], cs = (p1 == ni ? s_side : S[p1]) - (p0 == ni ? s_side : S[p0]);
            double lv = ss_level(s_cand[k], side ? HH - i : HH + 1 + i, p.m);
            if (side) lv = -lv;                               // distance from the centre, as |y|
            v = cn * lv * lv - 2.0 * lv * cs;
        }
#pragma unroll
        for (int o = C2 / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
        if (k < ncand && w % C2 == 0)
            s_curve[k] = !s_valid[k] ? __longlong_as_double(0x7FF0000000000000ll) : (nf > 0.0 ? (s_sq + v) / nf : 0.0);
    }
    __syncthreads();
}

// ---- the hard form: exact thresholds T(k, j) = smallest float with code >= j, found by bisection with the
// quantizer's own code function, sorted; an element finds its interval by binary search.  Rare (a tensor whose
// mean is hundreds of quantization steps away from zero), so one loop for every width, type and input.
struct SsHard {
    float *thr, *sorted;                                      // [M] in (k, j) order; [M] ascending
    unsigned *cnt, *lo, *hi;                                  // [(M + 1) << rs]: count, sum of the offsets' low 16 bits and of the rest
    int M, rs;
    float g_lo, g_hi;
    double u, inv_u;
};
__device__ inline void ss_hard_setup(const SsArgs& a, int ncand, const float4* s_cand, const int* s_valid, unsigned char* raw,
                                     double* sh, SsHard& h)
{
    const float inf = __int_as_float(0x7F800000);
    const int L1 = (1 << a.bits) - 1;
    double v2[2] = {(double)inf, (double)-inf};
    for (int k = threadIdx.x; k < ncand; k += SS_THREADS)
        if (s_valid[k]) { v2[0] = fmin(v2[0], (double)s_cand[k].x); v2[1] = fmax(v2[1], (double)s_cand[k].y); }
    ss_reduce<1, 2>(v2, sh);
    h.g_lo = (float)v2[0];
    h.g_hi = (float)v2[1];
    int e = 0;
    if (v2[1] > v2[0]) frexp(v2[1] - v2[0], &e);
    h.u = ldexp(1.0, e - 31);                                 // offsets stay below 2^31 units
    h.inv_u = ldexp(1.0, 31 - e);
    h.M = ncand * L1;
    h.thr = reinterpret_cast<float*>(raw);
    h.sorted = h.thr + h.M;
    h.cnt = reinterpret_cast<unsigned*>(h.sorted + h.M);
    h.rs = 3;
    while (h.rs > 0 && (size_t)8 * h.M + ((size_t)12 * (h.M + 1) << h.rs) > SS_TABLE_BYTES) --h.rs;
    h.lo = h.cnt + ((size_t)(h.M + 1) << h.rs);
    h.hi = h.lo + ((size_t)(h.M + 1) << h.rs);
    for (int t = threadIdx.x; t < h.M; t += SS_THREADS) {
        const int k = t / L1, j = 1 + t % L1;
        float out = inf;
        if (s_valid[k] && h.g_hi > h.g_lo) {
            const float4 q = s_cand[k];
            auto pred = [&](float x) { return (int)qp_code(x, q.x, q.y, q.w, (unsigned)L1) >= j; };
            if (!pred(h.g_lo) && pred(h.g_hi)) out = qp_first_true(h.g_lo, h.g_hi, pred);
        }
        h.thr[t] = out;
    }
    for (size_t i = threadIdx.x; i < ((size_t)3 * (h.M + 1) << h.rs); i += SS_THREADS) h.cnt[i] = 0u;
    __syncthreads();
    for (int t = threadIdx.x; t < h.M; t += SS_THREADS) {     // rank sort
        const float v = h.thr[t];
        int r = 0;
        for (int i = 0; i < h.M; ++i) { const float o = h.thr[i]; r += (o < v || (o == v && i < t)) ? 1 : 0; }
        h.sorted[r] = v;
    }
    __syncthreads();
}
__device__ __forceinline__ int ss_hard_at(const SsHard& h, float x)         // thresholds at or below x
{
    int lo = 0, hi = h.M;
    while (lo < hi) { const int mid = (lo + hi) >> 1; if (h.sorted[mid] <= x) lo = mid + 1; else hi = mid; }
    return lo;
}
__device__ __forceinline__ void ss_hard_one(const SsHard& h, float x, double& e_lo, double& e_hi)
{
    if (!qp_is_finite(x)) return;
    const float xc = fminf(fmaxf(x, h.g_lo), h.g_hi);
    if (x < xc) e_lo += (double)x - (double)xc;               // beyond the ends: the end's interval and the rest by itself
    if (x > xc) e_hi += (double)x - (double)xc;
    const size_t i = ((size_t)QP_CK(ss_hard_at(h, xc), h.M + 1) << h.rs) + (threadIdx.x & ((1 << h.rs) - 1));
    const unsigned d = __double2uint_rn(((double)xc - (double)h.g_lo) * h.inv_u);
    atomicAdd(&h.cnt[i], 1u);
    atomicAdd(&h.lo[i], d & 0xFFFFu);
    atomicAdd(&h.hi[i], d >> 16);
}
__device__ inline void ss_hard_flush(const SsHard& h, ulonglong2* row, bool first)
{
    for (int i = threadIdx.x; i <= h.M; i += SS_THREADS) {
        unsigned long long cn = first ? 0ull : row[i].x, cd = first ? 0ull : row[i].y;
        for (int r = 0; r < (1 << h.rs); ++r) {
            const size_t w = ((size_t)i << h.rs) + r;
            cn += h.cnt[w];
            cd += h.lo[w] + ((unsigned long long)h.hi[w] << 16);
            h.cnt[w] = h.lo[w] = h.hi[w] = 0u;
        }
        row[i] = make_ulonglong2(cn, cd);
    }
}
__device__ inline void ss_hard_finish(const SsArgs& a, const SsHard& h, float m, const qp_stats_t& st, int ncand, double e_lo,
                                      double e_hi, const float4* s_cand, const int* s_valid, double* s_curve, double* sh)
{
    // (behind the thresholds: the tables are done with)
    double* PN = reinterpret_cast<double*>(reinterpret_cast<unsigned char*>(h.thr) + ((size_t)8 * h.M + 15) / 16 * 16);
    double* PS = PN + (h.M + 2);
    for (int i = threadIdx.x; i <= h.M; i += SS_THREADS) {
        const ulonglong2 t = __ldcg(a.tot + i);
        PN[i] = (double)t.x;
        PS[i] = (double)t.x * ((double)h.g_lo - (double)m) + h.u * (double)t.y;
    }
    __syncthreads();
    ss_scan(PN, PS, h.M + 1, threadIdx.x, SS_THREADS, sh);
    const double nf = (double)(st.n - st.nonfinite), dm = st.mean - (double)m;
    const int L1 = (1 << a.bits) - 1;
    for (int k = threadIdx.x; k < ncand; k += SS_THREADS) {
        double t = nf * (st.var + dm * dm);
        int p0 = 0;
        for (int j = 0; s_valid[k] && j <= L1; ++j) {
            int p1 = h.M + 1;
            if (j < L1) {
                const float T = h.thr[k * L1 + j];
                if (T < __int_as_float(0x7F800000)) p1 = max(ss_hard_at(h, T), p0);
            }
            const double lv = ss_level(s_cand[k], j, m);
            double sum = PS[p1] - PS[p0];
            if (p0 == 0 && p1 > 0) sum += e_lo;
            if (p1 == h.M + 1 && p0 < h.M + 1) sum += e_hi;
            t += (PN[p1] - PN[p0]) * lv * lv - 2.0 * lv * sum;
            p0 = p1;
        }
        s_curve[k] = !s_valid[k] ? __longlong_as_double(0x7FF0000000000000ll) : (nf > 0.0 ? t / nf : 0.0);
    }
    __syncthreads();
}

__host__ __device__ constexpr int ss_ctile(int hh) { return hh >= 3 ? 512 : 1024; }   // phase C's tile: long code per element, short tile (instruction cache)

// STATS: phases A and B (otherwise the statistics come with st_in, and B runs only if they lack the histogram).
// HH: code boundaries above the centre, 2^bits / 2 - 1; -1: statistics only.
// What the last block out does, with what count_out returned (and whether the block itself gave up): one thread.
__device__ __forceinline__ void ss_out(const SsArgs& a, unsigned before)
{
    if (!qp_grid::last_out(before, gridDim.x)) return;
    if (before >= qp_grid::GAVE_UP)                           // (block 0 of an undisturbed launch has cleaned)
        for (int b = 0; b < a.nb; ++b) a.hist[b] = 0ull;
    qp_grid::reset(a.bar);
}

// Returns SS_GAVE_UP where a wait ran out, SS_OUT where the block has counted itself out (or is one of a cluster).
enum { SS_GAVE_UP, SS_DONE, SS_OUT };
template <typename T, bool STATS, int HH>
__device__ __forceinline__ int ss_run(const SsArgs& a)
{
    constexpr bool SEARCH = HH >= 0;
    constexpr int H = SEARCH ? HH : 0;
    extern __shared__ __align__(16) unsigned char raw[];
    __shared__ double s_red[SS_WARPS * 5];
    __shared__ int s_ok;
    __shared__ bool s_last;
    __shared__ qp_stats_t s_st;
    __shared__ qp_ds_setup s_setup;
    __shared__ SsPlan<H> s_plan;
    const T* x = static_cast<const T*>(a.x);
    const int lane = threadIdx.x & 31;
    const unsigned G = gridDim.x;
    const uint64_t first = (uint64_t)blockIdx.x * SS_WARPS + (threadIdx.x >> 5), step = (uint64_t)G * SS_WARPS;
    const uint64_t tail0 = a.ntiles * SS_TILE;
    const double inf = __longlong_as_double(0x7FF0000000000000ll);
    unsigned* bins = reinterpret_cast<unsigned*>(raw + SS_TABLE_BYTES);
    unsigned waits = 0;
    const bool cluster = a.cluster;
    auto meet = [&]() {
        if (cluster) {
            qp_grid::cluster_arrive();
            qp_grid::cluster_wait();
            return true;
        }
        ++waits;
        return qp_grid::barrier(a.bar, waits * G + a.bar_extra, a.spin_limit, a.status, &s_ok);
    };
    auto arrive = [&]() {
        __syncthreads();
        if (cluster) {
            qp_grid::cluster_arrive();
            return;
        }
        if (threadIdx.x == 0) qp_grid::arrive_release(a.bar);
    };
    auto wait = [&](unsigned target) {                        // behind arrive
        if (cluster) {
            qp_grid::cluster_wait();
            return true;
        }
        return qp_grid::wait(a.bar, target + a.bar_extra, a.spin_limit, a.status, &s_ok);
    };
    auto scratch_clean = [&]() {                              // one block, when nobody needs the scratch any more
        for (int b = threadIdx.x; b < a.nb; b += SS_THREADS) a.hist[b] = 0ull;
    };
    for (int i = threadIdx.x; i < ((a.nb + 1) << a.hist_shift); i += SS_THREADS) bins[i] = 0u;
    if constexpr (SEARCH) {                                   // (2 ni words << rep_shift are a multiple of 16 bytes)
        const int vecs = (SS_GRID + 1 + H * (a.steps + 1)) << a.rep_shift >> 1;
        for (int i = threadIdx.x; i < vecs; i += SS_THREADS)
            reinterpret_cast<uint4*>(raw)[i] = reinterpret_cast<uint4*>(raw + SS_SUMS_AT)[i] = make_uint4(0u, 0u, 0u, 0u);
    }

    // ---- phase A
    if constexpr (STATS) {
        using Tiles = SsTiles<T, SS_TILE>;
        SsMoments acc;
        acc.clear();
        Tiles::template run<false>(x, a.ntiles, first, step, lane, acc);
        if (acc.odd) {                                        // rare: this lane's share again, element by element
            acc.clear();
            for (uint64_t t = first; t < a.ntiles; t += step)
                for (int j = 0; j < SS_TILE / 32 / Tiles::EPV; ++j)
                    for (int i = 0; i < Tiles::EPV; ++i) acc.one(qp_load_one(x + t * SS_TILE + (j * 32 + lane) * Tiles::EPV + i));
        }
        if (blockIdx.x == G - 1)
            for (uint64_t i = tail0 + threadIdx.x; i < a.n; i += SS_THREADS) acc.one(qp_load_one(x + i));
        double v5[5] = {acc.s, acc.sa, (double)acc.mn, (double)acc.mx, acc.bad};
        ss_reduce<0, 0, 1, 2, 0>(v5, s_red);
        if (threadIdx.x == 0) {
            double* p = a.part + (size_t)blockIdx.x * 8;
            p[0] = v5[0]; p[1] = v5[1]; p[2] = v5[2]; p[3] = v5[3]; p[4] = v5[4];
        }
        if (!meet()) return SS_GAVE_UP;
        // one warp merges the partials (all loads in flight together), the rest of the block waits at the barrier below
        if (threadIdx.x < 32) {
            double m5[5] = {0.0, 0.0, inf, -inf, 0.0};
            for (unsigned b0 = lane; b0 < G; b0 += 32 * SS_MERGE) {
                double p[SS_MERGE][5];
#pragma unroll
                for (int u = 0; u < SS_MERGE; ++u)
#pragma unroll
                    for (int j = 0; j < 5; ++j)
                        p[u][j] = b0 + 32 * u < G ? __ldcg(a.part + (size_t)(b0 + 32 * u) * 8 + j) : (j == 2 ? inf : j == 3 ? -inf : 0.0);
#pragma unroll
                for (int u = 0; u < SS_MERGE; ++u) {
                    m5[0] += p[u][0];
                    m5[1] += p[u][1];
                    m5[2] = fmin(m5[2], p[u][2]);
                    m5[3] = fmax(m5[3], p[u][3]);
                    m5[4] += p[u][4];                         // exact: counts are far below 2^53
                }
            }
            ss_warp_reduce<0, 0, 1, 2, 0>(m5);
            if (lane == 0) {
                const unsigned long long bad = (unsigned long long)m5[4], nf = a.n - bad;
                s_st.n = a.n;
                s_st.nonfinite = bad;
                s_st.mean = nf ? m5[0] / (double)nf : 0.0;
                s_st.mean_abs = nf ? m5[1] / (double)nf : 0.0;
                s_st.min = nf ? m5[2] : 0.0;
                s_st.max = nf ? m5[3] : 0.0;
                s_st.mad = s_st.var = 0.0;
                s_st.hist_peak = 0;
                s_st.hist_bins = 0;
                s_st.reserved = 0;
            }
        }
    } else {
        if (threadIdx.x == 0) s_st = *a.st_in;
    }
    __syncthreads();

    // ---- phase B
    const bool guard = s_st.nonfinite != 0;
    const bool counting = STATS || (!a.promised && s_st.hist_bins != a.nb);
    if (counting) {
        const bool hist_on = s_st.max > s_st.min;
        {
            SsDeviations d;
            d.m = (float)s_st.mean;
            d.mn = (float)s_st.min;
            d.inv_w = hist_on ? (float)((double)a.nb / (s_st.max - s_st.min)) : 0.f;
            d.nb = (unsigned)a.nb;
            d.hist_mul = 4u << a.hist_shift;
            d.hist_base = (unsigned)__cvta_generic_to_shared(bins + (lane & ((1 << a.hist_shift) - 1))) - SS_ONE * d.hist_mul;
            d.sd[0] = d.sd[1] = d.sv[0] = d.sv[1] = 0.0;
            d.below = 0u;
            d.nm = qp_pack2(-d.m, -d.m);
            d.nmn = qp_pack2(-d.mn, -d.mn);
            if (guard || !ss_range_fits(s_st, d.inv_w)) {
                SsDeviations g = d;
                ss_guarded_deviations<T>(x, a.ntiles, first, step, lane, g);
                d.sd[0] = g.sd[0]; d.sd[1] = g.sd[1]; d.sv[0] = g.sv[0]; d.sv[1] = g.sv[1]; d.below = g.below;
            } else {
                SsDeviationsOf<STATS ? 0 : 1> f = {d};
                SsTiles<T, SS_TILE>::template run<true>(x, a.ntiles, first, step, lane, f);
            }
            if (blockIdx.x == G - 1)
                for (uint64_t i = tail0 + threadIdx.x; i < a.n; i += SS_THREADS) d.one(qp_load_one(x + i));
            double v3[3] = {d.sd[0] + d.sd[1], d.sv[0] + d.sv[1], (double)d.below};
            ss_reduce<0, 0, 0>(v3, s_red);                    // (its barriers also order the counters)
            if (STATS && threadIdx.x == 0)
#pragma unroll
                for (int j = 0; j < 3; ++j) a.part[(size_t)blockIdx.x * 8 + 5 + j] = v3[j];
        }
        const int reps = 1 << a.hist_shift;
        for (int b = threadIdx.x; hist_on && b < a.nb; b += SS_THREADS) {
            unsigned long long c = 0;
            for (int r = 0; r < reps; ++r) c += bins[(b << a.hist_shift) + ((r + threadIdx.x) & (reps - 1))];
            if (b == a.nb - 1)
                for (int r = 0; r < reps; ++r) c += bins[(a.nb << a.hist_shift) + r];
            if (c) atomicAdd(&a.hist[b], c);
        }
        if constexpr (SEARCH) {
            if (!meet()) return SS_GAVE_UP;
        } else {                                              // statistics only: the last block out finishes
            __threadfence();
            __syncthreads();
            if (threadIdx.x == 0) {
                const unsigned before = qp_grid::count_out(a.bar);
                s_last = before == G - 1;                     // (with a block that gave up among those before: no output)
                if (!s_last) ss_out(a, before);
            }
            __syncthreads();
            if (!s_last) return SS_OUT;
            __threadfence();
        }
        if (threadIdx.x < 32) {
            double v3[4] = {0.0, 0.0, 0.0, 0.0};              // sum |x - m|, sum (x - m)^2, elements below m; largest bin
            if (STATS)
                for (unsigned b0 = lane; b0 < G; b0 += 32 * SS_MERGE) {
                    double p[SS_MERGE][3];
#pragma unroll
                    for (int u = 0; u < SS_MERGE; ++u)
#pragma unroll
                        for (int j = 0; j < 3; ++j)
                            p[u][j] = b0 + 32 * u < G ? __ldcg(a.part + (size_t)(b0 + 32 * u) * 8 + 5 + j) : 0.0;
#pragma unroll
                    for (int u = 0; u < SS_MERGE; ++u)
#pragma unroll
                        for (int j = 0; j < 3; ++j) v3[j] += p[u][j];
                }
            if (hist_on)
                for (int b0 = lane; b0 < a.nb; b0 += 32 * 4) {
                    unsigned long long c[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) c[u] = b0 + 32 * u < a.nb ? __ldcg(&a.hist[b0 + 32 * u]) : 0ull;
#pragma unroll
                    for (int u = 0; u < 4; ++u) v3[3] = fmax(v3[3], (double)c[u]);
                }
            ss_warp_reduce<0, 0, 0, 2>(v3);
            if (lane == 0) {
                if (STATS) {
                    const double nf = (double)(a.n - s_st.nonfinite), dm = s_st.mean - (double)(float)s_st.mean;
                    s_st.mad = nf > 0.0 ? fmax(0.0, v3[0] - dm * (nf - 2.0 * v3[2])) / nf : 0.0;
                    s_st.var = nf > 0.0 ? fmax(0.0, v3[1] / nf - dm * dm) : 0.0;
                }
                s_st.hist_peak = (unsigned long long)v3[3];
                s_st.hist_bins = a.nb;
                if (STATS && (!SEARCH || blockIdx.x == 0)) {
                    *a.st_out = s_st;
                    if (s_st.nonfinite) atomicOr(a.status, QP_DEV_NONFINITE);
                }
            }
        }
        __syncthreads();
        if constexpr (!SEARCH) {
            scratch_clean();
            if (threadIdx.x == 0) qp_grid::reset(a.bar);
            return SS_OUT;
        }
    }

    // ---- phase C
    if constexpr (SEARCH) {
        constexpr int BITS = H == 0 ? 1 : H == 1 ? 2 : H == 3 ? 3 : 4;
        const int ncand = a.steps + 1, ni = SS_GRID + 1 + H * ncand;
        __shared__ float4 s_cand[QP_SS_MAX_CAND];
        __shared__ int s_valid[QP_SS_MAX_CAND];
        __shared__ double s_curve[QP_SS_MAX_CAND];
        __shared__ int s_edge[SS_GRID + 1];                   // interval that a grid cell starts with
        __shared__ unsigned char s_cell[SS_GRID + 1 + H * QP_SS_MAX_CAND];
        {                                                     // every thread the same set-up, then its part of the plan and its candidates
            const bool have = s_st.hist_bins == a.nb;
            if (!have && blockIdx.x == 0 && threadIdx.x == 0) atomicOr(a.status, QP_DEV_HIST_MISSING);
            qp_ds_setup su;
            qp_ds_make_setup(&s_st, have ? s_st.hist_peak : 0ull, a.nb, a.bmode, a.F, su);
            su.g_lo = su.g_hi = su.inv_gw = su.inv_u = su.gw = su.pad2 = 0.f;
            su.u = 0.0;
            if (threadIdx.x < 32) {
                if (lane == 0) s_setup = su;
                const double k = su.F * ((a.bmode & QP_B_MIDRISE) ? 1.0 - 1.0 / (double)(1 << BITS) : 1.0);
                ss_make_plan<H>(s_plan, (int)threadIdx.x - 1, s_st.mean, k * su.b_e, k * (su.degenerate ? su.b_e : su.b_r), su.degenerate ? 1 : ncand, BITS, SS_UNIT_BITS);
            } else {
                for (int k = threadIdx.x - 32; k < ncand; k += SS_THREADS - 32) {
                    float4 c;
                    int ok;
                    qp_ds_candidate(su, k, a.steps, BITS, a.bmode & QP_B_MIDRISE, c, ok);
                    s_cand[k] = c;
                    s_valid[k] = ok;
                }
            }
        }
        __syncthreads();
        const bool hard = s_plan.hard;
        SsHard h;
        h.M = 0;
        if (!hard) {
            constexpr int CT = ss_ctile(H);
            const SsPlan<H> p = s_plan;
            SsTable tb;
            tb.mul = 4u << a.rep_shift;
            tb.base = (unsigned)__cvta_generic_to_shared(raw) + 4u * (lane & ((1 << a.rep_shift) - 1)) - SS_ONE * tb.mul;
            tb.half = (unsigned)ni * tb.mul;
            tb.ni = (unsigned)ni;
            tb.ub = SS_UNIT_BITS;
            tb.scale = (float)(SS_GRID << SS_UNIT_BITS);
            ulonglong2* row = a.rows + (size_t)blockIdx.x * (2 * ni);
            const uint64_t per = (uint64_t)a.flush_tiles * step;      // tiles of all warps between two flushes
            const uint64_t ntiles = a.ntiles * (SS_TILE / CT);
            for (uint64_t t0 = 0; t0 < ntiles; t0 += per) {
                const uint64_t t1 = ntiles - t0 < per ? ntiles : t0 + per;
                if (t0) {
                    __syncthreads();
                    ss_flush<true>(raw, ni, a.rep_shift, row, t0 == per);
                    __syncthreads();
                }
                if (guard) {
                    SsCounter<H, true> f = {p, tb};
                    SsTiles<T, CT>::template run<false>(x, t1, t0 + first, step, lane, f);
                } else {
                    SsCounter<H, false> f = {p, tb};
                    SsTiles<T, CT>::template run<false>(x, t1, t0 + first, step, lane, f);
                }
            }
            if (blockIdx.x == G - 1)
                for (uint64_t i = tail0 + threadIdx.x; i < a.n; i += SS_THREADS) {
                    const float v = qp_load_one(x + i);
                    if (qp_is_finite(v)) ss_count<H>(p, tb, v);
                }
            __syncthreads();
            ss_flush<false>(raw, ni, a.rep_shift, row, ntiles <= per);
        } else {
            double e2[2] = {0.0, 0.0};
            ss_hard_setup(a, ncand, s_cand, s_valid, raw, s_red, h);
            ulonglong2* row = a.rows + (size_t)blockIdx.x * (h.M + 1);
            int since = 0;
            bool fresh = true;
            for (uint64_t t0 = 0; t0 < a.ntiles; t0 += step) {        // uniform over the block: the flush has barriers
                const uint64_t t = t0 + first;
                if (t < a.ntiles)
                    for (int i = lane; i < SS_TILE; i += 32) ss_hard_one(h, qp_load_one(x + t * SS_TILE + i), e2[0], e2[1]);
                if (++since == 3) {                           // 2^16 offset halves of 16 bits fill a word
                    __syncthreads();
                    ss_hard_flush(h, row, fresh);
                    __syncthreads();
                    since = 0;
                    fresh = false;
                }
            }
            if (blockIdx.x == G - 1)
                for (uint64_t i = tail0 + threadIdx.x; i < a.n; i += SS_THREADS) ss_hard_one(h, qp_load_one(x + i), e2[0], e2[1]);
            ss_reduce<0, 0>(e2, s_red);
            if (threadIdx.x == 0) {
                a.part[(size_t)blockIdx.x * 8] = e2[0];
                a.part[(size_t)blockIdx.x * 8 + 1] = e2[1];
            }
            ss_hard_flush(h, row, fresh);
        }
        const int count = hard ? h.M + 1 : 2 * ni;
        if (!cluster) {
            if (!meet()) return SS_GAVE_UP;
            ss_slices(a, count, raw + SS_TABLE_BYTES);
        }
        arrive();
        if (blockIdx.x == 0) {
            int* pos = reinterpret_cast<int*>(raw + SS_TABLE_BYTES);          // [ncand][H + 2] in the histogram's room (the slices are stored)
            if (!hard) ss_places<H>(s_plan, ncand, ni, s_edge, s_cell, pos);
            if (!wait((waits + 1) * G)) return SS_GAVE_UP;
            if (cluster) ss_all_slices(a, count);
            if (!hard) {
                ss_finish<H>(a, s_plan, s_st, ncand, ni, s_cell, pos, s_cand, s_valid, s_curve, s_red, reinterpret_cast<double*>(raw));
            } else {
                double v2[2] = {0.0, 0.0};
                for (unsigned b = threadIdx.x; b < G; b += SS_THREADS)
#pragma unroll
                    for (int j = 0; j < 2; ++j) v2[j] += __ldcg(a.part + (size_t)b * 8 + j);
                ss_reduce<0, 0>(v2, s_red);
                ss_hard_finish(a, h, s_plan.m, s_st, ncand, v2[0], v2[1], s_cand, s_valid, s_curve, s_red);
            }
            // (a warp that the pick does not wait for asks meanwhile)
            if (!cluster && !a.packed && threadIdx.x == SS_THREADS - 1) ss_out(a, qp_grid::count_out(a.bar));
            ss_pick(a, ncand, s_curve, s_cand, s_valid, s_setup);
            scratch_clean();
            if (!a.packed) return SS_OUT;
            arrive();
        } else {
            if (cluster) {
                wait(0);
                if (a.packed) arrive();
            }
            if (!a.packed) {
                if (threadIdx.x == 0) __threadfence();        // (the arrival, which nobody here polls for)
                return SS_DONE;
            }
        }
        if constexpr (STATS) {                                // the sender: everybody packs, from the tensor's end
            if (!wait((waits + 1) * G + 1)) return SS_GAVE_UP;
            const float lo = __ldcg(&a.qp_out->lo), hi = __ldcg(&a.qp_out->hi), inv = __ldcg(&a.qp_out->inv_scale);
            uint32_t* sw = reinterpret_cast<uint32_t*>(raw) + (threadIdx.x >> 5) * 256;
            const uint64_t tiles = (a.n + QP_TILE - 1) / QP_TILE;
            for (uint64_t it = first; it < tiles; it += step)
                qp_pack_tile<BITS, T, true>(x, a.n, tiles - 1 - it, lane, lo, hi, inv, a.packed, a.nwords, sw);
        }
    }
    return SS_DONE;
}

template <typename T, bool STATS, int HH>
__global__ void __launch_bounds__(SS_THREADS, 1) stats_search_kernel(const SsArgs a)
{
    const int how = ss_run<T, STATS, HH>(a);
    if (threadIdx.x != 0 || a.cluster || how == SS_OUT) return;
    const unsigned gave_up = how == SS_GAVE_UP ? qp_grid::GAVE_UP : 0u;
    ss_out(a, qp_grid::count_out(a.bar, gave_up) | gave_up);
}

template <typename T>
void* ss_kernel(bool stats, int bits)                         // bits 0: statistics only
{
    if (bits == 0) return (void*)stats_search_kernel<T, true, -1>;
    if (stats) return bits == 1 ? (void*)stats_search_kernel<T, true, 0> : bits == 2 ? (void*)stats_search_kernel<T, true, 1>
                    : bits == 3 ? (void*)stats_search_kernel<T, true, 3> : (void*)stats_search_kernel<T, true, 7>;
    return bits == 1 ? (void*)stats_search_kernel<T, false, 0> : bits == 2 ? (void*)stats_search_kernel<T, false, 1>
         : bits == 3 ? (void*)stats_search_kernel<T, false, 3> : (void*)stats_search_kernel<T, false, 7>;
}

// Whether this device can hold the launch (checked once per context).
bool ss_usable(qp_ctx* ctx)
{
    if (!ctx->ss_checked) {
        ctx->ss_checked = 1;
        int coop = 0, optin = 0;
        // the scratch that other forms own: block partials, and the interval path's rows
        bool ok = cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, ctx->device) == cudaSuccess && coop &&
                  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, ctx->device) == cudaSuccess &&
                  (size_t)ctx->sm_count * 8 * sizeof(double) <= sizeof(qp_stats_partial) * QP_MAX_BLOCKS &&
                  (size_t)ctx->sm_count * QP_SS_TOTALS * 2 <= (size_t)ctx->iv_blocks * (QP_IV_MAXB + 1);
        for (int bits = 0; ok && bits <= 4; ++bits)
            for (int v = 0; ok && v < (bits ? 4 : 2); ++v) {
                void* k = (v & 1) ? ss_kernel<unsigned short>(v < 2, bits) : ss_kernel<float>(v < 2, bits);
                cudaFuncAttributes fa;
                int per_sm = 0;
                ok = cudaFuncGetAttributes(&fa, k) == cudaSuccess && (size_t)optin >= fa.sharedSizeBytes + SS_DYN_BYTES &&
                     cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SS_DYN_BYTES) == cudaSuccess &&
                     cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, SS_THREADS, SS_DYN_BYTES) == cudaSuccess && per_sm >= 1;
            }
        ctx->ss_cluster = ok;
        for (int bits = 0; ok && bits <= 4; ++bits)
            for (int v = 0; v < (bits ? 4 : 2); ++v)
                ctx->ss_cluster &= qp_cluster_fits((v & 1) ? ss_kernel<unsigned short>(v < 2, bits) : ss_kernel<float>(v < 2, bits),
                                                   SS_THREADS, SS_DYN_BYTES);
        if (!ok) cudaGetLastError();
        ctx->ss_ok = ok ? 1 : 0;
    }
    return ctx->ss_ok != 0;
}

}  // namespace

// 16-byte aligned tensors; statistics with the histogram from 128 KB on (where qp_stats_carries_histogram says so), the search
// from 8 tiles on, at 4 bits from 128 KB: 12 to 23 us by width up to 2^20 elements, where the candidates scored one by one take 23 us at
// 2^15, 33 at 2^18 and 60 at 2^20.  (Below 128 KB the statistics carry no histogram and the launch counts it as well: 17 to 28 us at 1..3
// bits, 33 at 4, against 25 to 29.)  At 1..4 bits (each further code boundary costs two instructions per element: at 5 bits and up the
// interval pass with its table is the cheaper one) and up to 256 candidates (tables that leave a replica to every
// eighth lane at least).
bool qp_stats_search_applies(qp_ctx* ctx, const void* d_x, int dtype, uint64_t n, int hist_bins, int bits, int steps)
{
    if (((uintptr_t)d_x & 15u) || hist_bins < 1 || hist_bins > SS_MAX_HIST) return false;
    const bool small = n * (dtype == QP_F32 ? 4 : 2) < 131072;
    if (bits == 0 || bits == 4 ? small : n < 8 * SS_TILE) return false;
    if (bits && (bits > 4 || steps + 1 > QP_SS_MAX_CAND)) return false;
    return ss_usable(ctx);
}

// Statistics with the histogram (bits = 0), the search on the caller's statistics (st_in), or both, then with d_packed
// also the packed stream.
int32_t qp_launch_stats_search(qp_ctx* ctx, const void* d_x, int dtype, uint64_t n, const qp_stats_t* st_in, qp_stats_t* st_out,
                               int hist_bins, int bits, int bmode, int steps, double F, qp_ds_result_t* d_out,
                               qp_qparams_t* d_qp_out, void* d_packed, cudaStream_t s)
{
    static_assert(2 * (SS_GRID + 1 + 7 * QP_SS_MAX_CAND) <= QP_SS_TOTALS && 15 * QP_SS_MAX_CAND + 1 <= QP_SS_TOTALS, "interval totals");
    static_assert(QP_SS_MAX_CAND * 9 * sizeof(int) <= SS_HIST_BYTES && SS_WARPS * 32 * 16 <= SS_HIST_BYTES, "the histogram's room is used again");
    SsArgs a;
    a.x = d_x;
    a.n = n;
    a.ntiles = n / SS_TILE;
    a.nb = hist_bins;
    a.bits = bits;
    a.steps = steps;
    a.bmode = bmode & ~QP_B_HIST_IN_STATS;
    a.promised = (bmode & QP_B_HIST_IN_STATS) ? 1 : 0;
    a.F = F;
    a.st_in = st_in;
    a.st_out = st_out;
    a.ds_out = d_out;
    a.qp_out = d_qp_out;
    a.curve = ctx->d_curve;
    a.cand = ctx->d_cand;
    a.valid = ctx->d_valid;
    a.setup = ctx->d_setup;
    a.part = reinterpret_cast<double*>(ctx->d_part);
    unsigned char* f = static_cast<unsigned char*>(ctx->d_fused);
    a.bar = reinterpret_cast<unsigned*>(f) + 16;              // words 16, 17 (the sender uses 0, 1, the statistics 8..10 and 24, 25)
    a.hist = reinterpret_cast<unsigned long long*>(f + 256);
    a.tot = reinterpret_cast<ulonglong2*>(f + QP_FUSED_TOTALS_AT);
    a.rows = reinterpret_cast<ulonglong2*>(ctx->d_iv_part);
    a.status = ctx->d_status;
    a.spin_limit = ctx->spin_limit;
    a.bar_extra = (unsigned)ctx->bar_extra;
    a.packed = static_cast<uint32_t*>(d_packed);
    a.nwords = d_packed ? qp_packed_bytes(n, bits) / 4 : 0;
    // as many lane replicas as fit
    a.hist_shift = 5;
    while (a.hist_shift > 0 && ((size_t)(hist_bins + 1) << a.hist_shift) * sizeof(unsigned) > SS_HIST_BYTES) --a.hist_shift;
    const int hh = bits ? (1 << bits) / 2 - 1 : 0;
    const size_t ni = bits ? (size_t)SS_GRID + 1 + (size_t)hh * (steps + 1) : 0;
    a.rep_shift = 5;
    while (a.rep_shift > 0 && (4 * ni << a.rep_shift) * sizeof(unsigned) > SS_TABLE_BYTES) --a.rep_shift;
    // an offset is at most 2^19: 8191 of them stay below 2^32.  A tile of every warp is shared evenly by the replicas; 64 less
    // for the elements behind the last tile
    a.flush_tiles = ((8191 - 64) << a.rep_shift) / (SS_WARPS * ss_ctile(hh));
    if (a.flush_tiles < 1) return qp_fail(ctx, QP_ERR_INVALID_ARG, "statistics and search: tables too small");
    const uint64_t want = (a.ntiles + SS_WARPS - 1) / SS_WARPS;
    a.cluster = qp_cluster_wanted(ctx, ctx->ss_cluster, n);
    const unsigned most = a.cluster ? QP_CLUSTER_BLOCKS : (unsigned)ctx->sm_count;
    const unsigned G = (unsigned)(want < most ? want : most);
    void* k = dtype == QP_F32 ? ss_kernel<float>(st_in == nullptr, bits) : ss_kernel<unsigned short>(st_in == nullptr, bits);
    void* params[] = {&a};
    if (qp_launch_together(k, G, SS_THREADS, params, SS_DYN_BYTES, a.cluster, s) != cudaSuccess)
        return qp_check_launch(ctx, "statistics and search (cooperative launch)");
    ctx->launches += 1;
    return qp_check_launch(ctx, "statistics and search");
}
