// Statistics and directed search (paper Sec. 3, Eq. 1) of a large tensor, and in the sender the packing as well, in
// one cooperative launch (one block per SM).
//
//   phase A   sum x, sum |x|, min, max, non-finite count
//   barrier   grid-wide; every block merges the block partials in index order (the same bits everywhere)
//   phase B   sum |x - mean|, sum (x - mean)^2, histogram over [min, max]
//   barrier   every block: statistics, histogram peak -> b_R, the candidates
//   phase C   one pass that gathers, per interval between the candidates' decision thresholds, the count and
//             the sum of the elements; every block makes of its own sums its part of the error of every candidate
//   barrier   the parts are added up in 64-bit integers; every block takes the first minimum, and block 0 writes the result
//   packing   in the sender, from the tensor's end
//
// With one bit a side has one code, so that the statistics tell the errors: the sender packs behind phase B, and the separate search
// only counts the elements below the centre.
//
// Phase C needs no table of thresholds (qp_affine.cuh).  Its tables hold a replica per lane (per two lanes at 4 bits), so a
// warp's atomics meet neither the same counter nor the same bank.  They are emptied into 64-bit sums before they can
// wrap.  Integer sums: the result does not depend on the order.  Tensors whose clip ends are coarse against the quantization
// step take the "hard" form below, with the exact thresholds.
//
// What bounds it, by time stamps that the blocks took (each figure from the last block before it to its own last block; the
// stamps lengthen the launch by 2 to 3 us): on 129 MB (fp32, 2 bits) phase A 23 us, the read from DRAM; barrier and merge 3.5; B 17.5 and C
// 20, the read, most of which L2 still holds, and the instructions (A and B 19 per element together, C 19, at 4 bits 35; one shared
// atomic in B, two in C); between them histogram, barrier, merge and candidates 5; a block's prefix sums and errors 2, barrier and pick
// 3; packing 19.  On 39 MB at 4 bits, which L2 holds: A 8, then 3.5, B 5.5, 5, C 11, 4, 2.5 and the packing 4: 44 and 3 between launches.
// Both calls took 15 us longer with the blocks' intervals added up by all of them in slices, behind a barrier of their own, the scoring
// by block 0 alone with the others waiting, and block partials 64 bytes apart.  One image (151 K, a cluster of 10 blocks) at 2 bits, 17 us:
// A 1.2, 1.9, B 1.9, 4.4 up to the candidates, C 2.3, 2 and 2.5 for scoring and pick, packing 0.9.
// Shuffles by lanes that have parted cost 250 cycles each instead of 30 (the finish 3.6 us instead of 1.3; the whole launch on one
// image 3.3 us longer without the __syncwarp behind the tail's elements): hence the __syncwarp before them and the grid barrier whose
// whole warp polls.
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
    uint4* part;                                  // [4][grid] block partials, 16 bytes each
    unsigned long long* hist;                     // [nb]; the sender's own, otherwise zero at entry and at exit
    ulonglong2* rows;                             // [grid][intervals] count, sum: what a block emptied its tables of on the way
    unsigned long long* acc;                      // [ncand + 2]: errors of the candidates in fixed point (the sender's own); search only: the
                                                  // elements below the centre and the others, all zero at entry and at exit
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
    double s, sa;
    float mn, mx;
    unsigned bad;
    unsigned odd;                                             // tiles with a non-finite value (or an fp32 overflow)
    qp_f2 s2[2];
    float a4[4], lo, hi;
    __device__ __forceinline__ void clear()
    {
        s = sa = 0.0;
        mn = __int_as_float(0x7F800000);
        mx = -mn;
        bad = odd = 0u;
    }
    __device__ __forceinline__ void one(float v)              // element by element: skips and counts NaN / Inf
    {
        if (qp_is_finite(v)) {
            s += (double)v;
            sa += (double)fabsf(v);
            mn = fminf(mn, v);
            mx = fmaxf(mx, v);
        } else {
            ++bad;
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
// 101.3 us inlined, 98.9 as a call; 64 images at 4 bits 47.7 and 45.9).
template <typename T>
__device__ __noinline__ void ss_guarded_deviations(const T* x, uint64_t ntiles, uint64_t first, uint64_t step, int lane, SsDeviations& d)
{
    SsDeviationsOf<2> f = {d};
    SsTiles<T, SS_TILE>::template run<true>(x, ntiles, first, step, lane, f);
}

// One bit: how many elements lie below m, of how many.
struct SsSides {
    float m;
    bool guard;
    unsigned down, all;
    __device__ __forceinline__ void begin() {}
    __device__ __forceinline__ void pair(float a, float b, int) { one(a, guard); one(b, guard); }
    __device__ __forceinline__ void end() {}
    __device__ __forceinline__ void one(float v, bool check = true)
    {
        if (check && !qp_is_finite(v)) return;
        down += __float_as_uint(__fsub_rn(v, m)) >> 31;
        ++all;
    }
};

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

// The interval tables' contents go to this block's row (first: set, otherwise added) and the tables back to zero.  A thread
// takes four replicas of an interval (one 16-byte read of each table, consecutive threads consecutive vectors).
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
            cnt[u] = sum[u] = make_uint4(0u, 0u, 0u, 0u);
        }
        __syncwarp();
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

// The block's histogram goes into the tensor's; what x = max put into bin nb counts in the last one.
__device__ __forceinline__ void ss_hist_out(const unsigned* bins, int nb, int shift, unsigned long long* hist)
{
    const int ts = shift >= 2 ? shift - 2 : 0, units = (nb + 1) << ts;        // a thread takes four replicas of a bin, or all
    for (int u0 = threadIdx.x & ~31; u0 < units; u0 += SS_THREADS) {
        const int u = u0 + (threadIdx.x & 31);
        unsigned c = 0u;
        if (u < units) {
            if (shift >= 2) {
                const uint4 v = reinterpret_cast<const uint4*>(bins)[u];
                c = v.x + v.y + (v.z + v.w);
            } else {
                for (int r = 0; r < (1 << shift); ++r) c += bins[(u << shift) + r];
            }
        }
        __syncwarp();
        for (int o = 1; o < (1 << ts); o <<= 1) c += __shfl_xor_sync(0xFFFFFFFFu, c, o);
        if (u < units && (u & ((1 << ts) - 1)) == 0 && c) atomicAdd(&hist[min(u >> ts, nb - 1)], (unsigned long long)c);
    }
}

// A side's elements below interval i, this block's: counts and sums of |y| in units of p.u, exclusive prefix sums over the
// side's intervals, in the place of the interval's own counters (16 bytes of them; an interval has four counters at least).  Half the
// block per side, a thread takes `per` consecutive intervals.  per is odd, and the order in which a lane reads the vectors of an
// interval, as well as which of them becomes the slot, turns with the lane and with the interval, so that the eight lanes of a 16-byte
// access meet no bank twice (1.9 us at 4 bits, 4.3 without the turn, 2.6 with three intervals at a time).  A block's counts stay below 2^32 (the tensor would
// have to have 6e11 elements).  Returns (to everybody) the elements of the two sides.
__device__ __forceinline__ ulonglong2* ss_slot(unsigned char* raw, int e, int rs)
{
    return reinterpret_cast<ulonglong2*>(raw + ((size_t)e << (rs + 2)) + (((e >> (5 - rs)) & ((1 << (rs - 2)) - 1)) << 4));
}
__device__ __forceinline__ uint2 ss_prefix(unsigned char* raw, int ni, int rs, const ulonglong2* row, const int* s_edge, ulonglong2* sh)
{
    constexpr int HALF = SS_THREADS / 2, HW = SS_WARPS / 2;
    static_assert(SS_GRID == 64, "two steps of eight");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, side = threadIdx.x >= HALF, t = threadIdx.x - side * HALF;
    const int per = ((ni + HALF - 1) / HALF) | 1, vecs = 1 << (rs - 2), turn = lane >> (5 - rs);
    const int i0 = min(t * per, ni), i1 = min(i0 + per, ni);
    int cell = 0;                                             // the last cell that starts at or before i0
#pragma unroll
    for (int g = 8; g <= 64; g += 8) cell += s_edge[g] <= i0 ? 8 : 0;
    int more = 0;
#pragma unroll
    for (int g = 1; g < 8; ++g) more += s_edge[min(cell + g, SS_GRID + 1)] <= i0 ? 1 : 0;
    cell += more;
    // (every cell starts an interval, so that an interval is in the cell of the one before it or in the next: no loop that parts lanes)
    int next = s_edge[cell + 1];
    unsigned n = 0u;
    unsigned long long s = 0ull;
    for (int i = i0; i < i1; ++i) {
        const int e = side * ni + i;
        const uint4* cnt = reinterpret_cast<const uint4*>(raw) + ((size_t)e << (rs - 2));
        unsigned cn = 0u;                                     // (a flush's counts, and a block's, are below 2^32)
        unsigned long long cd = 0ull;
#pragma unroll 4
        for (int v = 0; v < vecs; ++v) {
            const int at = (v + turn) & (vecs - 1);
            const uint4 c = cnt[at], d = cnt[SS_SUMS_AT / 16 + at];
            cn += c.x + c.y + (c.z + c.w);
            cd += (unsigned long long)d.x + d.y + ((unsigned long long)d.z + d.w);
        }
        cell += next <= i ? 1 : 0;
        next = s_edge[cell + 1];
        if (row) { cn += (unsigned)row[e].x; cd += row[e].y; }
        *ss_slot(raw, e, rs) = make_ulonglong2(n, s);
        n += cn;
        s += cd + (((unsigned long long)cn * (unsigned)cell) << SS_UNIT_BITS);
    }
    __syncwarp();
    unsigned pn = n;                                          // inclusive over the warp, then over the warps of the side
    unsigned long long ps = s;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned tn = __shfl_up_sync(0xFFFFFFFFu, pn, o);
        const unsigned long long ts = __shfl_up_sync(0xFFFFFFFFu, ps, o);
        if (lane >= o) { pn += tn; ps += ts; }
    }
    if (lane == 31) sh[warp] = make_ulonglong2(pn, ps);
    __syncthreads();
    pn -= n;
    ps -= s;
#pragma unroll
    for (int w = 0; w < HW - 1; ++w) {
        const ulonglong2 o = sh[side * HW + w];
        if (w < (warp & (HW - 1))) { pn += (unsigned)o.x; ps += o.y; }
    }
#pragma unroll 3
    for (int i = i0; i < i1; ++i) {
        ulonglong2* at = ss_slot(raw, side * ni + i, rs);
        const ulonglong2 v = *at;
        *at = make_ulonglong2(v.x + pn, v.y + ps);
    }
    uint2 all = make_uint2(0u, 0u);
    for (int w = 0; w < HW; ++w) { all.x += (unsigned)sh[w].x; all.y += (unsigned)sh[HW + w].x; }
    return all;
}

// Where the boundaries of every candidate lie among the intervals: pos[k][b - 1], the first interval of code b = 1..HH of a
// side.  s_edge: the interval that a grid cell starts with; behind the last, none.
template <int HH>
__device__ __forceinline__ void ss_places(const SsPlan<HH>& p, int ncand, int ni, int* s_edge, int* pos)
{
    for (int w = threadIdx.x; w < ncand * HH; w += SS_THREADS) {
        const int k = w / HH, b = w - k * HH + 1;
        pos[w] = QP_CK(ss_place(p, k, b), ni);
    }
    for (int g = threadIdx.x; g <= SS_GRID + 1; g += SS_THREADS) s_edge[g] = g <= SS_GRID ? ss_cell_start(p, g) : 1 << 30;
}

// The error of candidate k is, over the elements,
//   sum y^2 + sum over both sides of sum_i (N_i level_i^2 - 2 level_i S_i),   N_i, S_i: count and sum of |y| of code i of the side,
// and with the prefix sums P(b) at the first interval of code b the sum over the codes i of a side is
//   N level_HH^2 - 2 S level_HH - sum over b = 1..HH of (P_N(b) (level_b^2 - level_(b-1)^2) - 2 P_S(b) (level_b - level_(b-1))).
// N and S of the whole sides are known from the statistics; the sum over the boundaries is a sum over the blocks, which they add up
// in 64-bit integers (any order, the same bits) with the unit 2^-fix.  It is below 2^62 units: the sides together come to less than
// 4 n E^2, E the power of two above the widest clip and every level.  A block's rounding to a unit is 2^-60 of that bound.
__device__ __forceinline__ int ss_fix(uint64_t n, int e) { return 60 - (64 - __clzll((long long)n)) - 2 * e; }
template <int HH>
__device__ __forceinline__ void ss_errors(const SsPlan<HH>& p, int ncand, int ni, int rs, int fix, unsigned char* raw, const int* pos,
                                          const float4* s_cand, const int* s_valid, unsigned long long* acc)
{
    constexpr int TPC = HH == 1 ? 2 : 4, RUN = (2 * HH + TPC - 1) / TPC;     // threads per candidate: one or two per side
    const double unit = ss_two_to(fix);
    for (int w0 = threadIdx.x & ~31; w0 < ncand * TPC; w0 += SS_THREADS) {
        const int w = w0 + (threadIdx.x & 31), k = w / TPC, part = w % TPC;
        const int side = part / (TPC / 2), b0 = 1 + (part % (TPC / 2)) * RUN;
        double v = 0.0;
        if (k < ncand && s_valid[k]) {
            const float4 c = s_cand[k];
            auto level = [&](int b) { const double l = ss_level(c, side ? HH - b : HH + 1 + b, p.m); return side ? -l : l; };
            double below = level(b0 - 1);
#pragma unroll
            for (int j = 0; j < RUN; ++j) {
                const int b = b0 + j;
                if (b > HH) break;
                const ulonglong2 P = *ss_slot(raw, side * ni + pos[k * HH + b - 1], rs);
                const double lv = level(b), step = lv - below;
                v += step * (2.0 * p.u * (double)P.y - (lv + below) * (double)P.x);
                below = lv;
            }
        }
        __syncwarp();
#pragma unroll
        for (int o = TPC / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
        if (k < ncand && part == 0) atomicAdd(acc + k, (unsigned long long)__double2ll_rn(v * unit));
    }
}

// What the finish needs of the hard form: levels of the codes that hold the elements beyond the ends, their sums.
struct SsBeyond { const double *lv_lo, *lv_hi; double e_lo, e_hi; };

// Every block, when the sums are complete: the error of every candidate into s_curve, the first minimum as the result (every block the
// same).  A thread per candidate, a warp's minimum by shuffles, the warps' through s_min, s_at [SS_WARPS].
template <int HH>
__device__ __forceinline__ int ss_finish(const SsArgs& a, float m, bool flat, const qp_stats_t& st, double n_up, double n_down, int ncand, int fix,
                                         const float4* s_cand, const int* s_valid, double* s_curve, const SsBeyond* hard, double* s_min, int* s_at)
{
    static_assert(QP_SS_MAX_CAND <= SS_THREADS, "a thread per candidate");
    const double inf = __longlong_as_double(0x7FF0000000000000ll);
    const int k = threadIdx.x, lane = threadIdx.x & 31, warps = (ncand + 31) >> 5;
    if ((k >> 5) < warps) {
        const double nf = (double)(st.n - st.nonfinite), dm = st.mean - (double)m;
        const double s_abs = nf * st.mad + dm * (n_up - n_down);              // sum |y|, sum y: the sides are half sum and half difference
        const double s_sq = nf * (st.var + dm * dm);
        const double s_up = 0.5 * (s_abs + nf * dm), s_down = 0.5 * (s_abs - nf * dm);
        double best = inf;
        if (k < ncand) {
            double v = HH || hard ? (double)(long long)__ldcg(a.acc + k) * ss_two_to(-fix) : 0.0;
            if (hard) {
                v -= 2.0 * (hard->lv_lo[k] * hard->e_lo + hard->lv_hi[k] * hard->e_hi);
            } else {
                const int top = flat ? 0 : HH;                // (flat: everything has the first code of its side)
                const double lu = ss_level(s_cand[k], HH + 1 + top, m), ld = -ss_level(s_cand[k], HH - top, m);
                v += n_up * lu * lu - 2.0 * lu * s_up + (n_down * ld * ld - 2.0 * ld * s_down);
            }
            v = !s_valid[k] ? inf : (nf > 0.0 ? (s_sq + v) / nf : 0.0);
            s_curve[k] = v;
            if (v < best) best = v;
        }
        __syncwarp();
        int at = best < inf ? k : 1 << 30;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const double ov = __shfl_xor_sync(0xFFFFFFFFu, best, o);
            const int ok = __shfl_xor_sync(0xFFFFFFFFu, at, o);
            if (ov < best || (ov == best && ok < at)) { best = ov; at = ok; }
        }
        if (lane == 0) { s_min[k >> 5] = best; s_at[k >> 5] = at; }
    }
    __syncthreads();
    double best = inf;
    int at = 0;                                               // (every error infinite or NaN: keep b_E)
    for (int w = 0; w < warps; ++w)
        if (s_min[w] < best) { best = s_min[w]; at = s_at[w]; }
    return at;
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
// Exclusive prefix sums of n[0..len), s[0..len) (n[len], s[len]: the totals); sh: 2 * SS_WARPS doubles.
__device__ inline void ss_scan(double* n, double* s, int len, double* sh)
{
    const int t = threadIdx.x, per = (len + SS_THREADS - 1) / SS_THREADS;
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
    if (t == SS_THREADS - 1) { n[len] = xa; s[len] = xb; }
    __syncthreads();
}
// This block's part of the errors, as ss_errors; lv_lo, lv_hi [ncand]: levels of the codes of the two ends.  Returns fix.
__device__ inline int ss_hard_errors(const SsArgs& a, const SsHard& h, float m, int ncand, const ulonglong2* row, const float4* s_cand,
                                     const int* s_valid, double* lv_lo, double* lv_hi, double* sh)
{
    // (behind the thresholds: the tables are done with)
    double* PN = reinterpret_cast<double*>(reinterpret_cast<unsigned char*>(h.thr) + ((size_t)8 * h.M + 15) / 16 * 16);
    double* PS = PN + (h.M + 2);
    for (int i = threadIdx.x; i <= h.M; i += SS_THREADS) {
        const ulonglong2 t = row[i];
        PN[i] = (double)t.x;
        PS[i] = (double)t.x * ((double)h.g_lo - (double)m) + h.u * (double)t.y;
    }
    __syncthreads();
    ss_scan(PN, PS, h.M + 1, sh);
    const double most = fmax(fabs((double)h.g_lo - (double)m), fabs((double)h.g_hi - (double)m));   // of levels and elements
    int e = 0;
    frexp(most, &e);
    const int fix = ss_fix(a.n, e);
    const double unit = most < __longlong_as_double(0x7FF0000000000000ll) ? ldexp(1.0, fix) : 0.0;
    const int L1 = (1 << a.bits) - 1;
    for (int k = threadIdx.x; k < ncand; k += SS_THREADS) {
        double t = 0.0;
        int p0 = 0;
        lv_lo[k] = lv_hi[k] = 0.0;
        for (int j = 0; s_valid[k] && j <= L1; ++j) {
            int p1 = h.M + 1;
            if (j < L1) {
                const float T = h.thr[k * L1 + j];
                if (T < __int_as_float(0x7F800000)) p1 = max(ss_hard_at(h, T), p0);
            }
            const double lv = ss_level(s_cand[k], j, m);
            if (p0 == 0 && p1 > 0) lv_lo[k] = lv;
            if (p1 == h.M + 1 && p0 < h.M + 1) lv_hi[k] = lv;
            t += (PN[p1] - PN[p0]) * lv * lv - 2.0 * lv * (PS[p1] - PS[p0]);
            p0 = p1;
        }
        // (ends that are not finite: the levels carry the infinity into the curve)
        if (unit > 0.0 && fabs(t) < 1e300) atomicAdd(a.acc + k, (unsigned long long)__double2ll_rn(t * unit));
        else lv_lo[k] = lv_hi[k] = __longlong_as_double(0x7FF8000000000000ll);
    }
    return fix;
}

__host__ __device__ constexpr int ss_ctile(int hh) { return hh >= 3 ? 512 : 1024; }   // phase C's tile: long code per element, short tile (instruction cache)

// What the last block out does, with what count_out returned (and whether the block itself gave up): one thread.
__device__ __forceinline__ void ss_out(const SsArgs& a, unsigned before)
{
    if (!qp_grid::last_out(before, gridDim.x)) return;
    if (before >= qp_grid::GAVE_UP && !(a.bits && !a.st_in)) {        // (block 0 of an undisturbed launch has cleaned)
        for (int b = 0; b < a.nb; ++b) a.hist[b] = 0ull;
        if (a.bits)
            for (int k = 0; k < a.steps + 3; ++k) a.acc[k] = 0ull;
    }
    qp_grid::reset(a.bar);
}

// STATS: phases A and B (otherwise the statistics come with st_in, and B runs only if they lack the histogram).
// HH: code boundaries above the centre, 2^bits / 2 - 1; -1: statistics only.
// Returns SS_GAVE_UP where a wait ran out, SS_OUT where the block has counted itself out (or is one of a cluster).
enum { SS_GAVE_UP, SS_DONE, SS_OUT };
template <typename T, bool STATS, int HH>
__device__ __forceinline__ int ss_run(const SsArgs& a)
{
    constexpr bool SEARCH = HH >= 0;
    constexpr int H = SEARCH ? HH : 0;
    extern __shared__ __align__(16) unsigned char raw[];
    __shared__ SsBlock s_block[2];
    __shared__ SsRows s_rows[STATS ? 4 : 1];
    __shared__ __align__(16) double s_red[SS_WARPS * 2];
    __shared__ int s_ok;
    __shared__ bool s_last;
    __shared__ qp_stats_t s_st;
    __shared__ double s_down;                                 // elements below the fp32 mean
    __shared__ qp_ds_setup s_setup;
    __shared__ SsPlan<H> s_plan;
    const T* x = static_cast<const T*>(a.x);
    const int lane = threadIdx.x & 31;
    const unsigned G = gridDim.x;
    const uint64_t step = (uint64_t)G * SS_WARPS, first = ss_first_tile(a.ntiles, step);
    const uint64_t tail0 = a.ntiles * SS_TILE;
    unsigned* bins = reinterpret_cast<unsigned*>(raw + SS_TABLE_BYTES);
    uint4* part = a.part + blockIdx.x;                        // this block's: row r at part[r * G]
    const bool cluster = a.cluster;
    // this block's partial into row r, by warp 0, and every block's rows r and r + 1 (behind a barrier; the statistics alone have none
    // behind phase B)
    auto pushed = [&](int r) { return cluster && (SEARCH || r < 2); };
    auto put = [&](int r, const uint4& v) {
        if (pushed(r)) ss_push(s_rows[r], G, v);
        else if (lane == 0) part[r * G] = v;
    };
    auto merge2 = [&](int r, auto&& take) {
        if (pushed(r)) ss_merge_pushed<2>(s_rows + r, G, take);
        else ss_merge<2>(a.part + r * G, G, take);
    };
    // (a block's shared memory may be written from outside once the block runs: the wait is in front of the first push)
    if (STATS && cluster) qp_grid::cluster_arrive();
    SsTail tail;
    tail.load(x, tail0, a.n, blockIdx.x == G - 1);
    unsigned waits = 0;
    auto meet = [&]() {
        if (cluster) {
            qp_grid::cluster_arrive();
            qp_grid::cluster_wait();
            return true;
        }
        ++waits;
        return qp_grid::barrier(a.bar, qp_grid::target(waits, G, a.bar_extra), a.spin_limit, a.status, &s_ok);
    };
    // for what warp 0 wrote and reads next; the others learn from s_ok behind the next block barrier
    auto meet_warp0 = [&]() {
        ++waits;
        if (cluster) {
            qp_grid::cluster_arrive();
            qp_grid::cluster_wait();
            if (threadIdx.x == 0) s_ok = 1;
            __syncwarp();
        } else if (threadIdx.x < 32) {
            qp_grid::barrier_warp0(a.bar, qp_grid::target(waits, G, a.bar_extra), a.spin_limit, a.status, &s_ok);
        }
    };
    auto empty = [&](int t, int threads) {                    // the tables, by threads t = 0 .. threads - 1
        for (int i = t; i < ((a.nb + 1) << a.hist_shift); i += threads) bins[i] = 0u;
        if constexpr (H > 0) {                                // (2 ni words << rep_shift are a multiple of 16 bytes)
            const int vecs = (SS_GRID + 1 + H * (a.steps + 1)) << a.rep_shift >> 1;
            for (int i = t; i < vecs; i += threads)
                reinterpret_cast<uint4*>(raw)[i] = reinterpret_cast<uint4*>(raw + SS_SUMS_AT)[i] = make_uint4(0u, 0u, 0u, 0u);
        }
    };

    // ---- phase A
    if constexpr (STATS) {
        if (SEARCH && blockIdx.x == 0) {                      // (their first use is behind the barrier)
            for (int k = threadIdx.x; k <= a.steps; k += SS_THREADS) a.acc[k] = 0ull;
            for (int b = threadIdx.x; b < a.nb; b += SS_THREADS) a.hist[b] = 0ull;
        }
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
        tail.each([&](float v) { acc.one(v); });
        if (cluster) qp_grid::cluster_wait();
        const SsParts v = ss_block_parts<true>({acc.s, acc.sa, acc.mn, acc.mx, acc.bad}, s_block[0]);
        if (threadIdx.x < 32) {
            put(0, ss_row(v.a, v.b));
            put(1, make_uint4(__float_as_uint(v.lo), __float_as_uint(v.hi), v.count, 0u));
        }
        if (threadIdx.x >= 32) empty(threadIdx.x - 32, SS_THREADS - 32);          // while warp 0 waits and merges
        meet_warp0();
        if (threadIdx.x < 32) {
            double s = 0.0, sa = 0.0, bad = 0.0;
            float mn = __int_as_float(0x7F800000), mx = -mn;
            merge2(0, [&](const uint4 (&p)[2]) {
                s += ss_row_first(p[0]);
                sa += ss_row_second(p[0]);
                mn = fminf(mn, __uint_as_float(p[1].x));
                mx = fmaxf(mx, __uint_as_float(p[1].y));
                bad += (double)p[1].z;                        // exact: counts are far below 2^53
            });
            __syncwarp();
            s = ss_pair_sum(s, sa);
            mn = ss_pair_min(mn, -mx);
            bad = ss_pair_sum(bad, 0.0);
            sa = __shfl_sync(0xFFFFFFFFu, s, 16);
            mx = -__shfl_sync(0xFFFFFFFFu, mn, 16);
            if (lane == 0) {
                const unsigned long long nbad = (unsigned long long)bad, nf = a.n - nbad;
                s_st.n = a.n;
                s_st.nonfinite = nbad;
                s_st.mean = nf ? s / (double)nf : 0.0;
                s_st.mean_abs = nf ? sa / (double)nf : 0.0;
                s_st.min = nf ? (double)mn : 0.0;
                s_st.max = nf ? (double)mx : 0.0;
                s_st.mad = s_st.var = 0.0;
                s_st.hist_peak = 0;
                s_st.hist_bins = 0;
                s_st.reserved = 0;
            }
        }
        __syncthreads();
        if (!s_ok) return SS_GAVE_UP;
    } else {
        empty(threadIdx.x, SS_THREADS);
        if (threadIdx.x == 0) s_st = *a.st_in;
        __syncthreads();
    }

    // ---- phase B
    const bool guard = s_st.nonfinite != 0;
    const bool counting = STATS || (!a.promised && s_st.hist_bins != a.nb);
    if (counting) {
        const bool hist_on = s_st.max > s_st.min;
        SsParts v = {0.0, 0.0, 0.f, 0.f, 0u};
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
            tail.each([&](float x) { d.one(x); });
            v = ss_block_parts<false>({d.sd[0] + d.sd[1], d.sv[0] + d.sv[1], 0.f, 0.f, d.below}, s_block[1]);   // (its barrier orders the counters)
            if (STATS && threadIdx.x < 32) {
                put(2, ss_row(v.a, v.b));
                put(3, make_uint4(v.count, 0u, 0u, 0u));
            }
        }
        if (hist_on) ss_hist_out(bins, a.nb, a.hist_shift, a.hist);
        if constexpr (SEARCH) {
            __syncthreads();
            meet_warp0();
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
            double sd = 0.0, sv = 0.0, below = 0.0, peak = 0.0;
            unsigned long long c[4];
            QP_LATE(SEARCH && G > 1 && blockIdx.x == G - 1);
#pragma unroll
            for (int u = 0; u < 4; ++u) c[u] = hist_on && lane + 32 * u < a.nb ? __ldcg(&a.hist[lane + 32 * u]) : 0ull;
            if (STATS)
                merge2(2, [&](const uint4 (&p)[2]) {
                    sd += ss_row_first(p[0]);
                    sv += ss_row_second(p[0]);
                    below += (double)p[1].x;
                });
#pragma unroll
            for (int u = 0; u < 4; ++u) peak = fmax(peak, (double)c[u]);
            if (hist_on)
                for (int b = lane + 128; b < a.nb; b += 32) peak = fmax(peak, (double)__ldcg(&a.hist[b]));
            __syncwarp();
            if (STATS) {
                sd = ss_pair_sum(sd, sv);
                below = ss_pair_sum(below, 0.0);
                sv = __shfl_sync(0xFFFFFFFFu, sd, 16);
            }
            for (int o = 16; o > 0; o >>= 1) peak = fmax(peak, __shfl_xor_sync(0xFFFFFFFFu, peak, o));
            if (lane == 0) {
                if (STATS) {
                    const double nf = (double)(a.n - s_st.nonfinite), dm = s_st.mean - (double)(float)s_st.mean;
                    s_st.mad = nf > 0.0 ? fmax(0.0, sd - dm * (nf - 2.0 * below)) / nf : 0.0;
                    s_st.var = nf > 0.0 ? fmax(0.0, sv / nf - dm * dm) : 0.0;
                    s_down = below;
                }
                s_st.hist_peak = (unsigned long long)peak;
                s_st.hist_bins = a.nb;
                if (!SEARCH) {                                // (the sender's go out with its result, behind its last barrier)
                    *a.st_out = s_st;
                    if (s_st.nonfinite) atomicOr(a.status, QP_DEV_NONFINITE);
                }
            }
        }
        __syncthreads();
        if constexpr (!SEARCH) {
            for (int b = threadIdx.x; b < a.nb; b += SS_THREADS) a.hist[b] = 0ull;
            if (threadIdx.x == 0) qp_grid::reset(a.bar);
            return SS_OUT;
        } else if (!s_ok) {
            return SS_GAVE_UP;
        }
    }

    // ---- phase C
    if constexpr (SEARCH) {
        constexpr int BITS = H == 0 ? 1 : H == 1 ? 2 : H == 3 ? 3 : 4;
        const int ncand = a.steps + 1, ni = SS_GRID + 1 + H * ncand;
        __shared__ float4 s_cand[QP_SS_MAX_CAND];
        __shared__ int s_valid[QP_SS_MAX_CAND];
        __shared__ double s_curve[QP_SS_MAX_CAND];
        __shared__ int s_edge[SS_GRID + 2];                   // interval that a grid cell starts with, and one that there is not
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
        const bool hard = s_plan.hard, flat = !(s_plan.inv_e > 0.f);
        int* pos = reinterpret_cast<int*>(bins);              // [ncand][H], or the hard form's levels [2][ncand]: the histogram is out
        double* lv = reinterpret_cast<double*>(bins);
        int fix = ss_fix(a.n, 127 - (int)(__float_as_uint(s_plan.inv_e) >> 23));  // (1 / E is a power of two)
        if constexpr (H == 0) {
            // one bit: a side has one code, and the statistics say what its elements come to; how many they are is the
            // one thing that the caller's statistics do not say
            if constexpr (!STATS) {
                const SsPlan<H> p = s_plan;
                SsSides f = {p.m, guard, 0u, 0u};
                SsTiles<T, SS_TILE>::template run<false>(x, a.ntiles, first, step, lane, f);
                tail.each([&](float x) { f.one(x); });
                const SsParts v = ss_block_parts<false>({(double)f.all, 0.0, 0.f, 0.f, f.down}, s_block[0]);
                if (threadIdx.x == 0) {
                    atomicAdd(a.acc + ncand, (unsigned long long)v.count);
                    atomicAdd(a.acc + ncand + 1, (unsigned long long)v.a - v.count);
                }
            }
        } else if (!hard) {
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
                    ss_flush(raw, ni, a.rep_shift, row, t0 == per);
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
            tail.each([&](float v) {
                if (qp_is_finite(v)) ss_count<H>(p, tb, v);
            });
            ss_places<H>(s_plan, ncand, ni, s_edge, pos);
            __syncthreads();
            const uint2 sides = ss_prefix(raw, ni, a.rep_shift, ntiles > per ? row : nullptr, s_edge, reinterpret_cast<ulonglong2*>(s_red));
            __syncthreads();
            if (!flat) ss_errors<H>(s_plan, ncand, ni, a.rep_shift, fix, raw, pos, s_cand, s_valid, a.acc);
            if (!STATS && threadIdx.x == 0) {
                atomicAdd(a.acc + ncand, (unsigned long long)sides.y);
                atomicAdd(a.acc + ncand + 1, (unsigned long long)sides.x);
            }
        } else {
            SsHard h;
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
            tail.each([&](float x) { ss_hard_one(h, x, e2[0], e2[1]); });
            const SsParts e = ss_block_parts<false>({e2[0], e2[1], 0.f, 0.f, 0u}, s_block[0]);
            if (threadIdx.x == 0) part[0] = ss_row(e.a, e.b);         // (every block is done with the first rows)
            ss_hard_flush(h, row, fresh);
            __syncthreads();
            fix = ss_hard_errors(a, h, s_plan.m, ncand, row, s_cand, s_valid, lv, lv + ncand, s_red);
        }
        if constexpr (H > 0 || !STATS) {
            __syncthreads();
            if (!a.packed && blockIdx.x != 0) {               // nobody waits for the result but block 0
                if (cluster) {
                    qp_grid::cluster_arrive();
                    qp_grid::cluster_wait();
                } else if (threadIdx.x == 0) {
                    qp_grid::arrive_release(a.bar);
                    __threadfence();                          // (the arrival, which nobody here polls for)
                }
                return SS_DONE;
            }
            if (!meet()) return SS_GAVE_UP;
        }
        SsBeyond beyond = {lv, lv + ncand, 0.0, 0.0};
        if (hard && H > 0) {
            if (threadIdx.x < 32) {
                ss_merge<1>(a.part, G, [&](const uint4 (&p)[1]) {
                    beyond.e_lo += ss_row_first(p[0]);
                    beyond.e_hi += ss_row_second(p[0]);
                });
                __syncwarp();
                const double e = ss_pair_sum(beyond.e_lo, beyond.e_hi);
                if ((lane & 15) == 0) s_red[lane >> 4] = e;
            }
            __syncthreads();
            beyond.e_lo = s_red[0];
            beyond.e_hi = s_red[1];
        }
        const double down = STATS ? s_down : (double)__ldcg(a.acc + ncand);
        const double up = STATS ? (double)(s_st.n - s_st.nonfinite) - down : (double)__ldcg(a.acc + ncand + 1);
        const int best = ss_finish<H>(a, s_plan.m, flat, s_st, up, down, ncand, fix, s_cand, s_valid, s_curve, hard && H > 0 ? &beyond : nullptr,
                                      s_block[0].sum, reinterpret_cast<int*>(s_block[0].count));
        if (blockIdx.x == 0) {
            if (threadIdx.x == SS_THREADS - 32) {             // (a warp that has a tile less to pack than the first, or none)
                qp_ds_write_result(best, s_curve, s_setup, a.steps, a.nb, BITS, s_cand[best], a.ds_out, a.qp_out, a.status);
                *a.setup = s_setup;
            }
            if (STATS && threadIdx.x == SS_THREADS - 64) {
                *a.st_out = s_st;
                if (s_st.nonfinite) atomicOr(a.status, QP_DEV_NONFINITE);
            }
            for (int k = threadIdx.x; k < ncand; k += SS_THREADS) {
                a.curve[k] = s_curve[k];
                a.cand[k] = s_cand[k];
                a.valid[k] = s_valid[k];
            }
            if constexpr (!STATS) {                           // (nobody needs them any more: every block has arrived since)
                for (int b = threadIdx.x; b < a.nb; b += SS_THREADS) a.hist[b] = 0ull;
                for (int k = threadIdx.x; k < ncand + 2; k += SS_THREADS) a.acc[k] = 0ull;
            }
        }
        if (!a.packed && !cluster && threadIdx.x == SS_THREADS - 1) ss_out(a, qp_grid::count_out(a.bar));
        if constexpr (!STATS) return SS_OUT;
        if constexpr (STATS) {                                // the sender: everybody packs, from the tensor's end
            const float4 q = s_cand[best];
            uint32_t* sw = reinterpret_cast<uint32_t*>(raw) + (threadIdx.x >> 5) * 256;
            const uint64_t tiles = (a.n + QP_TILE - 1) / QP_TILE;
            for (uint64_t it = first; it < tiles; it += step)
                qp_pack_tile<BITS, T, true>(x, a.n, tiles - 1 - it, lane, q.x, q.y, q.w, a.packed, a.nwords, sw);
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
                  (size_t)ctx->sm_count * 4 * sizeof(uint4) <= sizeof(qp_stats_partial) * QP_MAX_BLOCKS &&
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
// from 8 tiles on, at 4 bits from 128 KB: 8.4 to 17.2 us by width up to 2^20 elements, where the candidates scored one by one take 23 us at
// 2^15, 36 at 2^18 and 62 at 2^20.  Below 128 KB the statistics carry no histogram and the launch counts it as well: fp32 of 8192 to
// 32760 elements 13 to 15 us at 1 bit, 16 to 18 at 2, 17 to 19 at 3 and 19 to 21 at 4, against 25 to 27.  (The line at 4 bits was drawn
// when the launch took 33 us there.)  At 1..4 bits (each further code boundary costs two instructions per element: at 5 bits and up the
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
    static_assert(QP_SS_MAX_CAND * 7 * sizeof(int) <= SS_HIST_BYTES && QP_SS_MAX_CAND * 2 * sizeof(double) <= SS_HIST_BYTES, "the histogram's room is used again");
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
    a.part = reinterpret_cast<uint4*>(ctx->d_part);
    unsigned char* f = static_cast<unsigned char*>(ctx->d_fused);
    a.bar = reinterpret_cast<unsigned*>(f) + 16;              // words 16, 17 (the sender uses 0, 1, the statistics 8..10 and 24, 25)
    a.hist = reinterpret_cast<unsigned long long*>(f + (bits && !st_in ? QP_FUSED_SENDER_HIST_AT : 256));
    a.acc = reinterpret_cast<unsigned long long*>(f + QP_FUSED_TOTALS_AT) + (st_in ? QP_SS_MAX_CAND + 2 : 0);
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
    a.cluster = qp_cluster_wanted(ctx, ctx->ss_cluster, n);
    const unsigned G = qp_together_blocks(ctx, a.cluster, a.ntiles);
    void* k = dtype == QP_F32 ? ss_kernel<float>(st_in == nullptr, bits) : ss_kernel<unsigned short>(st_in == nullptr, bits);
    void* params[] = {&a};
    if (qp_launch_together(k, G, SS_THREADS, params, SS_DYN_BYTES, a.cluster, s) != cudaSuccess)
        return qp_check_launch(ctx, "statistics and search (cooperative launch)");
    ctx->launches += 1;
    return qp_check_launch(ctx, "statistics and search");
}
