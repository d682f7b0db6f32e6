// The candidates' partition of the directed search without a table of thresholds.
//
// The candidates' clip half-widths are a_k = a_0 + k d, so the thresholds of one code boundary i above the centre are the
// equally spaced points c_i a_k, and the number of them at or below |x - mean| is a clamped affine function of it:
// floor(K sat(A_i |y| + B_i)), two instructions.  The sum over the boundaries of one side, plus the cell of a uniform grid of
// 64 cells, numbers the intervals of the merged partition of that side.  Where a threshold really lies differs from that
// formula by the rounding of the clip ends, s ~ 1e-7 of the clip: an element between the two is exchanged between two codes
// whose reconstruction errors differ by less than 2 s, so a candidate's error moves by 12 (s / step)^2 relative (below 1e-8).
// Where the clip ends are coarse against the step (|mean| beyond 250 steps) the plan says `hard`, and the caller takes the exact
// thresholds or scores every candidate instead.
//
// Per element: 1 is added to the interval's count and d to its sum by two 32-bit shared-memory atomics, d = the
// offset from the grid cell's left edge.  The grid spans a power of two E above the widest clip, a cell is E / 2^6 and
// d counts units of cell / 2^ub; at ub = 19 d is exact for |y| >= E / 4 and rounded to half a unit below (which counts 2 level
// times in an element's squared error; the roundings of different elements are independent).
#pragma once

#include "qp_internal.cuh"

constexpr int SS_GRID = 64;                       // uniform cells per side
constexpr unsigned SS_ONE = 0x4B000000u;          // bits of 2^23: an integer sits in the low mantissa bits
constexpr float SS_MAGIC = 8388608.0f;
constexpr int SS_SUMS_AT = 100 * 1024;            // bytes from an interval's count to its sum in shared memory

// whether (x - min) * inv_w is a number for every x of [min, max]
__device__ __forceinline__ bool ss_range_fits(const qp_stats_t& st, float inv_w)
{
    return st.max - st.min <= 3.4028234663852886e38 && inv_w < __int_as_float(0x7F800000);
}

// 2^k as fp64, k from -1022 to 1023
__device__ __forceinline__ double ss_two_to(int k) { return __hiloint2double((k + 1023) << 20, 0); }

template <int HH>
struct SsPlan {
    float m;                                                  // fp32 mean; y = x - m
    float inv_e, cell;                                        // 1 / E; width of a grid cell E / 64: powers of two
    float kf;                                                 // number of candidates
    float span[HH ? HH : 1];                                  // 1 / A
    float A[HH ? HH : 1], B[HH ? HH : 1];                     // boundary i: thresholds passed / K = sat(A_i |y| + B_i)
    double u, w;
    int ncand, down, hard;                                    // down: the half-widths fall with k
};

// i = -1: the common part; i = 0 .. HH - 1: boundary i (each by a thread of its own).  mean, a0, a1: centre and half-widths of
// the first and the last valid candidate.
template <int HH>
__device__ inline void ss_make_plan(SsPlan<HH>& p, int i, double mean, double a0, double a1, int ncand, int bits, int ub)
{
    const double a_min = fmin(a0, a1), R = fmax(a0, a1), L1 = (double)((1 << bits) - 1);
    const bool any = R > 1e-30 && R < 1e30;
    if (i < 0) {
        const int e = any ? (int)((unsigned)__double2hiint(R) >> 20) - 1022 : 0;            // R < 2^e, a normal number
        p.m = (float)mean;
        p.ncand = ncand;
        p.kf = (float)ncand;
        p.down = a1 < a0;
        p.inv_e = any ? (float)ss_two_to(-e) : 0.f;
        p.w = any ? ss_two_to(e - 6) : 0.0;
        p.cell = (float)p.w;
        p.u = any ? ss_two_to(e - 6 - ub) : 1.0;
        // clip ends that are coarse against the smallest step (an ulp of the mean beyond 2^-15 of it, where a candidate's
        // error would move by 1e-8), or clips beyond what the formula's fp32 constants hold: the exact thresholds
        p.hard = HH > 0 && R > 0.0 && (!any || fabs(mean) * 1.1920928955078125e-7 > 3.0517578125e-5 * (2.0 * a_min / L1));
    } else if (i < HH) {
        const double c = 2.0 * (i + 1) / L1, t0 = c * a_min;
        const double gap = ncand > 1 ? c * (R - a_min) / (double)(ncand - 1) : 0.0;
        // thresholds t0 + q gap, q = 0 .. K - 1.  (Candidates closer together than 1e-6 of the clip are spread
        // that far: it moves a threshold by less than its element's share of the error can show.)
        const double span = fmax((double)ncand * gap, 1e-6 * c * R);
        p.A[i] = any ? (float)(1.0 / span) : 0.f;
        p.B[i] = any ? (float)(1.0 / (double)ncand - t0 / span) : 0.f;
        p.span[i] = (float)span;
    }
}

// |y| is clamped to E by the saturating product t = |y| / E, exact because E is a power of two; d = t as an integer in
// units of 2^-(6 + ub) (the conversion pipe is idle otherwise), less the grid cell's.  What lies beyond E counts in the last interval
// of its side, whose sum is not used: the sum over a whole side is known from the statistics.
// base of the table: byte address of this lane's replica of interval 0 of the upper side; the lower side
// follows `half` bytes later; the sums are SS_SUMS_AT bytes behind the counts.
// mul: bytes between intervals; scale = 2^(6 + ub).
struct SsTable { unsigned mul, base, half, ni, ub; float scale; };
template <int HH>
__device__ __forceinline__ void ss_count(const SsPlan<HH>& p, const SsTable& tb, float x)
{
    const float y = __fsub_rn(x, p.m), a = fabsf(y);
    const float t = __saturatef(__fmul_rn(a, p.inv_e));
    const float g = __fmaf_rd(t, (float)SS_GRID, SS_MAGIC);   // grid cell, then interval number, in the low bits
    float r = g;
#pragma unroll
    for (int i = 0; i < HH; ++i) r = __fmaf_rd(__saturatef(fmaf(a, p.A[i], p.B[i])), p.kf, r);
    const unsigned d = __float2uint_rn(__fmul_rn(t, tb.scale)) - (__float_as_uint(g) << tb.ub);
    unsigned addr = (QP_CK(__float_as_uint(r) - SS_ONE, tb.ni) + SS_ONE) * tb.mul + tb.base;
    addr += (__float_as_uint(y) >> 31) * tb.half;
    asm volatile("red.shared.add.u32 [%0], 1;" ::"r"(addr) : "memory");
    asm volatile("red.shared.add.u32 [%0+%2], %1;" ::"r"(addr), "r"(d), "n"(SS_SUMS_AT) : "memory");
}
// interval that x on a side belongs to, as ss_count numbers it
template <int HH>
__device__ __forceinline__ int ss_interval(const SsPlan<HH>& p, float x)
{
    float r = __fmaf_rd(__saturatef(__fmul_rn(x, p.inv_e)), (float)SS_GRID, SS_MAGIC);
#pragma unroll
    for (int i = 0; i < HH; ++i) r = __fmaf_rd(__saturatef(fmaf(x, p.A[i], p.B[i])), p.kf, r);
    return (int)(__float_as_uint(r) - SS_ONE);
}
// first interval of code b (1..HH) of candidate k on a side: the interval of its threshold, in which the thresholds of
// its own boundary, counted exactly, take the place of the formula's (which may be one off at the threshold itself)
template <int HH>
__device__ __forceinline__ int ss_place(const SsPlan<HH>& p, int k, int b)
{
    const int q = p.down ? p.ncand - 1 - k : k;
    const float A = p.A[b - 1], B = p.B[b - 1];
    const float T = ((float)(q + 1) * (1.0f / p.kf) - B) * p.span[b - 1];
    const int own = (int)(__float_as_uint(__fmaf_rd(__saturatef(fmaf(T, A, B)), p.kf, SS_MAGIC)) - SS_ONE);
    return ss_interval(p, T) - own + q + 1;
}
// interval that grid cell g starts with
template <int HH>
__device__ __forceinline__ int ss_cell_start(const SsPlan<HH>& p, int g)
{
    return g ? g + ss_interval(p, (float)g * p.cell) - (int)(__float_as_uint(__fmaf_rd(__saturatef(__fmul_rn((float)g * p.cell, p.inv_e)), (float)SS_GRID, SS_MAGIC)) - SS_ONE) : 0;
}
__device__ __forceinline__ double ss_level(const float4& q, int j, float m)   // reconstruction of code j, relative to m
{
    return (double)fmaf((float)j, q.z, q.x) - (double)m;
}
