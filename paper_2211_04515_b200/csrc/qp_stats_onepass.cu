// Statistics (paper Sec. 3), and in the sender with a closed-form clip the clip and the packing as well: one cooperative
// launch, one block of 16 independent warps per SM.  Two forms, chosen by the tensor's size.
//
// Two passes, while L2 still holds the tensor when the second one comes (which walks it backwards): sum x, sum |x|, min and
// max; a grid barrier; sum |x - mean| and sum (x - mean)^2; a second barrier, and every block knows the clip and packs.
// What bounds it: L2 and the instructions, then the barriers.  27 M bf16 elements at 6 bits (54 MB), by block 0's time stamps: first pass
// 10.5 us, parts, barrier and merge 3.8, second pass 6.2, 2.5, clip 0.5, packing 9.6: 34, and 37 between launches.  One image at 8 bits (10
// blocks, a cluster): passes 0.9 and 1.1, the steps between them 2.2 and 1.9, clip 0.5, packing 1.2: 8.6, and 10.3 between launches.
// With the blocks' partials 64 bytes apart, every quantity in a reduction of its own and every thread adding up the warps' sums
// they took 40 and 12.3.  (Lanes that have parted take a shuffle one after another: a __syncwarp less in front of the
// reductions and the image takes 16.4.)
//
// One pass above that.  sum |x - mean| needs the mean first, so the deviations are taken about a pilot centre c, y = x - c,
// and the split point is moved to the mean afterwards: with D = mean - c > 0
//     sum |x - mean| = sum |y| + D (N(y < 0) - N(y >= 0)) + 2 sum over 0 <= y < D of (D - y),
// mirrored for D < 0.  The last sum is over the few elements between c and the mean: the elements within delta of c (six
// standard errors of the pilot, under half a per cent of a bell-shaped tensor) are counted and added up in cells of 1/64
// octave of |y|, so that every cell but the mean's own lies on a known side.  That one is taken as evenly filled, which is
// accepted where even the worst filling could not change the result by 1e-8; otherwise (and where the mean lies further
// than delta from c, or a cell's counter might have wrapped) the second pass runs after all.
// What bounds it: the read.  1 GiB of fp32, i.i.d. Laplace, by the blocks' time stamps: the pass 177 us in the fastest block and 185 in
// the slowest (5.8 TB/s), the pilot 7 (3 for its loads: 64 bytes per sample, one DRAM burst; 16-byte samples took 16), the two
// barriers and merges behind the pass 8, so 194 us in all, where two passes took 319.  Data whose mean lies off the density's
// peak has fewer elements in the window (channels of different means: 170 to 177 us).  fp32 of 134, 268 and 537 MB: 41, 62 and
// 102 us against 45, 82 and 157.
// The window must cost next to nothing: one test per four elements, and behind it one predicated look-up for the lane's hit
// (all elements through the look-up took 275 us on 1 GiB, four look-ups behind the test 221).
//
// Packing here rather than in a launch of its own: 5 to 10 us less (no clip launch, no gaps, and what L2 still holds is not
// read again), 2^24 fp32 at 2 bits 35 us against 44; 1 GiB at 8 bits 384 us against 394, of which the packing 173 in the fastest
// block and 185 in the slowest.  (384 in runs of some milliseconds; in longer ones the GPU draws 975 W and clocks at 1.85 instead
// of 1.97 GHz: 392 to 410 us.)
#include "qp_gridbar.cuh"
#include "qp_packtile.cuh"
#include "qp_tiles.cuh"

QP_CK_UNIT

namespace {

constexpr int OP_SAMPLE = 4;                       // most pilot vectors per thread
constexpr int OP_OCTAVES = 8;                      // octaves of |y| below delta that have cells of their own
constexpr int OP_CELLS = 64 * OP_OCTAVES + 1;      // per side; cell 0: what is below them
constexpr int OP_REPS = 3;                         // log2 of the lane replicas of a cell
constexpr unsigned OP_FULL = 65000u;               // most elements of a cell's replica: offsets of 16 bits add up to a word
constexpr uint64_t OP_ONE_MIN_BYTES_F32 = 96ull << 20, OP_ONE_MIN_BYTES_BF16 = 224ull << 20;   // tensors from which one pass is the faster form
constexpr float OP_MAGIC = 8388608.0f;
constexpr unsigned OP_ONE = 0x4B000000u;
constexpr size_t OP_DYN_BYTES = (size_t)(2 * OP_CELLS * 2 << OP_REPS) * sizeof(unsigned);   // >= 16 KB: the packer's staging
constexpr int OP_SUMS_AT = (int)(OP_DYN_BYTES / 2);

// rows of block partials: of the pass (sum y, |x|; min, max, non-finite, below c; sum |y|, y^2), of the pilot (two), of the window
// (two), of the second pass (a slow block may still read an earlier one's)
enum { OP_PASS = 0, OP_PILOT = 3, OP_WINDOW = 5, OP_SECOND = 7, OP_ROWS = 8 };

struct OpArgs {
    const void* x;
    uint64_t n, ntiles;                            // ntiles: whole tiles
    qp_stats_t* st_out;
    qp_qparams_t* qp_out;                          // sender: the quantizer, and
    uint32_t* packed;                              // the packed stream
    uint64_t nwords;
    int method, bmode;
    double F;
    int one;                                       // one pass, or two
    int sample;                                    // pilot vectors per thread
    uint4* part;                                   // [OP_ROWS][grid] block partials, 16 bytes each
    unsigned* bar;                                 // [0] arrivals, [1] blocks that have left; zero at entry and at exit
    unsigned* status;
    unsigned spin_limit, bar_extra;
    int cluster;                                   // the grid is one thread-block cluster
};

// Where sample i lies in its part, in 2^-32 of it: the fractional part of i^2 times the golden ratio.  (The squares of
// the integers times an irrational number are evenly spread, by Weyl's theorem; multiples of one would be too, but can fall into
// step with the channels.  On channel means of 192 to 4096 channels, 4000 tensors of 96 MB and more, the pilot's mean is off by 1.0
// standard errors in the root mean square and 3.9 at most, as with independent random places.)
__device__ __forceinline__ unsigned op_place(unsigned i) { return i * i * 2654435769u; }

// ONE: the pass about the pilot centre; otherwise the first of two passes (c = 0, no deviations and no window)
template <bool ONE>
struct OpPass {
    float c, delta, inv_u;                         // inv_u: 2^16 / delta
    int cell_off;                                  // |y|'s top bits less this: cell - 1
    unsigned mul, base, half;                      // window table of this lane, as byte addresses
    double sy, sa, sv, sx;                         // sum y, |y|, y^2, |x|
    float mn, mx;
    unsigned below, odd;
    qp_f2 nc, y2[2], v2[2];
    float a2[2], x2[2], lo, hi, w0, w1;
    __device__ __forceinline__ void begin()
    {
        y2[0] = y2[1] = v2[0] = v2[1] = 0ull;
        a2[0] = a2[1] = x2[0] = x2[1] = 0.f;
        lo = mn;
        hi = mx;
    }
    __device__ __forceinline__ void window(float y) const
    {
        const float a = fabsf(y);
        const int cell = min(max((int)(__float_as_uint(a) >> 17) - cell_off, 0), OP_CELLS - 1);
        const unsigned addr = (unsigned)QP_CK(cell, OP_CELLS) * mul + base + (__float_as_uint(y) >> 31) * half;
        const unsigned d = __float_as_uint(fmaf(a, inv_u, OP_MAGIC)) - OP_ONE;
        asm volatile("{ .reg .pred p; setp.lt.f32 p, %3, %4; @p red.shared.add.u32 [%0], 1; @p red.shared.add.u32 [%0+%2], %1; }"
                     ::"r"(addr), "r"(d), "n"(OP_SUMS_AT), "f"(a), "f"(delta) : "memory");
    }
    __device__ __forceinline__ void pair(float a, float b, int i)
    {
        if constexpr (!ONE) {
            y2[i & 1] = qp_add2(y2[i & 1], qp_pack2(a, b));
            x2[0] += fabsf(a);
            x2[1] += fabsf(b);
            lo = qp_min3(lo, a, b);
            hi = qp_max3(hi, a, b);
            return;
        }
        const qp_f2 y = qp_add2(qp_pack2(a, b), nc);
        float ya, yb;
        qp_unpack2(y, ya, yb);
        y2[i & 1] = qp_add2(y2[i & 1], y);
        v2[i & 1] = qp_fma2(y, y, v2[i & 1]);
        a2[0] += fabsf(ya);
        a2[1] += fabsf(yb);
        x2[0] += fabsf(a);
        x2[1] += fabsf(b);
        lo = qp_min3(lo, a, b);
        hi = qp_max3(hi, a, b);
        below += __float_as_uint(ya) >> 31;
        below += __float_as_uint(yb) >> 31;
        // four elements per test: outside the branch the window costs an instruction and a half per element
        if (i & 1) {
            if (fminf(qp_min3(fabsf(w0), fabsf(w1), fabsf(ya)), fabsf(yb)) < delta) {
                const bool h0 = fabsf(w0) < delta, h1 = fabsf(w1) < delta, h2 = fabsf(ya) < delta, h3 = fabsf(yb) < delta;
                window(h0 ? w0 : h1 ? w1 : h2 ? ya : yb);
                if ((h0 & h1) | ((h0 | h1) & h2) | ((h0 | h1 | h2) & h3)) {
                    if (h0 && h1) window(w1);
                    if ((h0 || h1) && h2) window(ya);
                    if ((h0 || h1 || h2) && h3) window(yb);
                }
            }
        } else {
            w0 = ya;
            w1 = yb;
        }
    }
    __device__ __forceinline__ void end()
    {
        const float psa = a2[0] + a2[1], psx = x2[0] + x2[1];
        if ((ONE ? psa : 0.f) + psx < __int_as_float(0x7F800000)) {        // every element finite (and no fp32 overflow)
            float u, v;
            qp_unpack2(qp_add2(y2[0], y2[1]), u, v);
            sy += (double)(u + v);
            if constexpr (ONE) {
                qp_unpack2(qp_add2(v2[0], v2[1]), u, v);
                sv += (double)(u + v);
                sa += (double)psa;
            }
            sx += (double)psx;
            mn = lo;
            mx = hi;
        } else {
            ++odd;
        }
    }
};
// element by element: a lane's share with non-finite values, and what is behind the last tile
struct OpOnes {
    double sy = 0.0, sa = 0.0, sv = 0.0, sx = 0.0;
    unsigned below = 0u, bad = 0u;
    float mn, mx;
    __device__ __forceinline__ void one(float v, float c)
    {
        if (!qp_is_finite(v)) { ++bad; return; }
        const double y = (double)__fsub_rn(v, c);
        sy += y;
        sa += fabs(y);
        sv += y * y;
        sx += (double)fabsf(v);
        below += y < 0.0 ? 1u : 0u;
        mn = fminf(mn, v);
        mx = fmaxf(mx, v);
    }
};
// the second pass, where it has to run: deviations about the mean itself
template <bool GUARD>
struct OpDeviations {
    qp_f2 nhi, nlo;
    double sd, sv;
    float a2[2];
    qp_f2 v2;
    __device__ __forceinline__ void begin()
    {
        a2[0] = a2[1] = 0.f;
        v2 = 0ull;
    }
    __device__ __forceinline__ void pair(float a, float b, int)
    {
        qp_f2 d = qp_add2(qp_add2(qp_pack2(a, b), nhi), nlo);
        float da, db;
        qp_unpack2(d, da, db);
        if (GUARD) {
            da = qp_is_finite(a) ? da : 0.f;
            db = qp_is_finite(b) ? db : 0.f;
            d = qp_pack2(da, db);
        }
        v2 = qp_fma2(d, d, v2);
        a2[0] += fabsf(da);
        a2[1] += fabsf(db);
    }
    __device__ __forceinline__ void end()
    {
        float u, v;
        qp_unpack2(v2, u, v);
        sd += (double)(a2[0] + a2[1]);
        sv += (double)(u + v);
    }
};

template <int N> struct Rows { static constexpr int value = N; };

// BITS = 0: statistics only; 1..8 and 16: the sender.
template <typename T, int BITS>
__global__ void __launch_bounds__(SS_THREADS, 1) stats_onepass_kernel(const OpArgs a)
{
    extern __shared__ __align__(16) unsigned char raw[];
    using Tiles = SsTiles<T, SS_TILE>;
    constexpr int EPV = Tiles::EPV;
    __shared__ SsBlock s_block[3];
    __shared__ SsRows s_rows[OP_ROWS];
    __shared__ int s_ok, s_full, s_again;
    __shared__ float s_c, s_delta;
    __shared__ double s_D, s_abs, s_below;
    __shared__ qp_stats_t s_st;
    __shared__ qp_qparams_t s_qp;
    const T* x = static_cast<const T*>(a.x);
    const int lane = threadIdx.x & 31;
    const unsigned G = gridDim.x;
    const uint64_t step = (uint64_t)G * SS_WARPS, first = ss_first_tile(a.ntiles, step);
    const uint64_t tail0 = a.ntiles * SS_TILE;
    // (16 bits an element take one pass from 224 MB on, which is beyond what the sender brings here: no pilot and no window in its code)
    const bool one = (sizeof(T) == 4 || BITS == 0) && a.one;
    const double inf = __longlong_as_double(0x7FF0000000000000ll);
    unsigned* table = reinterpret_cast<unsigned*>(raw);
    uint4* part = a.part + blockIdx.x;             // this block's: row r at part[r * G]
    unsigned waits = 0;
    // for what warp 0 wrote and merges next; the others wait at the block barrier behind, and learn from s_ok
    auto meet_warp0 = [&]() {
        ++waits;
        if (a.cluster) {
            qp_grid::cluster_arrive();
            qp_grid::cluster_wait();
            if (threadIdx.x == 0) s_ok = 1;
            __syncwarp();
        } else if (threadIdx.x < 32) {
            qp_grid::barrier_warp0(a.bar, qp_grid::target(waits, G, a.bar_extra), a.spin_limit, a.status, &s_ok);
        }
    };
    // this block's partial into row r, by warp 0, and every block's rows
    auto put = [&](int r, const uint4& v) {
        if (a.cluster) ss_push(s_rows[r], G, v);
        else if (lane == 0) part[r * G] = v;
    };
    auto merge = [&](auto rows, int r, auto&& take) {
        if (a.cluster) ss_merge_pushed<decltype(rows)::value>(s_rows + r, G, take);
        else ss_merge<decltype(rows)::value>(a.part + r * G, G, take);
    };
    // (a block's shared memory may be written from outside once the block runs: the wait is in front of the first push, and a
    // cluster's tensors never have a pilot)
    if (a.cluster) qp_grid::cluster_arrive();
    SsTail tail;
    tail.load(x, tail0, a.n, blockIdx.x == G - 1);
    auto leave = [&](unsigned gave_up) {
        if (threadIdx.x == 0 && qp_grid::last_out(qp_grid::count_out(a.bar, gave_up), G)) qp_grid::reset(a.bar);
    };
    if (one)                                                  // the window's table
        for (int i = threadIdx.x; i < (int)(OP_DYN_BYTES / 16); i += SS_THREADS) reinterpret_cast<uint4*>(raw)[i] = make_uint4(0u, 0u, 0u, 0u);
    if (threadIdx.x == 0) s_full = 0;

    // ---- pilot: sample i, four neighbouring vectors (the bytes of one DRAM burst) by four lanes, lies at a random place of
    // the i-th of equal parts of the tensor
    float c = 0.f, delta = 1.f;
    if (one) {
        const uint64_t nv4 = a.n / (4 * EPV);
        const unsigned total = (unsigned)a.sample * G * (SS_THREADS / 4);
        const uint64_t each = nv4 / total;                    // >= 1
        float e[OP_SAMPLE][EPV];
#pragma unroll
        for (int j = 0; j < OP_SAMPLE; ++j) {
            const unsigned i = ((unsigned)j * G + blockIdx.x) * (SS_THREADS / 4) + threadIdx.x / 4;
            const uint64_t v = (i * each + ((uint64_t)op_place(i) * each >> 32)) * 4 + (lane & 3);
            if (j < a.sample) qp_load_vec(x + v * EPV, e[j]);
        }
        float x0 = qp_load_one(x);                            // (any value near the tensor's: the sums are taken about it)
        if (!qp_is_finite(x0)) x0 = 0.f;
        float p1 = 0.f, p2 = 0.f;
        unsigned pn = 0u;
#pragma unroll
        for (int j = 0; j < OP_SAMPLE; ++j) {
            if (j >= a.sample) break;
            float m = 0.f;
#pragma unroll
            for (int k = 0; k < EPV; ++k) m += e[j][k] - x0;
            m *= 0.25f / EPV;
            m += __shfl_xor_sync(0xFFFFFFFFu, m, 1);
            m += __shfl_xor_sync(0xFFFFFFFFu, m, 2);
            if (m * m < __int_as_float(0x7F800000)) { p1 += m; p2 = fmaf(m, m, p2); ++pn; }
        }
        const SsParts v = ss_block_parts<false>({(double)p1, (double)p2, 0.f, 0.f, pn}, s_block[0]);
        if (threadIdx.x < 32) {
            put(OP_PILOT, ss_row(v.a, v.b));
            put(OP_PILOT + 1, make_uint4(v.count, 0u, 0u, 0u));
        }
        meet_warp0();
        if (threadIdx.x < 32) {
            double t1 = 0.0, t2 = 0.0, tn = 0.0;
            merge(Rows<2>{}, OP_PILOT, [&](const uint4 (&p)[2]) {
                t1 += ss_row_first(p[0]);
                t2 += ss_row_second(p[0]);
                tn += (double)p[1].x;
            });
            __syncwarp();
            t1 = ss_pair_sum(t1, t2);
            tn = ss_pair_sum(tn, 0.0);
            t2 = __shfl_sync(0xFFFFFFFFu, t1, 16);
            if (lane == 0) {                                  // (every sample was counted by its four lanes)
                const double k = tn > 0.0 ? tn : 1.0, m = t1 / k, var = t2 / k - m * m;
                float centre = (float)((double)x0 + m);
                if (!qp_is_finite(centre)) centre = 0.f;
                const double want = fmax(fmax(12.0 * sqrt(fmax(var, 0.0) / k), fabs((double)centre) * 3.814697265625e-6), 1e-30);
                s_c = centre;
                s_delta = (float)fmin(want, 1e30);
            }
        }
        __syncthreads();
        if (!s_ok) { leave(qp_grid::GAVE_UP); return; }
        c = s_c;
        delta = s_delta;
    }

    // ---- the pass
    OpOnes o;
    const int cell_off = (int)(__float_as_uint(delta) >> 17) - (OP_CELLS - 1);   // delta's own cell is the last
    auto pass = [&](auto& f) {
        f.c = c;
        f.delta = delta;
        f.inv_u = 65536.0f / delta;
        f.cell_off = cell_off;
        f.mul = 4u << OP_REPS;
        f.base = (unsigned)__cvta_generic_to_shared(table + (lane & ((1 << OP_REPS) - 1)));
        f.half = (unsigned)OP_CELLS * f.mul;
        f.sy = f.sa = f.sv = f.sx = 0.0;
        f.mn = __int_as_float(0x7F800000);
        f.mx = -f.mn;
        f.below = f.odd = 0u;
        f.nc = qp_pack2(-c, -c);
        Tiles::template run<false>(x, a.ntiles, first, step, lane, f);
        o.mn = f.mn;
        o.mx = f.mx;
        if (f.odd) {                                          // rare: this lane's share again (its window counts stand)
            o.mn = __int_as_float(0x7F800000);
            o.mx = -o.mn;
            for (uint64_t t = first; t < a.ntiles; t += step)
                for (int j = 0; j < SS_TILE / 32 / EPV; ++j)
                    for (int i = 0; i < EPV; ++i) o.one(qp_load_one(x + t * SS_TILE + (j * 32 + lane) * EPV + i), c);
        } else {
            o.sy = f.sy; o.sa = f.sa; o.sv = f.sv; o.sx = f.sx;
            o.below = f.below;
        }
        tail.each([&](float v) {
            o.one(v, c);
            if (one && qp_is_finite(v)) f.window(__fsub_rn(v, c));
        });
    };
    if (one) {
        OpPass<true> f;
        pass(f);
    } else {
        OpPass<false> f;
        pass(f);
    }
    {
        if (a.cluster) qp_grid::cluster_wait();
        const SsParts v = ss_block_parts<true>({o.sy, o.sx, o.mn, o.mx, o.bad}, s_block[1]);       // (its barrier also orders the window's counters)
        SsParts u = {0.0, 0.0, 0.f, 0.f, 0u};
        if (one) u = ss_block_parts<false>({o.sa, o.sv, 0.f, 0.f, o.below}, s_block[2]);
        if (threadIdx.x < 32) {
            put(OP_PASS, ss_row(v.a, v.b));
            put(OP_PASS + 1, make_uint4(__float_as_uint(v.lo), __float_as_uint(v.hi), v.count, u.count));
            if (one) put(OP_PASS + 2, ss_row(u.a, u.b));
        }
    }
    meet_warp0();
    if (threadIdx.x < 32) {
        double sy = 0.0, sx = 0.0, sa = 0.0, sv = 0.0, bad = 0.0, below = 0.0;
        float mn = __int_as_float(0x7F800000), mx = -mn;
        auto first_two = [&](const uint4& p, const uint4& q) {
            sy += ss_row_first(p);
            sx += ss_row_second(p);
            mn = fminf(mn, __uint_as_float(q.x));
            mx = fmaxf(mx, __uint_as_float(q.y));
            bad += (double)q.z;                               // exact: counts are far below 2^53
        };
        if (one) {
            merge(Rows<3>{}, OP_PASS, [&](const uint4 (&p)[3]) {
                first_two(p[0], p[1]);
                below += (double)p[1].w;
                sa += ss_row_first(p[2]);
                sv += ss_row_second(p[2]);
            });
        } else {
            merge(Rows<2>{}, OP_PASS, [&](const uint4 (&p)[2]) { first_two(p[0], p[1]); });
        }
        __syncwarp();
        sy = ss_pair_sum(sy, sx);
        mn = ss_pair_min(mn, -mx);
        bad = ss_pair_sum(bad, below);
        sx = __shfl_sync(0xFFFFFFFFu, sy, 16);
        mx = -__shfl_sync(0xFFFFFFFFu, mn, 16);
        if (one) {
            sa = ss_pair_sum(sa, sv);
            sv = __shfl_sync(0xFFFFFFFFu, sa, 16);
            below = __shfl_sync(0xFFFFFFFFu, bad, 16);
        }
        if (lane == 0) {
            const unsigned long long nbad = (unsigned long long)bad;
            const double nf = (double)(a.n - nbad), D = nf > 0.0 ? sy / nf : 0.0;
            s_st.n = a.n;
            s_st.nonfinite = nbad;
            s_st.mean = nf > 0.0 ? (double)c + D : 0.0;
            s_st.mean_abs = nf > 0.0 ? sx / nf : 0.0;
            s_st.min = nf > 0.0 ? (double)mn : 0.0;
            s_st.max = nf > 0.0 ? (double)mx : 0.0;
            s_st.mad = s_st.var = 0.0;
            s_st.hist_peak = 0;
            s_st.hist_bins = 0;
            s_st.reserved = 0;
            if (one) {
                s_st.var = nf > 0.0 ? fmax(0.0, sv / nf - D * D) : 0.0;
                s_D = D;
                s_abs = sa;
                s_below = below;
            }
            s_again = !one || !(fabs(D) < (double)delta) || !(sv < inf);
        }
    }
    __syncthreads();
    if (!s_ok) { leave(qp_grid::GAVE_UP); return; }
    // ---- this block's share of the elements between c and the mean
    if (one && !s_again) {                                    // uniform over the grid
        const double D = s_D;
        const int side = D < 0.0;
        const float aD = (float)fabs(D);
        const int own = max((int)(__float_as_uint(aD) >> 17) - cell_off, 0);
        double vn = 0.0, vs = 0.0;                            // count and sum below the mean's cell
        unsigned in_own = 0u;                                 // count in it (a block's: below 2^32)
        for (int i = threadIdx.x; i < OP_CELLS; i += SS_THREADS) {
            const unsigned* cnt = table + ((size_t)(side * OP_CELLS + i) << OP_REPS);
            const unsigned* sum = reinterpret_cast<const unsigned*>(raw + OP_SUMS_AT) + ((size_t)(side * OP_CELLS + i) << OP_REPS);
            unsigned long long cn = 0ull, cs = 0ull;
            for (int r = 0; r < (1 << OP_REPS); ++r) {
                const int rr = (r + threadIdx.x) & ((1 << OP_REPS) - 1);
                cn += cnt[rr];
                cs += sum[rr];
                if (cnt[rr] > OP_FULL) s_full = 1;            // benign race: every writer writes 1
            }
            if (i < own) { vn += (double)cn; vs += (double)cs; }
            if (i == own) in_own += (unsigned)cn;
        }
        const SsParts v = ss_block_parts<false>({vn, vs, 0.f, 0.f, in_own}, s_block[0]);
        if (threadIdx.x < 32) {
            put(OP_WINDOW, ss_row(v.a, v.b));
            put(OP_WINDOW + 1, make_uint4(v.count, (unsigned)s_full, 0u, 0u));
        }
        meet_warp0();
        if (threadIdx.x < 32) {
            double tn = 0.0, ts = 0.0, to = 0.0, full = 0.0;
            merge(Rows<2>{}, OP_WINDOW, [&](const uint4 (&p)[2]) {
                tn += ss_row_first(p[0]);
                ts += ss_row_second(p[0]);
                to += (double)p[1].x;
                full += (double)p[1].y;
            });
            __syncwarp();
            tn = ss_pair_sum(tn, ts);
            to = ss_pair_sum(to, full);
            ts = __shfl_sync(0xFFFFFFFFu, tn, 16);
            full = __shfl_sync(0xFFFFFFFFu, to, 16);
            if (lane == 0) {
                const double nf = (double)(a.n - s_st.nonfinite), sum_abs = s_abs;
                const double d = fabs(D), u = (double)delta / 65536.0;
                const double lo = own ? (double)__uint_as_float((unsigned)(own + cell_off) << 17) : 0.0;
                const double hi = (double)__uint_as_float((unsigned)(own + 1 + cell_off) << 17), w = hi - lo;
                const double own_part = to * (d - lo) * (d - lo) / (2.0 * w);         // evenly filled
                const double between = d * tn - u * ts + own_part;
                const double neg = side ? nf - s_below : s_below;                     // elements on the other side of c
                const double sd = sum_abs + d * (neg - (nf - neg)) + 2.0 * between;
                s_st.mad = nf > 0.0 ? fmax(0.0, sd) / nf : 0.0;
                // (sum_abs 0: every element is c)
                s_again = sum_abs != 0.0 && (full > 0.0 || !(to * w * 0.5 <= 1e-8 * sum_abs));
            }
        }
        __syncthreads();
        if (!s_ok) { leave(qp_grid::GAVE_UP); return; }
    }
    if (s_again) {                                            // uniform over the grid
        const float m_hi = (float)s_st.mean, m_lo = (float)(s_st.mean - (double)m_hi);    // the mean as an unevaluated fp32 pair
        const qp_f2 nhi = qp_pack2(-m_hi, -m_hi), nlo = qp_pack2(-m_lo, -m_lo);
        double sd, sv;
        if (s_st.nonfinite) {
            OpDeviations<true> f = {nhi, nlo, 0.0, 0.0};
            Tiles::template run<true>(x, a.ntiles, first, step, lane, f);
            sd = f.sd; sv = f.sv;
        } else {
            OpDeviations<false> f = {nhi, nlo, 0.0, 0.0};
            Tiles::template run<true>(x, a.ntiles, first, step, lane, f);
            sd = f.sd; sv = f.sv;
        }
        tail.each([&](float v) {
            if (!qp_is_finite(v)) return;
            const float dd = __fsub_rn(__fsub_rn(v, m_hi), m_lo);
            sd += (double)fabsf(dd);
            sv += (double)(dd * dd);
        });
        const SsParts v = ss_block_parts<false>({sd, sv, 0.f, 0.f, 0u}, s_block[2]);
        if (threadIdx.x < 32) put(OP_SECOND, ss_row(v.a, v.b));
        meet_warp0();
        if (threadIdx.x < 32) {
            double td = 0.0, tv = 0.0;
            merge(Rows<1>{}, OP_SECOND, [&](const uint4 (&p)[1]) {
                td += ss_row_first(p[0]);
                tv += ss_row_second(p[0]);
            });
            __syncwarp();
            td = ss_pair_sum(td, tv);
            tv = __shfl_sync(0xFFFFFFFFu, td, 16);
            if (lane == 0) {
                const double nf = (double)(a.n - s_st.nonfinite);
                s_st.mad = nf > 0.0 ? td / nf : 0.0;
                s_st.var = nf > 0.0 ? tv / nf : 0.0;
            }
        }
    }
    if (threadIdx.x == 0) {                                   // (it has written s_st itself)
        const qp_stats_t st = s_st;
        if (blockIdx.x == 0 && s_ok) {
            *a.st_out = st;
            if (st.nonfinite) atomicOr(a.status, QP_DEV_NONFINITE);
        }
        if constexpr (BITS > 0) {
            double lo, hi;
            qp_clip_ends(st, a.method, QP_DIST_LAPLACE, a.bmode, BITS, a.F, lo, hi);
            const int rc = qp_fill_qparams(lo, hi, BITS, &s_qp);
            if (blockIdx.x == 0 && s_ok) {
                *a.qp_out = s_qp;
                if (rc == QP_WARN_DEGENERATE) atomicOr(a.status, QP_DEV_DEGENERATE);
            }
        }
    }
    __syncthreads();
    if (!s_ok) { leave(qp_grid::GAVE_UP); return; }
    if constexpr (BITS > 0) {                                 // from the tensor's end, which L2 holds
        uint32_t* sw = reinterpret_cast<uint32_t*>(raw) + (threadIdx.x >> 5) * 256;
        const float lo = s_qp.lo, hi = s_qp.hi, inv = s_qp.inv_scale;
        const uint64_t tiles = (a.n + QP_TILE - 1) / QP_TILE;
        for (uint64_t it = first; it < tiles; it += step) {
            if constexpr (BITS == 16) qp_pack_tile16<T>(x, a.n, tiles - 1 - it, lane, lo, hi, inv, a.packed, a.nwords);
            else qp_pack_tile<BITS, T, true>(x, a.n, tiles - 1 - it, lane, lo, hi, inv, a.packed, a.nwords, sw);
        }
    }
    if (a.cluster) return;
    __syncthreads();
    leave(0u);
}

template <typename T>
void* op_kernel(int bits)
{
    switch (bits) {
        case 0: return (void*)stats_onepass_kernel<T, 0>;
        case 1: return (void*)stats_onepass_kernel<T, 1>;
        case 2: return (void*)stats_onepass_kernel<T, 2>;
        case 3: return (void*)stats_onepass_kernel<T, 3>;
        case 4: return (void*)stats_onepass_kernel<T, 4>;
        case 5: return (void*)stats_onepass_kernel<T, 5>;
        case 6: return (void*)stats_onepass_kernel<T, 6>;
        case 7: return (void*)stats_onepass_kernel<T, 7>;
        case 8: return (void*)stats_onepass_kernel<T, 8>;
        default: return (void*)stats_onepass_kernel<T, 16>;
    }
}

bool op_usable(qp_ctx* ctx)
{
    if (!ctx->op_checked) {
        ctx->op_checked = 1;
        int coop = 0;
        bool ok = cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, ctx->device) == cudaSuccess && coop &&
                  (size_t)ctx->sm_count * OP_ROWS * sizeof(uint4) <= sizeof(qp_stats_partial) * QP_MAX_BLOCKS;
        for (int bits = 0; ok && bits <= 9; ++bits)           // (9: 16 bits)
            for (int v = 0; ok && v < 2; ++v) {
                void* k = v ? op_kernel<unsigned short>(bits) : op_kernel<float>(bits);
                int per_sm = 0;
                ok = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)OP_DYN_BYTES) == cudaSuccess &&
                     cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, SS_THREADS, OP_DYN_BYTES) == cudaSuccess && per_sm >= 1;
            }
        ctx->op_cluster = ok;
        for (int bits = 0; ok && bits <= 9; ++bits)
            for (int v = 0; v < 2; ++v)
                ctx->op_cluster &= qp_cluster_fits(v ? op_kernel<unsigned short>(bits) : op_kernel<float>(bits), SS_THREADS, OP_DYN_BYTES);
        if (!ok) cudaGetLastError();
        ctx->op_ok = ok ? 1 : 0;
    }
    return ctx->op_ok != 0;
}

}  // namespace

bool qp_stats_onepass_applies(qp_ctx* ctx, const void* d_x, uint64_t n)
{
    return !((uintptr_t)d_x & 15u) && n >= 8 * SS_TILE && op_usable(ctx);
}

// Statistics (bits = 0), or with bits 1..8 or 16 the sender with a closed-form clip.
int32_t qp_launch_stats_onepass(qp_ctx* ctx, const void* d_x, int dtype, uint64_t n, qp_stats_t* st_out, int bits, int method,
                                int bmode, double F, qp_qparams_t* d_qp_out, void* d_packed, cudaStream_t s)
{
    static_assert(OP_DYN_BYTES >= SS_WARPS * 1024, "the packer's staging");
    OpArgs a;
    a.x = d_x;
    a.n = n;
    a.ntiles = n / SS_TILE;
    a.st_out = st_out;
    a.qp_out = d_qp_out;
    a.packed = static_cast<uint32_t*>(d_packed);
    a.nwords = bits ? qp_packed_bytes(n, bits) / 4 : 0;
    a.method = method;
    a.bmode = bmode;
    a.F = F;
    a.part = reinterpret_cast<uint4*>(ctx->d_part);
    a.bar = reinterpret_cast<unsigned*>(ctx->d_fused) + 24;   // words 24, 25 of the barrier scratch
    a.status = ctx->d_status;
    a.spin_limit = ctx->spin_limit;
    a.bar_extra = (unsigned)ctx->bar_extra;
    a.cluster = qp_cluster_wanted(ctx, ctx->op_cluster, n);
    const unsigned G = qp_together_blocks(ctx, a.cluster, a.ntiles);
    const uint64_t share = n / (dtype == QP_F32 ? 4 : 8) / ((uint64_t)G * SS_THREADS * 16);   // a sixteenth of the tensor
    // Two passes while the second one finds enough of the tensor in L2 to cost less than the pilot and the window; fp32 of 67, 100 and
    // 134 MB: 24.5, 31.6 and 40.9 us in two passes, 28.6, 34.1 and 39.1 in one (the sender at 8 bits 32.9, 51.1 and 66.5, and 36.9, 51.5
    // and 61.5).  The pass with the window takes twice the elements a byte in bf16: 100, 134, 220 and 268 MB in 37.0, 47.3, 73.2 and 87.5 us in
    // two passes, 45.1, 52.9, 75.6 and 87.8 in one (the sender, up to 134 MB, 65.4 and 86, and 68.7 and 86).
    a.one = n * (dtype == QP_F32 ? 4 : 2) >= (dtype == QP_F32 ? OP_ONE_MIN_BYTES_F32 : OP_ONE_MIN_BYTES_BF16);
    a.sample = share < 1 ? 1 : share < OP_SAMPLE ? (int)share : OP_SAMPLE;
    void* k = dtype == QP_F32 ? op_kernel<float>(bits) : op_kernel<unsigned short>(bits);
    void* params[] = {&a};
    if (qp_launch_together(k, G, SS_THREADS, params, OP_DYN_BYTES, a.cluster, s) != cudaSuccess)
        return qp_check_launch(ctx, "one-pass statistics (cooperative launch)");
    ctx->launches += 1;
    return qp_check_launch(ctx, "one-pass statistics");
}
