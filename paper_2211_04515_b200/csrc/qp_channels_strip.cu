// Channel-wise statistics and directed search (paper Sec. 3, Eq. 1, run per column of a [rows, channels] tensor) in one
// launch: a cluster of S blocks owns a strip of w neighbouring channels, each block a part of the rows, so nothing is
// merged across the grid.
//
//   phase A   sum x, sum |x|, min, max, non-finite count per channel
//   phase B   sum |x - mean|, sum (x - mean)^2, histogram over the channel's [min, max]
//   phase C   per channel, the count and the sum of the elements of every interval between the candidates' thresholds
//             (qp_affine.cuh), in shared memory
//   finish    a team of four warps per channel (two scan a side each): prefix sums over the intervals, the error of every candidate from 2^bits
//             differences (a thread each), first minimum, quantizer
// Between the phases the blocks of a cluster add up their parts through distributed shared memory.  A thread stays with one
// channel and walks its rows, eight loads ahead; the first pass takes the strip from DRAM, the others from L2.
//
// What bounds it: the 32-byte sectors that a strip's rows touch (ct_choose), the instructions (A 4, B 11, C 14 + 2 per code
// boundary and element) with their shared atomics, and the chain of small steps around the passes.  12608 x 1024 fp32 at 4 bits (52 MB), by
// time stamps: A 14 us, its sums across the cluster 3, B 10 and 4, peaks and plans 5, C 20, interval sums across the cluster 6 (16
// bytes a load; 8 with 4 bytes), prefix sums 3 (13 with a `while` over the cells per interval and a warp per side), errors 5 (7 by
// codes instead of by boundaries), pick 1: 72, and the whole stage (receiver, this, packing) 104; with strips of 14 channels, whose rows start anywhere in a sector, and
// those two forms 101 and 134.  Unrolling the errors' loop or three vectors of the interval sums at a time costs 2 us each (straight
// code that runs once).  The ten kernels before (four for the statistics, histogram, set-up, thresholds sorted per
// channel, a pass with binary searches, error curves, pick) took 255 us.
#include <cooperative_groups.h>

#include <type_traits>

#include "qp_affine.cuh"

namespace cg = cooperative_groups;

QP_CK_UNIT

namespace {

constexpr int CT_THREADS = 1024;
constexpr int CT_TEAMS = 8;                        // teams of the finish: a channel each
constexpr int CT_TEAM = CT_THREADS / CT_TEAMS;     // threads of a team (two warps at least: a side each)
constexpr int CT_PEAK = 64;                        // threads that look for a histogram's peak
constexpr int CT_MAX_W = 16;                       // channels of a strip
constexpr int CT_MAX_S = 8;                        // blocks of a cluster
constexpr int CT_AHEAD = 8;                        // loads in flight per thread: a batch
constexpr int CT_PREFETCH = 4;                     // batches that the first pass is prefetched ahead of its loads
constexpr float CT_INF = __builtin_huge_valf();
constexpr int CT_MAX_CAND = QP_CH_MAX_STEPS + 1;
constexpr size_t CT_TABLE_BYTES = 2 * SS_SUMS_AT;  // interval tables (counts, then sums) of the strip
constexpr int CT_HIST_AT = 64 * 1024;              // phase B: the histogram with a replica per lane, where the interval tables will be
static_assert(5 * CT_MAX_W * (CT_THREADS / CT_MAX_W + 1) * sizeof(double) <= CT_HIST_AT && 5 * (CT_THREADS + 1) * sizeof(double) <= CT_HIST_AT, "sums before it");
static_assert(CT_HIST_AT + (QP_CH_MAX_HIST_BINS + 1) * 64 * sizeof(unsigned) <= CT_TABLE_BYTES, "room");
constexpr size_t CT_DYN_BYTES = CT_TABLE_BYTES + (size_t)CT_MAX_W * (QP_CH_MAX_HIST_BINS + 1) * sizeof(unsigned);

struct CtArgs {
    const void* x;
    uint64_t rows;
    uint32_t C;
    int w;                                         // channels per strip
    uint64_t rows_pb;                              // rows per block of a cluster
    int nb, steps, bmode, ncp, ub;
    int len;                                       // words of a channel's intervals, both sides, up to the next 16 bytes
    double F;
    const qp_stats_t* st_in;                       // search only: the caller's statistics
    qp_stats_t* st_out;
    float4* cand;                                  // [C][ncp]
    int* valid;                                    // [C][ncp]
    double* curve;                                 // [C][ncp]
    qp_ds_result_t* ds_out;
    qp_qparams_t* qp_out;
    unsigned* status;
};

// A thread's rows of a column: at byte offsets at, at + st, ... from the block's rows (32 bits: one instruction per address).
struct CtRows { const unsigned char* base; unsigned at, st; };

// CT_AHEAD loads ahead of their use: f.one(value) for each row, f.fold() after every CT_AHEAD of them and at the end.
// ahead(b) is called before batch b's loads are issued, b = 1, 2, ...
struct CtNothing { __device__ __forceinline__ void operator()(int) const {} };
template <typename T, typename F, typename A = CtNothing>
__device__ __forceinline__ void ct_column(const CtRows& rows, int m, F& f, const A& ahead = A())
{
    if (m <= 0) return;
    using Raw = typename std::conditional<sizeof(T) == 4, float, unsigned short>::type;
    unsigned at = rows.at;
    const unsigned st = rows.st;
    auto load = [&](int j) { return __ldg(reinterpret_cast<const Raw*>(rows.base + (at + (unsigned)j * st))); };
    auto value = [](Raw r) {
        if constexpr (sizeof(T) == 4) return (float)r;
        else return qp_bf16_to_f32(r);
    };
    Raw v[CT_AHEAD];
    const int full = m / CT_AHEAD, rest = m - full * CT_AHEAD;
    if (full) {
#pragma unroll
        for (int j = 0; j < CT_AHEAD; ++j) v[j] = load(j);
        for (int b = 1; b < full; ++b) {
            at += CT_AHEAD * st;
            ahead(b);
#pragma unroll
            for (int j = 0; j < CT_AHEAD; ++j) {
                const Raw r = v[j];
                v[j] = load(j);
                f.one(value(r));
            }
            f.fold();
        }
        at += CT_AHEAD * st;
#pragma unroll
        for (int j = 0; j < CT_AHEAD; ++j) f.one(value(v[j]));
        f.fold();
    }
    if (rest) {
#pragma unroll
        for (int j = 0; j < CT_AHEAD; ++j)
            if (j < rest) v[j] = load(j);
#pragma unroll
        for (int j = 0; j < CT_AHEAD; ++j)
            if (j < rest) f.one(value(v[j]));
        f.fold();
    }
}

struct CtMoments {
    double s = 0.0, sa = 0.0;
    float mn = CT_INF, mx = -CT_INF, ps = 0.f, psa = 0.f;
    __device__ __forceinline__ void one(float v)
    {
        ps += v;
        psa += fabsf(v);
        mn = fminf(mn, v);
        mx = fmaxf(mx, v);
    }
    __device__ __forceinline__ void fold()
    {
        s += (double)ps;
        sa += (double)psa;
        ps = psa = 0.f;
    }
};
struct CtMomentsGuarded {                          // a column with non-finite values (or an fp32 overflow)
    double s = 0.0, sa = 0.0, bad = 0.0;
    float mn = CT_INF, mx = -CT_INF;
    __device__ __forceinline__ void one(float v)
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
    __device__ __forceinline__ void fold() {}
};

// Deviations about the fp32 mean, summed in fp64 (as the per-tensor kernel), and the histogram.
template <bool SUMS, bool HIST, int CARE>                     // CARE: as in the per-tensor kernel
struct CtDeviations {
    float m, mn, inv_w;
    unsigned base, mul, nb;                        // byte address of the lane's first bin, less what the float's bits bring; from bin to bin
    double sd = 0.0, sv = 0.0;
    unsigned below = 0u;
    __device__ __forceinline__ void one(float v)
    {
        if (CARE == 2 && !qp_is_finite(v)) return;
        if (SUMS) {
            const float y = __fsub_rn(v, m);
            const double d = (double)y;
            sv = fma(d, d, sv);
            sd += fabs(d);
            below += __float_as_uint(y) >> 31;
        }
        if (HIST) {                                // bin = floor((x - min) * inv_w), each operation rounded; x = max may give nb
            float pos = __fmul_rn(__fsub_rn(v, mn), inv_w);
            if (CARE == 2) pos = fminf(fmaxf(pos, 0.f), (float)nb);
            unsigned bin = __float_as_uint(__fadd_rd(pos, SS_MAGIC)) - SS_ONE;
            if (CARE == 1) bin = min(bin, nb);
            asm volatile("red.shared.add.u32 [%0], 1;" ::"r"((QP_CK(bin, nb + 1) + SS_ONE) * mul + base) : "memory");
        }
    }
    __device__ __forceinline__ void fold() {}
};

template <int HH, bool GUARD>
struct CtCounter {
    const SsPlan<HH>& p;
    const SsTable& tb;
    __device__ __forceinline__ void one(float v)
    {
        if (!GUARD || qp_is_finite(v)) ss_count<HH>(p, tb, v);
    }
    __device__ __forceinline__ void fold() {}
};

// N quantities of every thread added up (OPS: 0 sum, 1 min, 2 max) over the row lanes of its channel: a warp takes a
// channel, in a fixed tree, and leaves the results in out[channel].  red: N * w * (nl | 1) doubles, a channel's values side by side.
template <int... OPS>
__device__ __forceinline__ void ct_reduce(const double (&v)[sizeof...(OPS)], double* red, int slot, int rl, int nl, int w,
                                          double (*out)[sizeof...(OPS)])
{
    constexpr int N = sizeof...(OPS);
    constexpr int ops[N] = {OPS...};
    const int pitch = nl | 1, lane = threadIdx.x & 31;
    if (rl < nl)
#pragma unroll
        for (int j = 0; j < N; ++j) red[(j * w + slot) * pitch + rl] = v[j];
    __syncthreads();
    for (int c = threadIdx.x >> 5; c < w; c += CT_THREADS / 32) {
#pragma unroll
        for (int j = 0; j < N; ++j) {
            const double* at = red + (j * w + c) * pitch;
            auto both = [&](double a, double b) { return ops[j] == 0 ? a + b : (ops[j] == 1 ? fmin(a, b) : fmax(a, b)); };
            double t = ops[j] == 0 ? 0.0 : (ops[j] == 1 ? (double)CT_INF : -(double)CT_INF);
            for (int i = lane; i < nl; i += 32) t = both(t, at[i]);
            __syncwarp();
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) t = both(t, __shfl_xor_sync(0xFFFFFFFFu, t, o));
            if (lane == 0) out[c][j] = t;
        }
    }
}

__device__ __forceinline__ void ct_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void ct_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void ct_team_sync(int team) { asm volatile("barrier.sync %0, %1;" ::"r"(team + 1), "n"(CT_TEAM) : "memory"); }

// STATS: phases A and B (otherwise the statistics come with st_in and B only counts the histogram).  HH: code boundaries above
// the centre, 2^bits / 2 - 1; -1: statistics only.
template <typename T, bool STATS, int HH>
__global__ void __launch_bounds__(CT_THREADS, 1) ch_strip_kernel(const CtArgs a)
{
    constexpr bool SEARCH = HH >= 0;
    constexpr int H = SEARCH ? HH : 0;
    constexpr int BITS = H == 0 ? 1 : H == 1 ? 2 : H == 3 ? 3 : 4;
    extern __shared__ __align__(16) unsigned char raw[];
    __shared__ double s_a[CT_MAX_W][5], s_b[CT_MAX_W][3];     // this block's parts, read by the whole cluster
    __shared__ qp_stats_t s_st[CT_MAX_W];
    const cg::cluster_group cluster = cg::this_cluster();
    const int S = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
    const int w = a.w, lane = threadIdx.x & 31;
    const uint32_t c0 = blockIdx.x / (unsigned)S * (uint32_t)w;
    const int nch = (int)min((uint32_t)w, a.C - c0);
    const int slot = threadIdx.x % w, rl = threadIdx.x / w, nl = CT_THREADS / w;
    const uint64_t r0 = min((uint64_t)rank * a.rows_pb, a.rows), r1 = min(r0 + a.rows_pb, a.rows);
    const bool active = rl < nl && slot < nch && r0 + rl < r1;
    const int m = active ? (int)((r1 - r0 - rl + nl - 1) / nl) : 0;                // rows of this thread
    const CtRows mine = {static_cast<const unsigned char*>(a.x) + r0 * a.C * sizeof(T),
                         active ? ((unsigned)rl * a.C + c0 + (unsigned)slot) * (unsigned)sizeof(T) : 0u,
                         (unsigned)nl * a.C * (unsigned)sizeof(T)};
    const double inf = __longlong_as_double(0x7FF0000000000000ll);
    double* red = reinterpret_cast<double*>(raw);
    unsigned* bins = reinterpret_cast<unsigned*>(raw + CT_TABLE_BYTES);            // [w][nb]
    // Phase B counts with a counter per bin and lane: 32 neighbouring threads meet 32 banks (as w divides 32, otherwise a few twice),
    // whatever their bins (12608 x 1024: 12.5 us with a channel's bins side by side, 10.4 so).
    unsigned* lane_bins = reinterpret_cast<unsigned*>(raw + CT_HIST_AT);           // [nb + 1][pitch], w * copies of the pitch used
    const int copies = (31 + w) / w, pitch = (w * copies + 31) & ~31;
    if constexpr (SEARCH)
        for (int i = threadIdx.x; i < (a.nb + 1) * pitch / 4; i += CT_THREADS) reinterpret_cast<uint4*>(lane_bins)[i] = make_uint4(0u, 0u, 0u, 0u);

    // ---- phase A
    if constexpr (STATS) {
        double v5[5] = {0.0, 0.0, inf, -inf, 0.0};
        {
            // The strips of a rank walk the same rows side by side.  Left to their own loads they ask DRAM for 4 w bytes at a
            // time and wait for it (52 MB: 25 us); so each brings its share of the rows that all of them need four batches
            // later into L2, in one contiguous piece.
            const uint64_t strips = (a.C + w - 1) / w, row_bytes = (uint64_t)a.C * sizeof(T), batch_rows = (uint64_t)nl * CT_AHEAD;
            const unsigned char* base = reinterpret_cast<const unsigned char*>(((uintptr_t)a.x + 15u) & ~(uintptr_t)15u);
            const uint64_t skip = (uint64_t)(base - static_cast<const unsigned char*>(a.x));
            auto prefetch = [&](uint64_t batch) {             // this strip's share of a batch of its rank's rows
                const uint64_t b0 = min((r0 + batch * batch_rows), r1) * row_bytes, b1 = min((r0 + (batch + 1) * batch_rows), r1) * row_bytes;
                const uint64_t share = ((b1 - b0) / strips + 16) & ~(uint64_t)15u, at = blockIdx.x / (unsigned)S * share;
                const uint64_t f0 = (b0 + at) & ~(uint64_t)15u, f1 = min(b0 + at + share, b1) & ~(uint64_t)15u;
                if (f1 > f0 && f1 + skip <= a.rows * row_bytes)
                    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(base + f0), "r"((unsigned)(f1 - f0)) : "memory");
            };
            if (threadIdx.x == 0)
                for (uint64_t b = 0; b < CT_PREFETCH; ++b) prefetch(b);
            CtMoments acc;
            ct_column<T>(mine, m, acc, [&](int b) {
                if (threadIdx.x == 0) prefetch((uint64_t)b - 1 + CT_PREFETCH);
            });
            if (acc.sa < inf) {
                v5[0] = acc.s; v5[1] = acc.sa; v5[2] = (double)acc.mn; v5[3] = (double)acc.mx;
            } else {                                          // rare: the column again, element by element
                CtMomentsGuarded g;
                ct_column<T>(mine, m, g);
                v5[0] = g.s; v5[1] = g.sa; v5[2] = (double)g.mn; v5[3] = (double)g.mx; v5[4] = g.bad;
            }
        }
        ct_reduce<0, 0, 1, 2, 0>(v5, red, slot, rl, nl, w, s_a);
        cluster.sync();
        if ((int)threadIdx.x < nch) {                         // every block the same sums, in rank order
            double t[5] = {0.0, 0.0, inf, -inf, 0.0};
            for (int r = 0; r < S; ++r) {
                const double* q = cluster.map_shared_rank(&s_a[threadIdx.x][0], r);
                t[0] += q[0];
                t[1] += q[1];
                t[2] = fmin(t[2], q[2]);
                t[3] = fmax(t[3], q[3]);
                t[4] += q[4];
            }
            const unsigned long long bad = (unsigned long long)t[4], nf = a.rows - bad;
            qp_stats_t& o = s_st[threadIdx.x];
            o.n = a.rows;
            o.nonfinite = bad;
            o.mean = nf ? t[0] / (double)nf : 0.0;
            o.mean_abs = nf ? t[1] / (double)nf : 0.0;
            o.min = nf ? t[2] : 0.0;
            o.max = nf ? t[3] : 0.0;
            o.mad = o.var = 0.0;
            o.hist_peak = 0;
            o.hist_bins = 0;
            o.reserved = 0;
        }
    } else {
        if ((int)threadIdx.x < nch) s_st[threadIdx.x] = a.st_in[c0 + threadIdx.x];
    }
    auto inv_w = [&](const qp_stats_t& q) { return SEARCH && q.max > q.min ? (float)((double)a.nb / (q.max - q.min)) : 0.f; };
    // a channel whose histogram positions are not all numbers
    const bool beyond = __syncthreads_or((int)threadIdx.x < nch && SEARCH && !ss_range_fits(s_st[threadIdx.x], inv_w(s_st[threadIdx.x])));
    bool odd = false;                                         // a channel with non-finite values: uniform over the cluster
    for (int i = 0; i < nch; ++i) odd |= s_st[i].nonfinite != 0;

    // ---- phase B
    {
        const qp_stats_t& my = s_st[slot < nch ? slot : 0];
        double v3[3];
        auto pass = [&](auto care) {
            CtDeviations<STATS, SEARCH, decltype(care)::value> d;
            d.m = (float)my.mean;
            d.mn = (float)my.min;
            d.inv_w = inv_w(my);
            d.nb = (unsigned)a.nb;
            d.mul = 4u * (unsigned)pitch;
            d.base = (unsigned)__cvta_generic_to_shared(lane_bins + threadIdx.x % (w * copies)) - SS_ONE * d.mul;
            ct_column<T>(mine, m, d);
            v3[0] = d.sd; v3[1] = d.sv; v3[2] = (double)d.below;
        };
        if (odd || beyond) pass(std::integral_constant<int, 2>{}); else pass(std::integral_constant<int, STATS ? 0 : 1>{});
        if constexpr (STATS) {
            ct_reduce<0, 0, 0>(v3, red, slot, rl, nl, w, s_b);
        }
        if constexpr (SEARCH) {                               // this block's bins; what x = max put into bin nb counts in the last one
            if (!STATS) __syncthreads();                      // (ct_reduce has one)
            for (int b = rl; b < a.nb && rl < nl; b += nl) {
                unsigned c = 0u;
                for (int j = 0; j < copies; ++j) {
                    const unsigned* at = lane_bins + b * pitch + j * w + slot;
                    c += at[0];
                    if (b == a.nb - 1) c += at[pitch];
                }
                bins[slot * a.nb + b] = c;
            }
            __syncthreads();                                  // (the interval tables lie where all this is)
        }
        ct_arrive();                                          // (orders the histogram counters of the cluster, too)
        if constexpr (SEARCH)
            for (int i = threadIdx.x; i < w * a.len / 4; i += CT_THREADS)
                reinterpret_cast<uint4*>(raw)[i] = reinterpret_cast<uint4*>(raw + SS_SUMS_AT)[i] = make_uint4(0u, 0u, 0u, 0u);
        ct_wait();
        if (STATS && (int)threadIdx.x < nch) {
            double t[3] = {0.0, 0.0, 0.0};
            for (int r = 0; r < S; ++r) {
                const double* q = cluster.map_shared_rank(&s_b[threadIdx.x][0], r);
#pragma unroll
                for (int j = 0; j < 3; ++j) t[j] += q[j];
            }
            qp_stats_t& o = s_st[threadIdx.x];
            const double nf = (double)(o.n - o.nonfinite), dm = o.mean - (double)(float)o.mean;
            o.mad = nf > 0.0 ? fmax(0.0, t[0] - dm * (nf - 2.0 * t[2])) / nf : 0.0;
            o.var = nf > 0.0 ? fmax(0.0, t[1] / nf - dm * dm) : 0.0;
            if (rank == 0) {
                if (a.st_out) a.st_out[c0 + threadIdx.x] = o;
                if (o.nonfinite) atomicOr(a.status, QP_DEV_NONFINITE);
            }
        }
    }

    // ---- phase C
    if constexpr (SEARCH) {
        __shared__ unsigned s_top[CT_MAX_W];
        __shared__ SsPlan<H> s_plan[CT_MAX_W];
        __shared__ qp_ds_setup s_setup[CT_MAX_W];
        // (in the histogram's room, which is free by then)
        double (*s_v)[CT_MAX_CAND] = reinterpret_cast<double (*)[CT_MAX_CAND]>(raw + CT_TABLE_BYTES);
        int (*s_edge)[SS_GRID + 2] = reinterpret_cast<int (*)[SS_GRID + 2]>(raw + CT_TABLE_BYTES + sizeof(double) * CT_TEAMS * CT_MAX_CAND);
        static_assert(CT_TEAMS * (CT_MAX_CAND * sizeof(double) + (SS_GRID + 2) * sizeof(int)) <= CT_DYN_BYTES - CT_TABLE_BYTES, "room");
        static_assert(CT_MAX_CAND <= CT_TEAM, "a thread per candidate");
        __shared__ uint2 s_n[CT_TEAMS][4];                    // per warp: elements, and the first candidate of the smallest error
        __shared__ unsigned long long s_sum[CT_TEAMS][4];
        const int ncand = a.steps + 1, ni = SS_GRID + 1 + H * ncand;
        if (threadIdx.x < CT_MAX_W) s_top[threadIdx.x] = 0u;
        __syncthreads();
        for (int sl = threadIdx.x / CT_PEAK; sl < nch; sl += CT_THREADS / CT_PEAK) {          // peak of the histogram
            unsigned top = 0u;
            for (int b = threadIdx.x % CT_PEAK; b < a.nb; b += CT_PEAK) {
                unsigned c = 0u;
                for (int r = 0; r < S; ++r) c += cluster.map_shared_rank(bins, r)[sl * a.nb + b];
                top = max(top, c);
            }
            __syncwarp();
            top = __reduce_max_sync(0xFFFFFFFFu, top);
            if (lane == 0) atomicMax(&s_top[sl], top);
        }
        __syncthreads();
        if ((int)threadIdx.x < nch * 8) {                     // eight threads per channel: the common part, and a boundary each
            const int sl = threadIdx.x >> 3, part = (threadIdx.x & 7) - 1;
            qp_ds_setup su;
            qp_ds_make_setup(&s_st[sl], s_st[sl].max > s_st[sl].min ? s_top[sl] : 0u, a.nb, a.bmode, a.F, su);
            su.g_lo = su.g_hi = su.inv_gw = su.inv_u = su.gw = su.pad2 = 0.f;
            su.u = 0.0;
            if (part < 0) s_setup[sl] = su;
            const double k = su.F * ((a.bmode & QP_B_MIDRISE) ? 1.0 - 1.0 / (double)(1 << BITS) : 1.0);
            ss_make_plan<H>(s_plan[sl], part, s_st[sl].mean, k * su.b_e, k * (su.degenerate ? su.b_e : su.b_r),
                            su.degenerate ? 1 : ncand, BITS, a.ub);
        }
        __syncthreads();
        {
            const SsPlan<H> p = s_plan[slot < nch ? slot : 0];
            SsTable tb;
            tb.mul = 4u;
            tb.base = (unsigned)__cvta_generic_to_shared(raw) + (unsigned)(slot * a.len) * 4u - SS_ONE * 4u;
            tb.half = (unsigned)ni * 4u;
            tb.ni = (unsigned)ni;
            tb.ub = (unsigned)a.ub;
            tb.scale = (float)(SS_GRID << a.ub);
            const int rows = p.hard ? 0 : m;                  // (a hard channel is scored candidate by candidate below)
            if (odd) {
                CtCounter<H, true> f = {p, tb};
                ct_column<T>(mine, rows, f);
            } else {
                CtCounter<H, false> f = {p, tb};
                ct_column<T>(mine, rows, f);
            }
        }
        cluster.sync();

        // ---- finish: channel slots rank, rank + S, ... of the strip are this block's.  Their totals over the cluster, in place:
        // count | high bits of the sum << 24 (rows <= 65535, at most 8 sums of 32 bits); 16 bytes a load, the peers one after another
        // from the next one on.
        if (S > 1) {
            const int own = (nch - rank + S - 1) / S, len = a.len / 4;
            uint4* cnt = reinterpret_cast<uint4*>(raw);
            uint4* sum = reinterpret_cast<uint4*>(raw + SS_SUMS_AT);
            for (int e0 = threadIdx.x; e0 < own * len; e0 += 2 * CT_THREADS) {
                uint4 n[2];
                unsigned long long t[2][4];
                int at[2];
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    const int e = min(e0 + j * CT_THREADS, own * len - 1), sl = e / len;
                    at[j] = (rank + sl * S) * len + (e - sl * len);
                    n[j] = cnt[at[j]];
                    const uint4 d = sum[at[j]];
                    t[j][0] = d.x; t[j][1] = d.y; t[j][2] = d.z; t[j][3] = d.w;
                }
                for (int o = 1; o < S; ++o) {
                    const int r = rank + o < S ? rank + o : rank + o - S;
                    const uint4* rc = cluster.map_shared_rank(cnt, r);
                    const uint4* rs = cluster.map_shared_rank(sum, r);
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        const uint4 c = rc[at[j]], d = rs[at[j]];
                        n[j].x += c.x; n[j].y += c.y; n[j].z += c.z; n[j].w += c.w;
                        t[j][0] += d.x; t[j][1] += d.y; t[j][2] += d.z; t[j][3] += d.w;
                    }
                }
#pragma unroll
                for (int j = 0; j < 2; ++j)
                    if (e0 + j * CT_THREADS < own * len) {
                        cnt[at[j]] = make_uint4(n[j].x | (unsigned)(t[j][0] >> 32) << 24, n[j].y | (unsigned)(t[j][1] >> 32) << 24,
                                                n[j].z | (unsigned)(t[j][2] >> 32) << 24, n[j].w | (unsigned)(t[j][3] >> 32) << 24);
                        sum[at[j]] = make_uint4((unsigned)t[j][0], (unsigned)t[j][1], (unsigned)t[j][2], (unsigned)t[j][3]);
                    }
            }
            __syncthreads();
        }
        // a team takes a channel: two warps a side for the prefix sums, then a thread per candidate
        const int team = threadIdx.x / CT_TEAM, tt = threadIdx.x % CT_TEAM, part = tt >> 5, side = part >> 1;
        for (int sl = rank + team * S; sl < nch; sl += CT_TEAMS * S) {
            const SsPlan<H>& p = s_plan[sl];
            if (p.hard) continue;                             // uniform over the team
            const uint32_t c = c0 + sl;
            unsigned* c_up = reinterpret_cast<unsigned*>(raw) + sl * a.len;
            unsigned* t_up = reinterpret_cast<unsigned*>(raw + SS_SUMS_AT) + sl * a.len;
            for (int g = tt; g <= SS_GRID + 1; g += CT_TEAM) s_edge[team][g] = g <= SS_GRID ? ss_cell_start(p, g) : 1 << 30;
            ct_team_sync(team);
            {
                // Consecutive intervals per thread, an odd number of them (no bank twice); an interval is in the cell of the one before
                // it or in the next, as every cell starts an interval.  No branch may part the lanes here: 25 intervals a lane behind a
                // `while` over the cells took 12 us.
                constexpr int HALF = CT_TEAM / 2;
                unsigned* cnt = c_up + side * ni;
                unsigned* sum = t_up + side * ni;
                const int* edge = s_edge[team];
                const int per = ((ni + HALF - 1) / HALF) | 1, i0 = min((tt & (HALF - 1)) * per, ni), i1 = min(i0 + per, ni);
                int cell0 = 0;                                // grid cell of interval i0
#pragma unroll
                for (int o = SS_GRID; o > 0; o >>= 1) cell0 += edge[min(cell0 + o, SS_GRID + 1)] <= i0 ? o : 0;
                // Exclusive prefix sums, in place: count in 17 bits | high bits of the sum << 17, low word of the sum.  First those of
                // the thread's own intervals, then what lies before them.
                unsigned n_all = 0u, at = (unsigned)cell0 << a.ub;
                unsigned long long s_all = 0ull;
                int cell = cell0, next = edge[cell + 1];
                for (int i = i0; i < i1; ++i) {
                    if (next <= i) { ++cell; at += 1u << a.ub; }
                    next = edge[cell + 1];
                    const unsigned cn = cnt[i], n = cn & 0xFFFFFFu, lo = sum[i];
                    cnt[i] = n_all | (unsigned)(s_all >> 32) << 17;
                    sum[i] = (unsigned)s_all;
                    n_all += n;
                    s_all += (unsigned long long)n * at + ((unsigned long long)(cn >> 24) << 32 | lo);
                }
                __syncwarp();
                unsigned np = n_all;
                unsigned long long sp = s_all;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const unsigned tn = __shfl_up_sync(0xFFFFFFFFu, np, o);
                    const unsigned long long ts = __shfl_up_sync(0xFFFFFFFFu, sp, o);
                    if (lane >= o) { np += tn; sp += ts; }
                }
                if (lane == 31) { s_n[team][part].x = np; s_sum[team][part] = sp; }
                ct_team_sync(team);
                np -= n_all;
                sp -= s_all;
                if (part & 1) { np += s_n[team][part - 1].x; sp += s_sum[team][part - 1]; }
                const unsigned before = np | (unsigned)(sp >> 32) << 17, low = (unsigned)sp;
                for (int i = i0; i < i1; ++i) {
                    const unsigned lo = sum[i] + low;
                    cnt[i] += before + (lo < low ? 1u << 17 : 0u);
                    sum[i] = lo;
                }
            }
            ct_team_sync(team);

            const qp_stats_t& q = s_st[sl];
            const qp_ds_setup& su = s_setup[sl];
            const double nf = (double)(q.n - q.nonfinite), dm = q.mean - (double)p.m;
            const double up = (double)(s_n[team][0].x + s_n[team][1].x), down = (double)(s_n[team][2].x + s_n[team][3].x);
            const double s_abs = nf * q.mad + dm * (up - down);
            const double s_up = 0.5 * (s_abs + nf * dm), s_down = 0.5 * (s_abs - nf * dm);     // sum |y| of each side
            const bool flat = !(p.inv_e > 0.f);
            const int k = tt;
            float4 cd = make_float4(0.f, 0.f, 0.f, 0.f);
            double mse = inf;
            if (k < ncand) {
                int ok;
                qp_ds_candidate(su, k, a.steps, BITS, a.bmode & QP_B_MIDRISE, cd, ok);
                a.cand[(size_t)c * a.ncp + k] = cd;
                a.valid[(size_t)c * a.ncp + k] = ok;
                // integers below 2^52 to fp64 by the exponent of 2^52 (the conversion unit is a quarter of the fp64 one's rate)
                auto whole = [](unsigned hi, unsigned lo) { return __hiloint2double((int)(0x43300000u | hi), (int)lo) - 4503599627370496.0; };
                // sum over the codes i of a side of N_i l_i^2 - 2 l_i S_i, by the boundaries between them: with P below a boundary,
                // N l_top^2 - 2 S l_top - sum of (l_i - l_(i-1)) ((l_i + l_(i-1)) P_N - 2 P_S)
                double v = 0.0;
                if (ok) {
                    const int top = flat ? 0 : H;             // (flat: everything has the first code of its side)
                    double a1 = ss_level(cd, H + 1, p.m), a2 = -ss_level(cd, H, p.m);            // distances from the centre
#pragma unroll 1
                    for (int i = 1; i <= top; ++i) {          // boundary i of both sides, outwards
                        const int at = QP_CK(ss_place(p, k, i), ni);
                        const unsigned w1 = c_up[at], w2 = c_up[ni + at];
                        const double l1 = ss_level(cd, H + 1 + i, p.m), l2 = -ss_level(cd, H - i, p.m);
                        v += (l1 - a1) * (2.0 * p.u * whole(w1 >> 17, t_up[at]) - (l1 + a1) * whole(0u, w1 & 0x1FFFFu));
                        v += (l2 - a2) * (2.0 * p.u * whole(w2 >> 17, t_up[ni + at]) - (l2 + a2) * whole(0u, w2 & 0x1FFFFu));
                        a1 = l1;
                        a2 = l2;
                    }
                    v += (up * a1 * a1 - 2.0 * a1 * s_up) + (down * a2 * a2 - 2.0 * a2 * s_down);
                }
                mse = !ok ? inf : nf > 0.0 ? (nf * (q.var + dm * dm) + v) / nf : 0.0;
                a.curve[(size_t)c * a.ncp + k] = mse;
                s_v[team][k] = mse;
            }
            {                                                 // the first minimum, by all of the team
                double bv = mse < inf ? mse : inf;            // (NaN: not below anything)
                int bk = mse < inf ? k : 1 << 30;
                __syncwarp();
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    const double ov = __shfl_xor_sync(0xFFFFFFFFu, bv, o);
                    const int ok = __shfl_xor_sync(0xFFFFFFFFu, bk, o);
                    if (ov < bv || (ov == bv && ok < bk)) { bv = ov; bk = ok; }
                }
                if (lane == 0) s_n[team][part].y = (unsigned)bk;
                ct_team_sync(team);
                double least = inf;
                int best = 0;                                 // (every error infinite or NaN: keep b_E)
#pragma unroll
                for (int j = 0; j < CT_TEAM / 32; ++j) {
                    const unsigned at = s_n[team][j].y;
                    if (at < (unsigned)ncand && s_v[team][at] < least) { least = s_v[team][at]; best = (int)at; }
                }
                if (k == best)
                    qp_ds_write_result(best, s_v[team], su, a.steps, a.nb, BITS, cd, a.ds_out ? a.ds_out + c : nullptr,
                                       a.qp_out + c, a.status);
            }
            ct_team_sync(team);                               // s_v, s_edge, s_n and s_sum are free again
        }

        // ---- hard channels (clip ends coarse against the step): every candidate scored on every element
        bool any_hard = false;
        for (int i = 0; i < nch; ++i) any_hard |= s_plan[i].hard != 0;
        cluster.sync();                                       // nobody reads this block's tables any more
        if (!any_hard) return;                                // uniform over the cluster
        constexpr int K = QP_EVAL_K;
        const int groups = (ncand + K - 1) / K, lanes = CT_THREADS / groups;
        const int g = threadIdx.x % groups, sub = threadIdx.x / groups;
        for (int sl = 0; sl < nch; ++sl) {
            if (!s_plan[sl].hard) continue;
            const uint32_t c = c0 + sl;
            const qp_ds_setup su = s_setup[sl];
            float4 q[K];
            int ok[K];
            double acc[K];
#pragma unroll
            for (int k = 0; k < K; ++k) {
                qp_ds_candidate(su, min(g * K + k, ncand - 1), a.steps, BITS, a.bmode & QP_B_MIDRISE, q[k], ok[k]);
                acc[k] = 0.0;
            }
            if (sub < lanes)
                for (uint64_t r = r0 + sub; r < r1; r += lanes) {
                    const float v = qp_load_one(static_cast<const T*>(a.x) + r * a.C + c);
                    if (!qp_is_finite(v)) continue;
#pragma unroll
                    for (int k = 0; k < K; ++k) {
                        const float pos = qp_grid_pos(v, q[k].x, q[k].y, q[k].w);
                        const float lev = __fsub_rn(__fadd_rn(pos, QP_MAGIC), QP_MAGIC);
                        const float d = __fsub_rn(fmaf(lev, q[k].z, q[k].x), v);
                        acc[k] += (double)(d * d);
                    }
                }
            __syncthreads();
#pragma unroll
            for (int k = 0; k < K; ++k) red[threadIdx.x * K + k] = acc[k];
            __syncthreads();
            for (int k = threadIdx.x; k < ncand; k += CT_THREADS) {
                double t = 0.0;
                for (int l = 0; l < lanes; ++l) t += red[(l * groups + k / K) * K + k % K];
                s_v[0][k] = t;
            }
            cluster.sync();
            if (sl % S == rank) {
                const double nf = (double)(s_st[sl].n - s_st[sl].nonfinite);
                for (int k = threadIdx.x; k < ncand; k += CT_THREADS) {
                    double t = 0.0;
                    for (int r = 0; r < S; ++r) t += *cluster.map_shared_rank(&s_v[0][k], r);
                    float4 cd;
                    int valid;
                    qp_ds_candidate(su, k, a.steps, BITS, a.bmode & QP_B_MIDRISE, cd, valid);
                    a.cand[(size_t)c * a.ncp + k] = cd;
                    a.valid[(size_t)c * a.ncp + k] = valid;
                    const double mse = !valid ? inf : nf > 0.0 ? t / nf : 0.0;
                    a.curve[(size_t)c * a.ncp + k] = mse;
                    s_v[1][k] = mse;
                }
                __syncthreads();
                if (threadIdx.x == 0) {
                    int best = 0;
                    for (int k = 1; k < ncand; ++k)
                        if (s_v[1][k] < s_v[1][best]) best = k;
                    float4 cd;
                    int valid;
                    qp_ds_candidate(su, best, a.steps, BITS, a.bmode & QP_B_MIDRISE, cd, valid);
                    qp_ds_write_result(best, s_v[1], su, a.steps, a.nb, BITS, cd, a.ds_out ? a.ds_out + c : nullptr, a.qp_out + c,
                                       a.status);
                }
            }
            cluster.sync();
        }
    } else {
        cluster.sync();                                       // nobody leaves while its parts may still be read
    }
}

template <typename T>
void* ct_kernel(bool stats, int bits)                         // bits 0: statistics only
{
    if (bits == 0) return (void*)ch_strip_kernel<T, true, -1>;
    if (stats) return bits == 1 ? (void*)ch_strip_kernel<T, true, 0> : bits == 2 ? (void*)ch_strip_kernel<T, true, 1>
                    : bits == 3 ? (void*)ch_strip_kernel<T, true, 3> : (void*)ch_strip_kernel<T, true, 7>;
    return bits == 1 ? (void*)ch_strip_kernel<T, false, 0> : bits == 2 ? (void*)ch_strip_kernel<T, false, 1>
         : bits == 3 ? (void*)ch_strip_kernel<T, false, 3> : (void*)ch_strip_kernel<T, false, 7>;
}

cudaLaunchConfig_t ct_config(cudaLaunchAttribute* at, unsigned blocks, int S, cudaStream_t s)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(CT_THREADS);
    cfg.dynamicSmemBytes = CT_DYN_BYTES;
    cfg.stream = s;
    at->id = cudaLaunchAttributeClusterDimension;
    at->val.clusterDim.x = (unsigned)S;
    at->val.clusterDim.y = at->val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cfg;
}

// Once per context: whether the device holds the kernels, and how many clusters of each size at a time.
bool ct_usable(qp_ctx* ctx)
{
    if (!ctx->ct_checked) {
        ctx->ct_checked = 1;
        int optin = 0;
        bool ok = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, ctx->device) == cudaSuccess;
        for (int bits = 0; ok && bits <= 4; ++bits)
            for (int v = 0; ok && v < (bits ? 4 : 2); ++v) {
                void* k = (v & 1) ? ct_kernel<unsigned short>(v < 2, bits) : ct_kernel<float>(v < 2, bits);
                cudaFuncAttributes fa;
                ok = cudaFuncGetAttributes(&fa, k) == cudaSuccess && (size_t)optin >= fa.sharedSizeBytes + CT_DYN_BYTES &&
                     cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)CT_DYN_BYTES) == cudaSuccess;
            }
        for (int S = 1; ok && S <= CT_MAX_S; ++S) {
            cudaLaunchAttribute at;
            const cudaLaunchConfig_t cfg = ct_config(&at, (unsigned)(S * ctx->sm_count), S, nullptr);
            if (cudaOccupancyMaxActiveClusters(&ctx->ct_clusters[S], ct_kernel<float>(true, 4), &cfg) != cudaSuccess) {
                cudaGetLastError();
                ctx->ct_clusters[S] = 0;
            }
        }
        ok = ok && ctx->ct_clusters[1] > 0;
        if (!ok) cudaGetLastError();
        ctx->ct_ok = ok ? 1 : 0;
    }
    return ctx->ct_ok != 0;
}

// Strip width w and cluster size S by the time of the busiest SM, in ns: of a row, 0.18 per element, 1.5 per 32-byte sector (what a
// load fetches: a strip that starts and ends inside sectors fetches half as much again, and the neighbours fetch it, too) and 2
// whatever its width; and 20 us per wave (prologue, plan and finish).  Measured on 12608 x 1024 fp32 at 4 bits: w 14, S 2 (148 blocks,
// 2.6 sectors a row) 134 us, w 16, S 2 (128 blocks, 2 sectors) 124, w 8, S 1 (128 blocks, 1 sector, four lines a load) 126.  A
// block's part stays below 8192 rows where clusters allow it, so that offsets keep 19 bits.
void ct_choose(const qp_ctx* ctx, const void* x, int size, uint64_t rows, uint32_t C, int max_w, int& w, int& S)
{
    double best = 1e300;
    w = S = 1;
    const bool whole = (((uintptr_t)x | (uint64_t)C * size) & 31u) == 0;          // every row starts with a sector
    for (int s = 1; s <= CT_MAX_S; ++s) {
        if (ctx->ct_clusters[s] < 1 || (s > 1 && (uint64_t)s > rows)) continue;
        for (int v = 1; v <= max_w && (uint32_t)v <= C; ++v) {
            const uint64_t strips = (C + v - 1) / v, waves = (strips + ctx->ct_clusters[s] - 1) / ctx->ct_clusters[s];
            const uint64_t rows_pb = (rows + s - 1) / s;
            const double sectors = (v * size + (whole && v * size % 32 == 0 ? 0 : 32 - size)) / 32.0;
            double cost = (double)waves * ((double)rows_pb * (0.18 * v + 1.5 * sectors + 2.0) + 20000.0);
            if (rows_pb > 8191) cost *= 4.0;
            if (cost < best) { best = cost; w = v; S = s; }
        }
    }
}

}  // namespace

// Statistics per channel (bits = 0), the search on the caller's statistics (st_in), or both.  Rows up to 65535: the packed
// prefix sums hold 17 bits of count (and a block's byte offsets, below 65536 * 4096 * 4, 32 bits).
bool qp_channel_strips_apply(qp_ctx* ctx, uint64_t rows, uint32_t C, int bits)
{
    return rows >= 1 && rows <= 65535 && bits <= 4 && C <= QP_MAX_CHANNELS && ct_usable(ctx);
}

int32_t qp_launch_channel_strips(qp_ctx* ctx, const void* d_x, int dtype, uint64_t rows, uint32_t C, const qp_stats_t* st_in,
                                 qp_stats_t* st_out, int bits, int bmode, int steps, int ncp, int nb, double F, float4* cand,
                                 int* valid, double* curve, qp_ds_result_t* d_out, qp_qparams_t* d_qp_out, cudaStream_t s)
{
    // (statistics always with the strips of the default search, so that they come out the same with and without it)
    const int hh = bits ? (1 << bits) / 2 - 1 : 0;
    const int ni = SS_GRID + 1 + hh * (steps + 1);
    const int len = (2 * ni + 3) & ~3;
    int max_w = CT_MAX_W;
    while (max_w > 1 && (size_t)max_w * len * sizeof(unsigned) > (size_t)SS_SUMS_AT) --max_w;
    int w, S;
    ct_choose(ctx, d_x, dtype == QP_F32 ? 4 : 2, rows, C, max_w, w, S);
    CtArgs a;
    a.len = len;
    a.x = d_x;
    a.rows = rows;
    a.C = C;
    a.w = w;
    a.rows_pb = (rows + S - 1) / S;
    a.nb = nb;
    a.steps = steps;
    a.bmode = bmode;
    a.ncp = ncp;
    // offsets are at most 2^ub and a block's sums of them stay below 2^32; 22 bits keep the grid's integers below 2^28
    a.ub = 22;
    while (a.ub > 0 && (a.rows_pb << a.ub) >= (1ull << 32)) --a.ub;
    a.F = F;
    a.st_in = st_in;
    a.st_out = st_out;
    a.cand = cand;
    a.valid = valid;
    a.curve = curve;
    a.ds_out = d_out;
    a.qp_out = d_qp_out;
    a.status = ctx->d_status;
    void* k = dtype == QP_F32 ? ct_kernel<float>(st_in == nullptr, bits) : ct_kernel<unsigned short>(st_in == nullptr, bits);
    cudaLaunchAttribute at;
    const cudaLaunchConfig_t cfg = ct_config(&at, (unsigned)((C + w - 1) / w * S), S, s);
    void* params[] = {&a};
    if (cudaLaunchKernelExC(&cfg, k, params) != cudaSuccess) return qp_check_launch(ctx, "channel strips");
    ctx->launches += 1;
    return qp_check_launch(ctx, "channel strips");
}
