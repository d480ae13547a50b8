// walk.cu -- the walk-on-boundary kernels:
//   k_dl_lines   Dirichlet problems, double-layer formulation, ray (line)
//                sampling with all-hits queries (Sec. 4.1, 4.4.1)
//   k_sl_walks_ff / k_sl_walks_ris
//                Neumann / Robin problems, single-layer formulation, area
//                sampling / resampled importance sampling (Sec. 4.3)
//   k_nd_lines   Neumann problems through the direct boundary integral
//                equation (Sec. 4.2)
//   k_reduce*    per-query FP64 mean and variance (Sec. 4.1.1)
// plus the debug kernels behind wob_trace_lines / wob_line_axes /
// wob_philox4x32_10.
//
// One thread owns one walk (line walks of calls with few walks: a group of
// lanes, line_engine.cuh); the values of 32 consecutive walks are summed per
// query in a fixed order into (sum, sum of squares) partials
// (add_tile_partials), which k_reduce_part combines per query in a fixed
// order, so results do not depend on scheduling.  Debug solves also write
// every walk's value.
#include <cmath>
#include <cstddef>
#include <cstdlib>

#include "bits.cuh"
#include "ff.cuh"
#include "line_engine.cuh"
#include "wob_host.h"

namespace wob {

namespace {

constexpr double kFourPi = 12.566370614359172953850573533118;

// Line walks: six blocks of 128 threads per SM (80 registers; see
// line_engine.cuh), 24 warps of the grouped form; the forms that need more
// registers than that to keep out of local memory get fewer blocks.
constexpr int kLineBlocks = 6;
constexpr int kNdBlocks = 7;  // direct BIE: 72 registers hold it (20.0 ms on the torus; the step from 6 was 6%)
constexpr int kDebugBlocks = 4;
constexpr int kGroupBlocks = 24 / kG;
// Calls of at most this many walks per SM run with a group of lanes per walk.
// 32,768 walks (216 per SM) take the group and the single lane 141 and 139 us
// (4 lines each, 1,280 triangles), 1,316 and 1,149 us (16 lines, 81,920) and
// 1,033 and 911 us (direct BIE, 12 lines); half as many 88 against 131, 753
// against 1,040 and 587 against 897 us; twice as many 213 against 168, 2,083
// against 1,347 and 1,610 against 1,077 us.
constexpr int64_t kGroupWalksPerSm = 200;
// Single-layer walks with area sampling: 7 blocks of 128 threads per SM (72
// registers, no spills) hide the latency of the CDF search: 4.31 ms for 2.0e8
// samples of the torus with 200,000 triangles, 4.51 with 6 blocks.
#ifndef WOB_SL_MIN_BLOCKS
#define WOB_SL_MIN_BLOCKS 7
#endif
// Resampled single-layer walks: 7 blocks of 128 threads per SM (71 registers, no
// spills with the walk's sums and n_x in shared memory; 1.42 ms for 1.05e6 walks of
// the mixed torus, 6 blocks with n_x in registers 1.48).
constexpr int kRisBlocks = 7, kRisThreads = 128;

// Tiles of 32 consecutive walks of one problem from its global counter
// (dynamic balance), the 64-bit bookkeeping of the two tiles under way and
// the per-tile sums: what the engine's single-problem policies share.
struct WalkTiles {
    const WalkParams& p;
    int64_t total;
    int64_t first0 = 0, first1 = 0;  // first walk of the tile in either slot
    __device__ __forceinline__ explicit WalkTiles(const WalkParams& p_)
        : p(p_), total(p_.Q * (int64_t)p_.N)
    {
    }
    __device__ __forceinline__ bool take(unsigned long long tile, int slot, int& cnt)
    {
        const int64_t first = (int64_t)tile * 32;
        if (first >= total) return false;
        if (slot) first1 = first; else first0 = first;
        cnt = total - first < 32 ? (int)(total - first) : 32;
        return true;
    }
    __device__ __forceinline__ bool fetch(int slot, int& cnt)
    {
        unsigned long long tile = 0;
        if ((threadIdx.x & 31) == 0) tile = atomicAdd(p.tile_counter, 1ull);
        return take(__shfl_sync(kAllLanes, tile, 0), slot, cnt);
    }
    // a tile for the whole block (into slot 0)
    __device__ __forceinline__ bool fetch_block(unsigned long long* shared, int& cnt)
    {
        if (threadIdx.x == 0) *shared = atomicAdd(p.tile_counter, 1ull);
        __syncthreads();
        const unsigned long long tile = *shared;
        __syncthreads();
        return take(tile, 0, cnt);
    }
    __device__ __forceinline__ int64_t index(const LaneWalk& lw) const
    {
        return (lw.id < 32 ? first0 : first1) + (lw.id & 31);
    }
    // stream ids and coordinates of the walk's query; returns the query's row
    template <class Mem>
    __device__ __forceinline__ int64_t start(const Mem& mem, const LaneWalk& lw, float3& x) const
    {
        const int64_t idx = index(lw);
        const int64_t qi = idx / p.N;
        mem.set_ids(p.q_base + (uint32_t)qi, (uint32_t)(p.walk_begin + (idx - qi * p.N)));
        x = make_float3(p.queries[3 * qi], p.queries[3 * qi + 1], p.queries[3 * qi + 2]);
        return qi;
    }
    __device__ __forceinline__ void close(int slot, int cnt, double v) const
    {
        if (!p.part) return;
        const int lane = threadIdx.x & 31;
        const bool live = lane < cnt;
        const int64_t idx = (slot ? first1 : first0) + lane;
        const int64_t qi = live ? idx / p.N : 0;
        add_tile_partials(v, live, qi, idx - qi * p.N, p.tpq, p.part);
    }
    __device__ __forceinline__ StreamKey key(const LaneWalk&) const { return {p.key0, p.key1}; }
    __device__ __forceinline__ LineGeom geom(const LaneWalk&) const
    {
        return {p.nodes, p.tv, p.edge_thr_L, p.tauL, p.graze, p.iter_limit};
    }
    // debug solves: per-line outputs of the walk
    __device__ __forceinline__ LineOut lines(const LaneWalk& lw) const
    {
        const int64_t lk = index(lw) * p.M;
        return {p.line_m ? p.line_m + lk : nullptr, p.line_prim ? p.line_prim + lk : nullptr,
                p.line_flag ? p.line_flag + lk : nullptr};
    }
};

// Dirichlet walks (double layer) of one problem.
template <bool DEBUG, bool GRAD>
struct DlWalks : WalkTiles {
    using Base = WalkTiles;
    using Base::p;
    __device__ __forceinline__ explicit DlWalks(const WalkParams& p_) : Base(p_) {}
    template <class Mem>
    __device__ __forceinline__ void begin(const Mem& mem, LaneWalk& lw)
    {
        float3 x;
        const int64_t qi = Base::start(mem, lw, x);
        int start = -1;
        if (p.query_prim) {  // density walks from boundary points
            const int32_t prim = p.query_prim[qi];
            start = (prim >= 0 && prim < p.T) ? p.inv_order[prim] : -1;
        }
        dl_begin(mem, lw, x, start, p.data, p.tv, (double)p.phi, p.M);
        if (GRAD) p.per_walk[Base::index(lw)] = __hiloint2double(0, -1);  // no first hit yet
        if (DEBUG) {
            const LineOut lo = Base::lines(lw);
            for (int k = 0; k < p.M; ++k) lo.put(k, -1, -1, 0);
        }
    }
    template <class Mem>
    __device__ __forceinline__ bool depart(const Mem&, const LaneWalk& lw) const
    {
        return lw.k < p.M;
    }
    template <class Mem>
    __device__ __forceinline__ bool land(const Mem& mem, LaneWalk& lw, int m, int pos, int flag)
    {
        if (DEBUG) {
            lw.flag |= flag;
            Base::lines(lw).put(lw.k, m, pos >= 0 ? (int)prim_of(p.tv, pos) : -1, flag);
        }
        if (m == 0) return false;
        const bool first = GRAD && lw.k == 0;
        dl_land(mem, lw, m, pos, p.data, p.tv, (double)p.phi, p.M);
        if (first) park(Base::index(lw), pos, mem.x(0), mem.x(1), mem.x(2));
        return lw.k < p.M;
    }
    template <class Mem>
    __device__ __forceinline__ double value(const Mem& mem, const LaneWalk& lw) const
    {
        const double v = mem.get(kAccS);
        if (DEBUG) {
            const int64_t idx = Base::index(lw);
            if (p.per_walk) p.per_walk[idx] = v;
            if (p.walk_flag) p.walk_flag[idx] = (uint8_t)lw.flag;
        }
        return v;
    }
    // The first hit of a walk waits in the walk's own output slots until its
    // tile is complete: its gradient factor takes FP64 square roots and
    // divisions, which cost the warp the same for one lane as for 32.
    __device__ __forceinline__ void park(int64_t idx, int pos, ff y0, ff y1, ff y2) const
    {
        const ff y[3] = {y0, y1, y2};
        p.per_walk[idx] = __hiloint2double(0, pos);
        for (int c = 0; c < 3; ++c)
            p.per_walk_grad[c * Base::total + idx] =
                __hiloint2double(__float_as_int(y[c].hi), __float_as_int(y[c].lo));
    }
    __device__ __forceinline__ void close(int slot, int cnt, double v) const
    {
        Base::close(slot, cnt, v);
        const int lane = threadIdx.x & 31;
        if (GRAD && lane < cnt) {  // gradient of a walk: first-step factor x walk value
            const int64_t idx = (slot ? Base::first1 : Base::first0) + lane;
            const int pos = __double2loint(p.per_walk[idx]);
            double3 g = make_double3(0.0, 0.0, 0.0);
            if (pos >= 0) {
                double y[3];
                for (int c = 0; c < 3; ++c) {
                    const double b = p.per_walk_grad[c * Base::total + idx];
                    y[c] = ff_join({__int_as_float(__double2hiint(b)), __int_as_float(__double2loint(b))});
                }
                const float* x = p.queries + 3 * (idx / p.N);
                g = grad_factor(p.tv, pos, make_double3(x[0], x[1], x[2]), make_double3(y[0], y[1], y[2]));
            }
            p.per_walk[idx] = v;
            p.per_walk_grad[idx] = g.x * v;
            p.per_walk_grad[Base::total + idx] = g.y * v;
            p.per_walk_grad[2 * Base::total + idx] = g.z * v;
        }
    }
};

template <bool COUNT, bool DEBUG, bool GRAD>
__global__ void __launch_bounds__(kLineThreads, DEBUG ? kDebugBlocks : kLineBlocks) k_dl_lines(WalkParams p)
{
    __shared__ LineShared sm;
    extern __shared__ int line_stack[];
    int err = 0;
    WalkCount c{0, 0, 0, 0, 0};
    DlWalks<DEBUG, GRAD> pol(p);
    run_lines<DlWalks<DEBUG, GRAD>, COUNT>(pol, sm.lane(line_stack), sm.vals, p.stack_levels, err, c);
    if (err) atomicOr(p.error_word, err);
    if (COUNT) {
        atomicAdd(p.counters + 0, c.lines);
        atomicAdd(p.counters + 1, c.nodes);
        atomicAdd(p.counters + 2, c.tris);
        atomicAdd(p.counters + 3, c.hits);
        atomicAdd(p.counters + 4, c.flag);
    }
}

template <bool GRAD>
__global__ void __launch_bounds__(kGroupThreads, kGroupBlocks) k_dl_groups(WalkParams p)
{
    __shared__ GroupShared sm;
    extern __shared__ int line_stack[];
    int err = 0;
    DlWalks<false, GRAD> pol(p);
    run_line_groups(pol, sm, line_stack, p.stack_levels, err);
    if (err) atomicOr(p.error_word, err);
}

// Data of the single-layer problems at y on triangle j (original order):
// with condition bc (wob_bc) the field h (Dirichlet), its normal derivative
// dh/dn (Neumann) or dh/dn + alpha h (Robin); P1 mode: the vertex values.
__device__ __forceinline__ double sl_data(const WalkParams& p, int64_t j, double3 y, double b0,
                                          double b1, double b2, double3 n, int bc)
{
    const DataDev& D = p.data;
    if (D.mode == WOB_DATA_VERTEX_P1) {
        const int32_t* t = D.tris + 3 * j;
        return b0 * __ldg(D.vdata + t[0]) + b1 * __ldg(D.vdata + t[1]) + b2 * __ldg(D.vdata + t[2]);
    }
    double h, gx, gy, gz;
    if (D.mode == WOB_DATA_POLY) {
        const float* c = D.poly;
        h = c[0] + c[1] * y.x + c[2] * y.y + c[3] * y.z + c[4] * y.x * y.x + c[5] * y.y * y.y +
            c[6] * y.z * y.z + c[7] * y.x * y.y + c[8] * y.y * y.z + c[9] * y.z * y.x;
        gx = c[1] + 2.0 * c[4] * y.x + c[7] * y.y + c[9] * y.z;
        gy = c[2] + 2.0 * c[5] * y.y + c[7] * y.x + c[8] * y.z;
        gz = c[3] + 2.0 * c[6] * y.z + c[8] * y.y + c[9] * y.x;
    } else {
        const double rx = y.x - D.x0[0], ry = y.y - D.x0[1], rz = y.z - D.x0[2];
        const double rl = sqrt(rx * rx + ry * ry + rz * rz);
        h = D.scale / rl;
        const double f = -D.scale / (rl * rl * rl);
        gx = f * rx;
        gy = f * ry;
        gz = f * rz;
    }
    if (bc == WOB_BC_DIRICHLET) return h;
    const double dhdn = n.x * gx + n.y * gy + n.z * gz;
    return bc == WOB_BC_ROBIN ? dhdn + (double)p.alpha * h : dhdn;
}

// Index of the triangle whose area-CDF interval holds the 53-bit uniform
// U = (hi, lo) times the total area: the first j with cdf[j] > fl(U 2^-53
// |Gamma|), else T - 1 (inverse CDF).  The guide table brackets the answer
// by the top bits of U (about one triangle per bucket), and a binary search
// inside the bracket makes the same comparisons as one over the whole CDF.
// Non-negative doubles order as their bit patterns: the search compares
// 64-bit integers (the same decisions as double compares, off the FP64
// pipe, which issues at 1/64 of the FP32 rate on this GPU).  The target is
// one FP64 multiply, (U 2^-53) |Gamma|; U 2^-53 is exact and formed from its
// bit pattern in the integer pipes (u53_unit).
__device__ __forceinline__ int64_t area_pick(const WalkParams& p, uint32_t hi, uint32_t lo)
{
    const uint64_t U = ((uint64_t)hi << 21) | (uint64_t)(lo >> 11);
    const long long target = __double_as_longlong(u53_unit(U) * p.area);
    const uint32_t b = hi >> (32 - p.guide_bits);  // top guide_bits bits of U
    int32_t a = __ldg(p.guide + b), e = __ldg(p.guide + b + 1);
    const int32_t last = (int32_t)p.T - 1;
    e = e < last ? e : last;
    while (a < e) {
        const int32_t mid = a + ((e - a) >> 1);
        if (__double_as_longlong(__ldg(p.cdf + mid)) > target) e = mid; else a = mid + 1;
    }
    return a;
}

// ---------------------------------------------------------------------------
// Single-layer walks with area sampling in compensated FP32.  Each sample
// point is kept as its triangle's first vertex v0 (FP32, exact) plus the
// offset p = b1 e1 + b2 e2 in float-float (hi + lo, about 44 bits); the
// difference of two points is (v0_y - v0_x) + (p_y - p_x), with the vertex
// difference exact (Knuth's two-sum), so it is accurate relative to its own
// length however close the points are.  r . n_x (which cancels to ~r^2 / 2
// near x on a smooth surface) and the Robin numerator alpha r^2 + r . n_x
// (whose terms can cancel) are float-float sums; 1 / r, G and dG/dn_x are
// FP32 with relative error ~1e-7.  The product of weights is an FP32
// significand renormalised every step with an integer exponent; FP64 holds
// only the sum of terms (one add per step, the term assembled exactly from
// its bits by scale2) and the CDF target (one multiply).
// ---------------------------------------------------------------------------

// Two float-float values as the lanes of packed FP32x2 operations, each lane
// rounded as ff.cuh's operations round it.  The low parts are kept negated (an
// exact change): the packed operations take no negated operands, and the errors
// come out of fma(a, -b, ab) and of differences without extra instructions.
// Resampled walks 1.52 -> 1.37 ms against the scalar form (1.05e6 walks x 4
// vertices x 16 candidates), single-layer walks, which wait for their loads
// rather than for issue, 4.53 -> 4.51 ms.
struct ff2 {
    float2 hi, nlo;
};
__device__ __forceinline__ float2 sub2(float2 a, float2 b)
{
    return __ffma2_rn(b, make_float2(-1.f, -1.f), a);
}
__device__ __forceinline__ ff2 two_sum2(float2 a, float2 b)
{
    const float2 s = __fadd2_rn(a, b), bb = sub2(s, a);
    return {s, __fadd2_rn(sub2(sub2(s, bb), a), sub2(bb, b))};
}
__device__ __forceinline__ ff2 two_diff2(float2 a, float2 b)
{
    const float2 s = sub2(a, b), bb = sub2(s, a);
    return {s, __fadd2_rn(sub2(sub2(s, bb), a), __fadd2_rn(bb, b))};
}
// fast_two_sum(a, -n)
__device__ __forceinline__ ff2 fast_two_sub2(float2 a, float2 n)
{
    const float2 s = sub2(a, n);
    return {s, __fadd2_rn(n, sub2(s, a))};
}
__device__ __forceinline__ ff2 ff_mul_f2(ff2 a, float2 b)
{
    const float2 nb = sub2(make_float2(0.f, 0.f), b), p = __fmul2_rn(a.hi, b);
    return fast_two_sub2(p, __ffma2_rn(a.nlo, b, __ffma2_rn(a.hi, nb, p)));
}
// (ah + al) b
__device__ __forceinline__ ff2 ff_mul2(float2 ah, float2 al, ff2 b)
{
    const float2 nb = sub2(make_float2(0.f, 0.f), b.hi), p = __fmul2_rn(ah, b.hi);
    return fast_two_sub2(p, __ffma2_rn(ah, b.nlo, __ffma2_rn(al, nb, __ffma2_rn(ah, nb, p))));
}

// A boundary point in the compensated representation.
struct FFPoint {
    float v0[3];  // the triangle's first vertex
    ff p[3];      // offset from v0
    ff n[3];      // unit normal of the triangle
};

// Area-uniform boundary point of stream (q, w, step) in the compensated
// form: triangle j by area_pick, then (frame_point_ff, uniforms uz, uw) the
// square-root warp b1 = sqrt(u1) (1 - u2), b2 = sqrt(u1) u2 with sqrt(u1) in
// float-float and the offset p = b1 e1 + b2 e2 in float-float from the
// triangle's frame (six 16-byte loads); b0..b2 in FP32 for P1 data.
__device__ __forceinline__ void frame_point_ff(const WalkParams& p, int64_t j, uint32_t uz,
                                               uint32_t uw, FFPoint& y, float& b0, float& b1f,
                                               float& b2f)
{
    const float4* F = reinterpret_cast<const float4*>(p.tri_f + j);
    const float4 f0 = __ldg(F), f1 = __ldg(F + 1), f2 = __ldg(F + 2), f3 = __ldg(F + 3),
                 f4 = __ldg(F + 4), f5 = __ldg(F + 5);
    const float u2 = u24f(uw);
    const ff su = ff_sqrt(u24f(uz));
    // (b1, b2) = sqrt(u1) (1 - u2, u2)
    const ff2 b = ff_mul_f2({make_float2(su.hi, su.hi), make_float2(-su.lo, -su.lo)},
                            make_float2(1.f - u2, u2));
    b0 = 1.f - su.hi;
    b1f = b.hi.x;
    b2f = b.hi.y;
    const float2 eh[3] = {{f1.x, f1.y}, {f1.z, f1.w}, {f2.x, f2.y}};
    const float2 el[3] = {{f2.z, f2.w}, {f3.x, f3.y}, {f3.z, f3.w}};
    const float v0[3] = {f0.x, f0.y, f0.z};
    const float nh[3] = {f4.x, f4.y, f4.z}, nl[3] = {f4.w, f5.x, f5.y};
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        y.v0[c] = v0[c];
        y.n[c] = {nh[c], nl[c]};
        const ff2 t = ff_mul2(eh[c], el[c], b);  // (e1 b1, e2 b2)
        const ff s = two_sum(t.hi.x, t.hi.y);
        y.p[c] = fast_two_sum(s.hi, rn_sub(s.lo, rn_add(t.nlo.x, t.nlo.y)));
    }
}

// r = y - x of two points, component by component the float-float sum of the
// exact difference of their first vertices and the difference of their offsets.
__device__ __forceinline__ void point_diff(const FFPoint& y, const FFPoint& x, ff (&r)[3])
{
    const ff2 v = two_diff2(make_float2(y.v0[0], y.v0[1]), make_float2(x.v0[0], x.v0[1]));
    ff2 d = two_diff2(make_float2(y.p[0].hi, y.p[1].hi), make_float2(x.p[0].hi, x.p[1].hi));
    const float2 l = sub2(make_float2(y.p[0].lo, y.p[1].lo), make_float2(x.p[0].lo, x.p[1].lo));
    d = fast_two_sub2(d.hi, sub2(d.nlo, l));
    const ff2 s = two_sum2(v.hi, d.hi);
    d = fast_two_sub2(s.hi, __fadd2_rn(s.nlo, __fadd2_rn(v.nlo, d.nlo)));
    r[0] = {d.hi.x, -d.nlo.x};
    r[1] = {d.hi.y, -d.nlo.y};
    r[2] = ff_add(two_sum(y.v0[2], -x.v0[2]), ff_sub(y.p[2], x.p[2]));
}

__device__ __forceinline__ int64_t area_sample_ff(const WalkParams& p, StreamKey key, uint32_t q,
                                                  uint32_t w, uint32_t step, FFPoint& y,
                                                  float& b0, float& b1f, float& b2f)
{
    const u32x4 u = stream_block(key, q, w, step, kPurposeArea, 0u, 0u);
    const int64_t j = area_pick(p, u.x, u.y);
    frame_point_ff(p, j, u.z, u.w, y, b0, b1f, b2f);
    return j;
}

// Data of the single-layer problems at the point (v0 + p, normal n, on
// triangle j with barycentrics b0..b2), as sl_data, rounded to FP32: P1
// values in FP32, the point-source field in FP32 with n . grad h by FMAs (its
// error ~1e-7 of |grad h|; with precise_dn the projection n . (y - x0) is a
// float-float dot product, so the error is ~1e-7 of n . grad h itself),
// polynomial data in FP64 at the FP64 position (its monomials cancel) and
// then rounded.
__device__ __forceinline__ float sl_data_ff(const WalkParams& p, int64_t j, const FFPoint& y,
                                            float b0, float b1, float b2, int bc,
                                            bool precise_dn = false)
{
    const DataDev& D = p.data;
    if (D.mode == WOB_DATA_VERTEX_P1) {
        const int32_t* t = D.tris + 3 * j;
        return __fmaf_rn(b0, __ldg(D.vdata + t[0]),
                         __fmaf_rn(b1, __ldg(D.vdata + t[1]), b2 * __ldg(D.vdata + t[2])));
    }
    if (D.mode == WOB_DATA_POLY) {
        double3 yd, nd;
        yd.x = (double)y.v0[0] + ((double)y.p[0].hi + (double)y.p[0].lo);
        yd.y = (double)y.v0[1] + ((double)y.p[1].hi + (double)y.p[1].lo);
        yd.z = (double)y.v0[2] + ((double)y.p[2].hi + (double)y.p[2].lo);
        nd = make_double3((double)y.n[0].hi + (double)y.n[0].lo, (double)y.n[1].hi + (double)y.n[1].lo,
                          (double)y.n[2].hi + (double)y.n[2].lo);
        return (float)sl_data(p, j, yd, (double)b0, (double)b1, (double)b2, nd, bc);
    }
    const float dx = (y.v0[0] - D.x0[0]) + y.p[0].hi;
    const float dy = (y.v0[1] - D.x0[1]) + y.p[1].hi;
    const float dz = (y.v0[2] - D.x0[2]) + y.p[2].hi;
    const float ri = rsqrt_ftz(__fmaf_rn(dx, dx, __fmaf_rn(dy, dy, dz * dz)));
    const float h = D.scale * ri;
    if (bc == WOB_BC_DIRICHLET) return h;
    float dn = __fmaf_rn(y.n[0].hi, dx, __fmaf_rn(y.n[1].hi, dy, y.n[2].hi * dz));
    if (precise_dn) {  // n . (y - x0) as a float-float dot product (it cancels where
                       // the field runs along the surface)
        ff d[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) d[c] = ff_add(two_sum(y.v0[c], -D.x0[c]), y.p[c]);
        dn = ff_dot3(y.n, d).hi;
    }
    const float dhdn = -h * ri * ri * dn;
    return bc == WOB_BC_ROBIN ? __fmaf_rn(p.alpha, h, dhdn) : dhdn;
}

// Single-layer walks (Table 1, Sec. 4.3) with area sampling (p.ris <= 1), one
// thread per walk, in the compensated FP32 arithmetic above:
// u(x0) = int G mu and mu(x) = int K(x, y) mu(y) + src(x) with K = G (query),
// -2 phi dG/dn_x (Neumann), -2 phi (dG/dn_x + alpha G) (Robin), -(k/p_k) G
// (Dirichlet, moving branch), dG/dn_x = (y - x) . n_x / (4 pi r^3), 0 for
// r < 1e-12 L; src = 2 phi q (Neumann), 2 phi (q + alpha h) (Robin), k u_D
// (Dirichlet parts of mixed problems, whose mu(x) = mu(x) - k S mu + k u_D is
// sampled by moving with probability p_k or staying at x with weight
// 1 / (1 - p_k)).  The last source is halved (Sec. 4.1.2).
template <bool DEBUG>
__global__ void __launch_bounds__(128, WOB_SL_MIN_BLOCKS) k_sl_walks_ff(WalkParams p)
{
    constexpr float kInv4Pi = 0.0795774715459476678f;
    const StreamKey key{p.key0, p.key1};
    const int64_t total = p.Q * (int64_t)p.N;
    const float two_phi = 2.f * (float)p.phi;
    const float rmin2 = (float)(1e-24 * p.L * p.L);
    const int uniform_bc = p.kind == WOB_ROBIN_SL ? WOB_BC_ROBIN : WOB_BC_NEUMANN;
    // weight factors: |Gamma| (query), -|Gamma| k / p_k (Dirichlet parts),
    // -2 phi |Gamma| (Neumann / Robin), rounded to FP32 once
    const float w_query = (float)p.area;
    const float w_dirichlet = (float)(-p.area * (double)(p.kmix / p.pk));
    const float w_layer = (float)(-2.0 * (double)p.phi * p.area);
    const float w_stay = (float)(1.0 / (1.0 - (double)p.pk));
    const int lane = threadIdx.x & 31;
    for (int64_t base = blockIdx.x * (int64_t)blockDim.x + (threadIdx.x & ~31); base < total;
         base += (int64_t)gridDim.x * blockDim.x) {
        const int64_t idx = base + lane;
        const bool live = idx < total;
        const int64_t qi = live ? idx / p.N : 0;
        const int64_t wi = idx - qi * p.N;
        double value = 0.0;
        if (live) {
            const uint32_t q = p.q_base + (uint32_t)qi;
            const uint32_t w = (uint32_t)(p.walk_begin + wi);
            // x: the query (v0 = its coordinates, p = 0) or the last sample
            FFPoint x;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                x.v0[c] = p.queries[3 * qi + c];
                x.p[c] = {0.f, 0.f};
                x.n[c] = {0.f, 0.f};
            }
            int bx = -1;
            int64_t jx = -1;
            // the weight product P = Pm 2^Pe (FP32 significand renormalised to
            // [1, 2) every step, integer exponent: no overflow over long walks)
            // and the sum of terms S in FP64
            double S = 0.0;
            float Pm = 1.f, W0 = 0.f;
            int Pe = 0;
            for (int k = 0; k < p.M; ++k) {
                bool stay = false;
                if (bx == WOB_BC_DIRICHLET) {
                    const u32x4 u = stream_block(key, q, w, (uint32_t)k, kPurposeBranch, 0u, 0u);
                    stay = u24f(u.x) >= p.pk;  // both exact in FP32
                }
                FFPoint y;
                int64_t j;
                float b0 = 0.f, b1f = 0.f, b2f = 0.f;  // mixed problems' stays take analytic data
                float wf;
                if (stay) {
                    y = x;
                    j = jx;
                    wf = w_stay;
                } else {
                    j = area_sample_ff(p, key, q, w, (uint32_t)k, y, b0, b1f, b2f);
                    ff r[3];
                    point_diff(y, x, r);
                    const float r2 =
                        __fmaf_rn(r[0].hi, r[0].hi, __fmaf_rn(r[1].hi, r[1].hi, r[2].hi * r[2].hi));
                    if (r2 < rmin2) break;  // empty sample
                    const float ri = rsqrt_ftz(r2);
                    const float G = kInv4Pi * ri;
                    if (bx < 0) {
                        wf = w_query * G;
                    } else if (bx == WOB_BC_DIRICHLET) {
                        wf = w_dirichlet * G;
                    } else {
                        ff num = ff_dot3(x.n, r);  // r . n_x
                        if (bx == WOB_BC_ROBIN) {
                            // alpha r^2 + r . n_x, r^2 as a float-float sum of squares
                            const ff rr = ff_dot3(r, r);
                            num = ff_add(num, ff_mul_f(rr, p.alpha));
                        }
                        wf = w_layer * (num.hi * (ri * ri) * G);
                    }
                }
                if (k == 0) {
                    W0 = wf;
                } else {
                    Pm *= wf;
                    const uint32_t pb = __float_as_uint(Pm);
                    const int pe = (int)((pb >> 23) & 0xFFu);
                    if (pe != 0 && pe != 255) {  // zero, subnormal, inf, NaN stay as they are
                        Pe += pe - 127;
                        Pm = __uint_as_float((pb & 0x807FFFFFu) | 0x3F800000u);
                    }
                }
                const int by = p.bc_type ? (int)__ldg(p.bc_type + j) : uniform_bc;
                const float dat = sl_data_ff(p, j, y, b0, b1f, b2f, by);
                float src = (by == WOB_BC_DIRICHLET ? p.kmix : two_phi) * dat;
                if (k == p.M - 1) src *= 0.5f;
                S += scale2(Pm * src, Pe);
                x = y;
                bx = by;
                jx = j;
            }
            value = (double)W0 * S;
            if (p.per_walk) p.per_walk[idx] = value;
            if (DEBUG && p.walk_flag) p.walk_flag[idx] = 0;
        }
        if (p.part) add_tile_partials(value, live, qi, wi, p.tpq, p.part);
    }
}

// ---------------------------------------------------------------------------
// Single-layer walks with resampled importance sampling (Talbot et al. 2005):
// the next point is drawn from p.ris area-uniform candidates with target |K|,
// weight sign(K) |Gamma| (sum of |K| over the candidates) / ris; walks, K and
// sources as in k_sl_walks_ff.  The pick compares running sums of |K|, so a
// rounding can move it to another candidate: points, kernels and sums are
// float-float (44 bits and more; a pick moves about once in 10^11 draws), and
// the walk's weights, terms and sums FP64.  What bounds it: a candidate's guide,
// CDF and frame reads (L1 80% busy) and some 500 instructions, where about 60 FP64
// instructions, each worth 64 FP32 issue slots on this GPU, took 14.1 ms for 1.05e6
// walks x 4 vertices x 16 candidates (200,000 triangles).  Now 1.42 ms; 2.5 ms while
// lanes that stayed or had another condition branched apart (16 of 32 active).
// ---------------------------------------------------------------------------

// A query further than this many L from the boundary takes its own distance as
// the unit of length for its step: in units of L its r^2 leaves FP32's range, and
// 1 / r loses its low part before.
constexpr float kRisFar = 0x1p30f;

// 1 / sqrt(a) for a normal a: the fast root y, corrected to second order in
// e = 1 - a y^2 (y (1 + e / 2 + 3 e^2 / 8); e ~ 1e-7).
__device__ __forceinline__ ff ff_rsqrt(ff a)
{
    const float y = rsqrt_ftz(a.hi);
    const ff t = ff_mul(a, two_prod(y, y));
    const float e = rn_sub(rn_sub(1.f, t.hi), t.lo);
    return fast_two_sum(y, rn_mul(rn_mul(y, e), rn_fma(0.375f, e, 0.5f)));
}

// 2^-e for 2^e <= d < 2^(e + 1), within FP32's normal range.
__device__ __forceinline__ float unit_of(float d)
{
    return __int_as_float(max(254 - (__float_as_int(d) >> 23), 1) << 23);
}

// K without its constant factor, at the candidate y of the vertex x (condition
// bx, bx < 0: the query), as float-float and in units of 2^s_e lengths (scale =
// 2^-s_e, about 1 / L, and alpha in these units: the powers of r stay in FP32's
// range on boundaries of any size): 1 / r (query, Dirichlet), r . n_x / r^3
// (Neumann), (r . n_x + alpha r^2) / r^3 (Robin).  Candidates closer than about L / 128 are left
// to ris_kernel_close: their K, the largest of all and cancelling the most (r . n_x
// falls as r^2), dominate the variance, and stay what FP64 gives for them.
constexpr float kRisClose2 = 0x1p-14f;

__device__ __forceinline__ ff ris_kernel(int bx, const FFPoint& x, const FFPoint& y, float scale,
                                         float alpha, bool& close)
{
    ff r[3];
    point_diff(y, x, r);
#pragma unroll
    for (int c = 0; c < 3; ++c) r[c] = {rn_mul(r[c].hi, scale), rn_mul(r[c].lo, scale)};
    const ff rr = ff_dot3(r, r);
    close = rr.hi < kRisClose2;
    // every condition's lanes together: alpha is 0 but on Robin parts
    const ff ri = ff_rsqrt(rr);
    const ff num = ff_add(ff_dot3(x.n, r), ff_mul_f(rr, bx == WOB_BC_ROBIN ? alpha : 0.f));
    const ff K = ff_mul(ff_mul(num, ri), ff_mul(ri, ri));
    return bx < 0 || bx == WOB_BC_DIRICHLET ? ri : K;
}

// The same value for a candidate within L / 128 of the vertex, all in FP64 and
// absolute coordinates; triangle jx and the uniforms ux (jx < 0: the query xq),
// jy and uy.  Rare (one candidate in 10^4 on a torus), and out of line.
__device__ __noinline__ ff ris_kernel_close(const WalkParams& p, int bx, int64_t jx, float2 ux,
                                            const float* xq, int64_t jy, float2 uy, float scale)
{
    auto point = [&](int64_t j, float2 u) {
        const double su = sqrt((double)u.x), u2 = (double)u.y;
        const double b0 = 1.0 - su, b1 = su * (1.0 - u2), b2 = su * u2;
        const int32_t* t = p.tris + 3 * j;
        const float *v0 = p.verts + 3 * (int64_t)t[0], *v1 = p.verts + 3 * (int64_t)t[1],
                    *v2 = p.verts + 3 * (int64_t)t[2];
        return make_double3(b0 * (double)v0[0] + b1 * (double)v1[0] + b2 * (double)v2[0],
                            b0 * (double)v0[1] + b1 * (double)v1[1] + b2 * (double)v2[1],
                            b0 * (double)v0[2] + b1 * (double)v1[2] + b2 * (double)v2[2]);
    };
    const double3 x = jx < 0 ? make_double3(xq[0], xq[1], xq[2]) : point(jx, ux), y = point(jy, uy);
    const double rx = y.x - x.x, ry = y.y - x.y, rz = y.z - x.z;
    const double r2 = rx * rx + ry * ry + rz * rz, rl = sqrt(r2);
    if (rl < 1e-12 * p.L) return {0.f, 0.f};
    if (bx < 0 || bx == WOB_BC_DIRICHLET) return ff_split(1.0 / (rl * (double)scale));
    const NormalArea n = p.tri_n[jx];
    double num = rx * n.nx + ry * n.ny + rz * n.nz;
    if (bx == WOB_BC_ROBIN) num += (double)p.alpha * r2;
    return ff_split(num / (r2 * rl * (double)scale * (double)scale));
}

// sl_data at y (uniforms su_u, u2 of its draw) with the point-source field in
// FP32 from a float-float difference and the normal derivative n . grad h in
// FP64 (it cancels where the field runs along the surface).
__device__ __forceinline__ double ris_data(const WalkParams& p, int64_t j, const FFPoint& y,
                                           float su_u, float u2, int bc)
{
    const DataDev& D = p.data;
    if (D.mode != WOB_DATA_POINT) {
        const double su = ff_join(ff_sqrt(su_u));
        double3 yd, nd;
        yd.x = (double)y.v0[0] + ff_join(y.p[0]);
        yd.y = (double)y.v0[1] + ff_join(y.p[1]);
        yd.z = (double)y.v0[2] + ff_join(y.p[2]);
        nd = make_double3(ff_join(y.n[0]), ff_join(y.n[1]), ff_join(y.n[2]));
        return sl_data(p, j, yd, 1.0 - su, su * (1.0 - (double)u2), su * (double)u2, nd, bc);
    }
    ff d[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) d[c] = ff_add(two_sum(y.v0[c], -D.x0[c]), y.p[c]);
    const float ri = rsqrtf(ff_dot3(d, d).hi);
    const float h = D.scale * ri;
    if (bc == WOB_BC_DIRICHLET) return (double)h;
    const float f = -h * ri * ri;
    double dhdn = 0.0;
#pragma unroll
    for (int c = 0; c < 3; ++c) dhdn = fma(ff_join(y.n[c]), (double)(f * d[c].hi), dhdn);
    return bc == WOB_BC_ROBIN ? dhdn + (double)p.alpha * (double)h : dhdn;
}

// The unit of length and |Gamma| / ris times the constant factors of K and the
// unit's powers.  Formed by the host: as three FP64 quotients in a row in the first
// thread of each block they took 2 of the 8.9 us of a call of two walks.
struct RisUnits {
    float unit, alpha;               // 1 / length; alpha in it
    double query, dirichlet, layer;  // G, (k / p_k) G, 2 dG/dn_x
};

RisUnits ris_units(const WalkParams& p)
{
    RisUnits u;
    u.unit = std::ldexp(1.f, -std::ilogb(p.L));
    u.alpha = p.alpha / u.unit;
    u.query = p.area / (double)p.ris / kFourPi * (double)u.unit;
    u.dirichlet = u.query * ((double)p.kmix / (double)p.pk);
    u.layer = 2.0 * u.query * (double)u.unit;
    return u;
}

template <bool DEBUG>
__global__ void __launch_bounds__(kRisThreads, kRisBlocks) k_sl_walks_ris(WalkParams p, RisUnits ru)
{
    const StreamKey key{p.key0, p.key1};
    const int64_t total = p.Q * (int64_t)p.N;
    const double phi = (double)p.phi;
    const float unit = ru.unit, alpha = ru.alpha;
    // each walk's sums and normal: in shared memory, off the candidates' registers
    enum { kSum, kProduct, kFirst };
    __shared__ double walk[3][kRisThreads];
    __shared__ volatile float normal[6][kRisThreads];  // n_x
    const int uniform_bc = p.kind == WOB_ROBIN_SL ? WOB_BC_ROBIN : WOB_BC_NEUMANN;
    ff wc[kMaxRis];
    const int lane = threadIdx.x & 31;
    // warp-uniform loop over groups of 32 consecutive walks
    for (int64_t base = blockIdx.x * (int64_t)blockDim.x + (threadIdx.x & ~31); base < total;
         base += (int64_t)gridDim.x * blockDim.x) {
        const int64_t idx = base + lane;
        const bool live = idx < total;
        const int64_t qi = live ? idx / p.N : 0;
        const int64_t wi = live ? idx - qi * p.N : 0;
        const uint32_t q = p.q_base + (uint32_t)qi;
        const uint32_t w = (uint32_t)(p.walk_begin + wi);
        const float* vertex = p.verts + 3 * (int64_t)__ldg(p.tris);
        float dist = 0.f;  // of the query from the boundary
        FFPoint x;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            x.v0[c] = p.queries[3 * qi + c];
            dist = fmaxf(dist, fabsf(x.v0[c] - __ldg(vertex + c)));
            x.p[c] = {0.f, 0.f};
            x.n[c] = {0.f, 0.f};
            normal[2 * c][threadIdx.x] = normal[2 * c + 1][threadIdx.x] = 0.f;
        }
        float scale = dist * unit > kRisFar ? unit_of(dist) : unit;
        int bx = -1;
        int32_t jx = -1;
        float ux = 0.f, u2x = 0.f;
        walk[kSum][threadIdx.x] = walk[kFirst][threadIdx.x] = 0.0;
        walk[kProduct][threadIdx.x] = 1.0;
        bool going = live;
        // every lane takes part in every step: a walk that stays, or has ended,
        // draws its candidates too and drops them (the warp would wait for the
        // others' all the same)
        for (int k = 0; k < p.M && __any_sync(kAllLanes, going); ++k) {
            bool stay = false;
            if (bx == WOB_BC_DIRICHLET) {
                const u32x4 u = stream_block(key, q, w, (uint32_t)k, kPurposeBranch, 0u, 0u);
                stay = u24f(u.x) >= p.pk;  // both exact in FP32
            }
            FFPoint y;
            ff sumw = {0.f, 0.f};
            float b0, b1, b2;
            for (int c = 0; c < p.ris; ++c) {
                __syncwarp();
                const u32x4 u = stream_block(key, q, w, (uint32_t)k, kPurposeArea, (uint32_t)c, 0u);
                const int64_t j = area_pick(p, u.x, u.y);
                __syncwarp();  // the searches differ in length
                frame_point_ff(p, j, u.z, u.w, y, b0, b1, b2);
                bool close;
#pragma unroll
                for (int d = 0; d < 3; ++d)
                    x.n[d] = {normal[2 * d][threadIdx.x], normal[2 * d + 1][threadIdx.x]};
                ff K = ris_kernel(bx, x, y, scale, alpha, close);
                if (close && going && !stay)
                    K = ris_kernel_close(p, bx, jx, make_float2(ux, u2x), p.queries + 3 * qi, j,
                                         make_float2(u24f(u.z), u24f(u.w)), scale);
                wc[c] = K;
                sumw = ff_add(sumw, K.hi < 0.f ? ff{-K.hi, -K.lo} : K);
            }
            __syncwarp();
            if (!stay && !(sumw.hi > 0.f)) going = false;  // every candidate has a zero kernel
            if (going) {
                double wfac;
                if (stay) {
                    wfac = 1.0 / (1.0 - (double)p.pk);
                } else {
                    u32x4 u = stream_block(key, q, w, (uint32_t)k, kPurposeRis, 0u, 0u);
                    // the 53-bit uniform as 24 + 29 bits
                    const ff t = ff_mul(fast_two_sum(rn_mul((float)(u.x >> 8), 0x1p-24f),
                                                     rn_mul((float)(((u.x & 0xFFu) << 21) | (u.y >> 11)),
                                                            0x1p-53f)),
                                        sumw);
                    ff acc = {0.f, 0.f};
                    int pick = p.ris - 1;
                    for (int c = 0; c < p.ris; ++c) {
                        const ff K = wc[c];
                        acc = ff_add(acc, K.hi < 0.f ? ff{-K.hi, -K.lo} : K);
                        if (acc.hi > t.hi || (acc.hi == t.hi && acc.lo > t.lo)) {
                            pick = c;
                            break;
                        }
                    }
                    u = stream_block(key, q, w, (uint32_t)k, kPurposeArea, (uint32_t)pick, 0u);
                    const int64_t j = area_pick(p, u.x, u.y);
                    frame_point_ff(p, j, u.z, u.w, y, b0, b1, b2);
                    // sign(K): positive for G, -phi sign(wc) on Neumann and Robin
                    // parts, negative on Dirichlet parts (and for a zero kernel)
                    const float sg = bx < 0 ? wc[pick].hi : bx == WOB_BC_DIRICHLET ? -1.f
                                                          : -(float)p.phi * wc[pick].hi;
                    double wk = bx < 0 ? ru.query : bx == WOB_BC_DIRICHLET ? ru.dirichlet : ru.layer;
                    if (scale != unit) {  // a far query's step is over
                        wk *= (double)scale / (double)unit;
                        scale = unit;
                    }
                    wfac = (sg > 0.f ? wk : -wk) * ff_join(sumw);
                    x = y;
#pragma unroll
                    for (int d = 0; d < 3; ++d) {
                        normal[2 * d][threadIdx.x] = y.n[d].hi;
                        normal[2 * d + 1][threadIdx.x] = y.n[d].lo;
                    }
                    jx = (int32_t)j;
                    ux = u24f(u.z);
                    u2x = u24f(u.w);
                }
                if (k == 0) walk[kFirst][threadIdx.x] = wfac; else walk[kProduct][threadIdx.x] *= wfac;
                const int by = p.bc_type ? (int)__ldg(p.bc_type + jx) : uniform_bc;
#pragma unroll
                for (int d = 0; d < 3; ++d)
                    x.n[d] = {normal[2 * d][threadIdx.x], normal[2 * d + 1][threadIdx.x]};
                const double dat = ris_data(p, jx, x, ux, u2x, by);
                double src = by == WOB_BC_DIRICHLET ? (double)p.kmix * dat : 2.0 * phi * dat;
                if (k == p.M - 1) src *= 0.5;
                walk[kSum][threadIdx.x] = fma(walk[kProduct][threadIdx.x], src, walk[kSum][threadIdx.x]);
                bx = by;
            }
        }
        const double value = walk[kFirst][threadIdx.x] * walk[kSum][threadIdx.x];
        if (live) {
            if (p.per_walk) p.per_walk[idx] = value;
            if (DEBUG && p.walk_flag) p.walk_flag[idx] = 0;
        }
        if (p.part) add_tile_partials(value, live, qi, wi, p.tpq, p.part);
    }
}

// Neumann walks through the direct boundary integral equation (Sec. 4.2):
// at a point x off the boundary u = phi (S q - int dG/dn_y u), on it
// u = 2 phi (S q - int dG/dn_y u).  Each vertex takes one area-uniform
// point x' for the source (|Gamma| G(x, x') q(x'), times c = phi off the
// boundary, 2 phi on it, halved at the last vertex x_M -- Sec. 4.1.2) and
// one line for the dG/dn_y term (weight phi (m/2) s from x0, phi m s from a
// boundary vertex, as the double-layer walks).  A query on triangle
// query_prim is boundary vertex 1 with weight 1.  One thread per walk.
template <bool DEBUG>
struct NdWalks : WalkTiles {
    using Base = WalkTiles;
    using Base::p;
    __device__ __forceinline__ explicit NdWalks(const WalkParams& p_) : Base(p_) {}
    template <class Mem>
    __device__ __forceinline__ void begin(const Mem& mem, LaneWalk& lw)
    {
        float3 x;
        const int64_t qi = Base::start(mem, lw, x);
        mem.set_x(0, {x.x, 0.f});
        mem.set_x(1, {x.y, 0.f});
        mem.set_x(2, {x.z, 0.f});
        mem.set(kAccS, 0.0);
        mem.set(kAccP, 1.0);
        lw.self = -1;
        lw.k = 0;
        lw.flag = 0;
        if (p.query_prim) {
            const int32_t prim = p.query_prim[qi];
            if (prim >= 0 && prim < p.T) {
                lw.self = p.inv_order[prim];
                lw.k = 1;
            }
        }
        if (DEBUG) {
            const LineOut lo = Base::lines(lw);
            for (int k = 0; k < p.M; ++k) lo.put(k, -1, -1, 0);
        }
    }
    // source at vertex k
    template <class Mem>
    __device__ __forceinline__ bool depart(const Mem& mem, const LaneWalk& lw) const
    {
        FFPoint y;
        float b0, b1, b2;
        const int64_t j = area_sample_ff(p, Base::key(lw), mem.q(), mem.w(), (uint32_t)lw.k, y, b0,
                                         b1, b2);
        float r2 = 0.f;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const float rc = ff_add(ff_sub({y.v0[c], 0.f}, mem.x(c)), y.p[c]).hi;
            r2 = __fmaf_rn(rc, rc, r2);
        }
        const float rmin2 = (float)(1e-24 * p.L * p.L);
        if (r2 >= rmin2) {
            const float f = sl_data_ff(p, j, y, b0, b1, b2, WOB_BC_NEUMANN);
            float c = (lw.k == 0) ? (float)p.phi : 2.f * (float)p.phi;
            if (lw.k == p.M) c *= 0.5f;
            const float G = 0.0795774715459476678f * rsqrt_ftz(r2);
            mem.set(kAccS, fma(mem.get(kAccP), (double)(c * (float)p.area * G * f), mem.get(kAccS)));
        }
        return lw.k < p.M;
    }
    // line from vertex k to vertex k + 1
    template <class Mem>
    __device__ __forceinline__ bool land(const Mem& mem, LaneWalk& lw, int m, int pos, int flag)
    {
        if (DEBUG) {
            lw.flag |= flag;
            Base::lines(lw).put(lw.k, m, pos >= 0 ? (int)prim_of(p.tv, pos) : -1, flag);
        }
        if (m == 0) return false;
        const double phi = (double)p.phi;
        const ff x[3] = {mem.x(0), mem.x(1), mem.x(2)};
        const ff d[3] = {mem.d(0), mem.d(1), mem.d(2)};
        ff y[3];
        const double ms = (double)(m * refine_hit_ff(p.tv, pos, x, d, y));
        mem.set(kAccP, mem.get(kAccP) * ((lw.k == 0) ? 0.5 * phi * ms : phi * ms));
#pragma unroll
        for (int c = 0; c < 3; ++c) mem.set_x(c, y[c]);
        lw.self = pos;
        ++lw.k;
        return true;
    }
    template <class Mem>
    __device__ __forceinline__ double value(const Mem& mem, const LaneWalk& lw) const
    {
        const double v = mem.get(kAccS);
        if (DEBUG) {
            const int64_t idx = Base::index(lw);
            if (p.per_walk) p.per_walk[idx] = v;
            if (p.walk_flag) p.walk_flag[idx] = (uint8_t)lw.flag;
        }
        return v;
    }
};

template <bool DEBUG>
__global__ void __launch_bounds__(kLineThreads, DEBUG ? kDebugBlocks : kNdBlocks) k_nd_lines(WalkParams p)
{
    __shared__ LineShared sm;
    extern __shared__ int line_stack[];
    int err = 0;
    WalkCount c{0, 0, 0, 0, 0};
    NdWalks<DEBUG> pol(p);
    run_lines<NdWalks<DEBUG>, false>(pol, sm.lane(line_stack), sm.vals, p.stack_levels, err, c);
    if (err) atomicOr(p.error_word, err);
}

__global__ void __launch_bounds__(kGroupThreads, kGroupBlocks) k_nd_groups(WalkParams p)
{
    __shared__ GroupShared sm;
    extern __shared__ int line_stack[];
    int err = 0;
    NdWalks<false> pol(p);
    run_line_groups(pol, sm, line_stack, p.stack_levels, err);
    if (err) atomicOr(p.error_word, err);
}

// ---------------------------------------------------------------------------
// Forward (adjoint) single-layer Neumann paths (Sec. 4.4.3).  With
// u(x) = int G(x, y) mu(y) dA, mu = T mu + f, T's kernel
// K(y, z) = -2 phi dG/dn_x(y, z) and f = 2 phi q, a path reads the truncated
// series sum_j c_j <G(x, .), T^j f> from its source end: z_0 ~ p on the
// boundary, a_0 = f(z_0) / p(z_0); from z_j a line (all hits, one picked,
// as the double-layer walks) gives z_{j+1} and K(z_{j+1}, z_j) / p = phi m s,
// so a_{j+1} = a_j phi m s; vertex j then contributes c_j a_j G(x, z_j) to
// every evaluation point x (c_j = 1, 1/2 for the last, Sec. 4.1.2).
// Streams: path p draws as query p, walk kForwardWalk.
// ---------------------------------------------------------------------------
constexpr uint32_t kForwardWalk = 0xFFFFFFFFu;

// Start weight of triangle j for boundary-value-weighted paths, first part:
// area x |q(centroid)|.
__global__ void k_fwd_qc(WalkParams p, double* __restrict__ aq)
{
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < p.T;
         j += (int64_t)gridDim.x * blockDim.x) {
        const int32_t* t = p.tris + 3 * j;
        double c[3] = {0.0, 0.0, 0.0};
        for (int k = 0; k < 3; ++k)
            for (int d = 0; d < 3; ++d) c[d] += (double)__ldg(p.verts + 3 * (int64_t)__ldg(t + k) + d);
        const double3 y = make_double3(c[0] / 3.0, c[1] / 3.0, c[2] / 3.0);
        const NormalArea na = p.tri_n[j];
        const double3 n = make_double3(na.nx, na.ny, na.nz);
        const double q = sl_data(p, j, y, 1.0 / 3.0, 1.0 / 3.0, 1.0 / 3.0, n, WOB_BC_NEUMANN);
        aq[j] = na.area * fabs(q);
    }
}

// ... second part: + beta mean|q| area (mean over the boundary, from the
// inclusive sums of the first part); inclusive sums of the result are the CDF.
__global__ void k_fwd_mix(WalkParams p, const double* __restrict__ aq_incl, double beta,
                          double* __restrict__ w)
{
    const double qbar = aq_incl[p.T - 1] / p.area;
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < p.T;
         j += (int64_t)gridDim.x * blockDim.x) {
        const double aq = aq_incl[j] - (j > 0 ? aq_incl[j - 1] : 0.0);
        w[j] = aq + beta * qbar * p.tri_n[j].area;
    }
}

// Start triangle, point and weight a_0 = 2 phi q(z_0) / p(z_0) of a path.
__device__ __forceinline__ int64_t fwd_start(const WalkParams& p, StreamKey key, uint32_t path,
                                             int start_mode, const double* wcdf, FFPoint& y, double& a)
{
    const double* cdf = start_mode == 1 ? wcdf : p.cdf;
    const double tot = start_mode == 1 ? wcdf[p.T - 1] : p.area;
    const u32x4 u = stream_block(key, path, kForwardWalk, 0u, kPurposeArea, 0u, 0u);
    const long long target = __double_as_longlong(u53(u.x, u.y) * tot);
    int64_t lo = 0, hi = p.T - 1;
    while (lo < hi) {
        const int64_t mid = lo + ((hi - lo) >> 1);
        if (__double_as_longlong(__ldg(cdf + mid)) > target) hi = mid; else lo = mid + 1;
    }
    float b0, b1, b2;
    frame_point_ff(p, lo, u.z, u.w, y, b0, b1, b2);
    const double pdf = start_mode == 1
                           ? ((cdf[lo] - (lo > 0 ? cdf[lo - 1] : 0.0)) / p.tri_n[lo].area) / tot
                           : 1.0 / p.area;
    a = 2.0 * (double)p.phi * (double)sl_data_ff(p, lo, y, b0, b1, b2, WOB_BC_NEUMANN, true) / pdf;
    return lo;
}

// The starts of every path, for the form with a lane per path: in the engine's
// hand-out the search and the FP64 quotients run for the few lanes that begin
// together (1e6 paths of two vertices on 1,280 triangles 698 -> 614 us with this
// kernel, of eight on 200,000 8.36 -> 7.40 ms; at most 97,000 paths, which begin
// together anyway, take 3 us more).  The triangle waits in the bits of the path's
// first coordinate, the weight in its first weight.
__global__ void __launch_bounds__(128) k_fwd_starts(WalkParams p, int64_t n, int start_mode,
                                                    const double* __restrict__ wcdf,
                                                    double* __restrict__ zpos, double* __restrict__ zw)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        FFPoint y;
        double a;
        const int64_t j =
            fwd_start(p, StreamKey{p.key0, p.key1}, (uint32_t)i, start_mode, wcdf, y, a);
        zpos[3 * i * p.M] = __longlong_as_double((long long)j);
        zw[i * p.M] = a;
    }
}

// The paths as the line engine's walks (p.Q x p.N = paths): a path's weight
// a_j waits in the first accumulator, its vertices and weights go to zpos
// and zw.  STARTED: after k_fwd_starts.
template <bool STARTED>
struct FwdPaths : WalkTiles {
    using Base = WalkTiles;
    using Base::p;
    int start_mode;
    const double* wcdf;
    double *zpos, *zw;
    uint8_t* flags;
    __device__ __forceinline__ FwdPaths(const WalkParams& p_, int start_mode_, const double* wcdf_,
                                        double* zpos_, double* zw_, uint8_t* flags_)
        : Base(p_), start_mode(start_mode_), wcdf(wcdf_), zpos(zpos_), zw(zw_), flags(flags_)
    {
    }
    template <class Mem>
    __device__ __forceinline__ void begin(const Mem& mem, LaneWalk& lw)
    {
        const uint32_t q = (uint32_t)Base::index(lw);
        mem.set_ids(q, kForwardWalk);
        FFPoint y;
        int64_t j;
        if (STARTED) {
            const int64_t r = Base::index(lw) * p.M;
            j = __double_as_longlong(zpos[3 * r]);
            mem.set(kAccS, zw[r]);
            const u32x4 u = stream_block(Base::key(lw), q, kForwardWalk, 0u, kPurposeArea, 0u, 0u);
            float b0, b1, b2;
            frame_point_ff(p, j, u.z, u.w, y, b0, b1, b2);
        } else {
            double a;
            j = fwd_start(p, Base::key(lw), q, start_mode, wcdf, y, a);
            mem.set(kAccS, a);
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) mem.set_x(c, ff_add({y.v0[c], 0.f}, y.p[c]));
        lw.self = p.inv_order[j];
        lw.k = 0;
        lw.flag = 0;
    }
    __device__ __forceinline__ void put(const LaneWalk& lw, int j, ff x, ff y, ff z, double w) const
    {
        const int64_t r = Base::index(lw) * p.M + j;
        zpos[3 * r] = ff_join(x);
        zpos[3 * r + 1] = ff_join(y);
        zpos[3 * r + 2] = ff_join(z);
        zw[r] = w;
    }
    template <class Mem>
    __device__ __forceinline__ bool depart(const Mem& mem, const LaneWalk& lw) const
    {
        const double a = mem.get(kAccS);
        const bool last = lw.k == p.M - 1;
        put(lw, lw.k, mem.x(0), mem.x(1), mem.x(2), last ? 0.5 * a : a);
        return !last;
    }
    template <class Mem>
    __device__ __forceinline__ bool land(const Mem& mem, LaneWalk& lw, int m, int pos, int flag)
    {
        lw.flag |= flag;
        if (m == 0) return false;
        const ff x[3] = {mem.x(0), mem.x(1), mem.x(2)};
        const ff d[3] = {mem.d(0), mem.d(1), mem.d(2)};
        ff y[3];
        const int s = refine_hit_ff(p.tv, pos, x, d, y);
        mem.set(kAccS, mem.get(kAccS) * ((double)p.phi * (double)(m * s)));
#pragma unroll
        for (int c = 0; c < 3; ++c) mem.set_x(c, y[c]);
        lw.self = pos;
        ++lw.k;
        return true;
    }
    // a path that a missed line ended: its remaining records are zero
    template <class Mem>
    __device__ __forceinline__ double value(const Mem&, const LaneWalk& lw) const
    {
        const ff zero = {0.f, 0.f};
        for (int j = lw.k + 1; j < p.M; ++j) put(lw, j, zero, zero, zero, 0.0);
        if (flags) flags[Base::index(lw)] = (uint8_t)lw.flag;
        return 0.0;
    }
    __device__ __forceinline__ void close(int, int, double) const {}
};

__global__ void __launch_bounds__(kLineThreads, kLineBlocks - 1)
    k_fwd_lines(WalkParams p, double* __restrict__ zpos, double* __restrict__ zw,
                uint8_t* __restrict__ flags)
{
    __shared__ LineShared sm;
    extern __shared__ int line_stack[];
    int err = 0;
    WalkCount c{0, 0, 0, 0, 0};
    FwdPaths<true> pol(p, 0, nullptr, zpos, zw, flags);
    run_lines<FwdPaths<true>, false>(pol, sm.lane(line_stack), sm.vals, p.stack_levels, err, c);
    if (err) atomicOr(p.error_word, err);
}

__global__ void __launch_bounds__(kGroupThreads, kGroupBlocks)
    k_fwd_groups(WalkParams p, int start_mode, const double* __restrict__ wcdf,
                 double* __restrict__ zpos, double* __restrict__ zw, uint8_t* __restrict__ flags)
{
    __shared__ GroupShared sm;
    extern __shared__ int line_stack[];
    int err = 0;
    FwdPaths<false> pol(p, start_mode, wcdf, zpos, zw, flags);
    run_line_groups(pol, sm, line_stack, p.stack_levels, err);
    if (err) atomicOr(p.error_word, err);
}

// Explicit connection of every path vertex to every query (an N-body sum):
// per query, v_p = sum_j w_pj G(x, z_pj) for each path, est = mean of v_p,
// var = their unbiased variance.
//
// k_fwd_pack turns each path into M float4 records (position, w / 4 pi; a
// vertex of weight 0 -- after a missed line -- sits far away with weight 0,
// so the inner loop needs no branch) and one live byte (0: every record of
// the path is 0, the path adds nothing but still counts in the mean).
// k_fwd_connect: work items are (block of kFwdThreads x kFwdQ queries, split
// of the paths); a persistent grid takes them in turn.  Whole paths are
// staged in shared memory; each thread keeps kFwdQ queries in registers as
// pairs, so one broadcast shared load feeds kFwdQ pairs and the distances,
// squared distances and the sum of w G run as packed FP32x2 operations (two
// queries per instruction, each lane rounded as the scalar operation would
// be), which leaves the reciprocal square roots (one MUFU operation per
// pair) as the bound; distances, G and v_p in FP32.
// The sums over paths run in FP32 for kFwdFold paths and are then folded into
// FP64 sums kept in shared memory (FP64 issues at 1/64 of the FP32 rate on
// this GPU: one FP64 add per path and query would cost as much as the
// pairs).  k_fwd_finish adds the
// splits' FP64 partial sums in a fixed order.
constexpr int kFwdTile = 1024;     // vertex records per tile (max_len <= kFwdTile)
constexpr int kFwdThreads = 128;
constexpr int kFwdQ = 8;           // queries per thread
static_assert(kFwdQ % 2 == 0, "queries are processed in pairs");
constexpr int kFwdFold = 32;       // paths summed in FP32 before an FP64 fold
constexpr float kFwdFar = 1e18f;   // |r|^2 ~ 3e36 stays finite in FP32

__global__ void k_fwd_pack(const double* __restrict__ zpos, const double* __restrict__ zw,
                           int64_t n_paths, int M, float4* __restrict__ rec,
                           uint8_t* __restrict__ live)
{
    constexpr double kInv4Pi = 0.0795774715459476678844418816862571810;
    for (int64_t path = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; path < n_paths;
         path += (int64_t)gridDim.x * blockDim.x) {
        int any = 0;
        for (int j = 0; j < M; ++j) {
            const int64_t r = path * M + j;
            const float w = (float)(zw[r] * kInv4Pi);
            rec[r] = w != 0.f ? make_float4((float)zpos[3 * r], (float)zpos[3 * r + 1],
                                            (float)zpos[3 * r + 2], w)
                              : make_float4(kFwdFar, kFwdFar, kFwdFar, 0.f);
            any |= w != 0.f;
        }
        live[path] = (uint8_t)any;
    }
}

__global__ void __launch_bounds__(kFwdThreads)
    k_fwd_connect(const float* __restrict__ queries, int64_t Q, const float4* __restrict__ rec_g,
                  const uint8_t* __restrict__ live_g, int64_t n_paths, int M, int64_t q_blocks,
                  int splits, int64_t per_split, double* __restrict__ part)
{
    __shared__ float4 rec[kFwdTile];
    __shared__ uint8_t live[kFwdTile];
    __shared__ double fsum[kFwdQ][kFwdThreads], fsq[kFwdQ][kFwdThreads];  // FP64 folds
    const int ppt = kFwdTile / M;  // whole paths per tile
    const int64_t items = q_blocks * splits;
    const int t = threadIdx.x;
    for (int64_t item = blockIdx.x; item < items; item += gridDim.x) {
        const int64_t qb = item % q_blocks;
        const int sp = (int)(item / q_blocks);
        const int64_t pb = (int64_t)sp * per_split;
        const int64_t pe = pb + per_split < n_paths ? pb + per_split : n_paths;
        // negated query coordinates, queries 2i and 2i + 1 in pair i: c - x
        // is computed as c + (-x), which rounds identically
        float2 nx[kFwdQ / 2], ny[kFwdQ / 2], nz[kFwdQ / 2];
        float s32[kFwdQ], ss32[kFwdQ];
#pragma unroll
        for (int k = 0; k < kFwdQ; ++k) {
            const int64_t qi = (qb * kFwdQ + k) * kFwdThreads + t;
            const bool ok = qi < Q;
            const float qx = ok ? -queries[3 * qi] : 0.f, qy = ok ? -queries[3 * qi + 1] : 0.f,
                        qz = ok ? -queries[3 * qi + 2] : 0.f;
            if (k & 1) {
                nx[k / 2].y = qx;
                ny[k / 2].y = qy;
                nz[k / 2].y = qz;
            } else {
                nx[k / 2].x = qx;
                ny[k / 2].x = qy;
                nz[k / 2].x = qz;
            }
            s32[k] = ss32[k] = 0.f;
            fsum[k][t] = fsq[k][t] = 0.0;
        }
        int cnt = 0;
        for (int64_t p0 = pb; p0 < pe; p0 += ppt) {
            const int np = (int)(pe - p0 < ppt ? pe - p0 : ppt);
            __syncthreads();
            for (int i = t; i < np * M; i += kFwdThreads) rec[i] = rec_g[p0 * M + i];
            for (int i = t; i < np; i += kFwdThreads) live[i] = live_g[p0 + i];
            __syncthreads();
            for (int pp = 0; pp < np; ++pp) {
                if (!live[pp]) continue;  // the same path for the whole block
                float2 v2[kFwdQ / 2];
#pragma unroll
                for (int k = 0; k < kFwdQ / 2; ++k) v2[k] = make_float2(0.f, 0.f);
                const float4* rp = rec + pp * M;
#pragma unroll 2
                for (int j = 0; j < M; ++j) {
                    const float4 c = rp[j];
                    const float2 cx = make_float2(c.x, c.x), cy = make_float2(c.y, c.y),
                                 cz = make_float2(c.z, c.z), cw = make_float2(c.w, c.w);
#pragma unroll
                    for (int k = 0; k < kFwdQ / 2; ++k) {
                        const float2 dx = __fadd2_rn(cx, nx[k]), dy = __fadd2_rn(cy, ny[k]),
                                     dz = __fadd2_rn(cz, nz[k]);
                        const float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
                        v2[k] = __ffma2_rn(cw, make_float2(rsqrt_ftz(r2.x), rsqrt_ftz(r2.y)), v2[k]);
                    }
                }
#pragma unroll
                for (int k = 0; k < kFwdQ; ++k) {
                    const float v = (k & 1) ? v2[k / 2].y : v2[k / 2].x;
                    s32[k] += v;
                    ss32[k] = fmaf(v, v, ss32[k]);
                }
                if (++cnt == kFwdFold) {
#pragma unroll
                    for (int k = 0; k < kFwdQ; ++k) {
                        fsum[k][t] += (double)s32[k];
                        fsq[k][t] += (double)ss32[k];
                        s32[k] = ss32[k] = 0.f;
                    }
                    cnt = 0;
                }
            }
        }
#pragma unroll
        for (int k = 0; k < kFwdQ; ++k) {
            const int64_t qi = (qb * kFwdQ + k) * kFwdThreads + t;
            if (qi < Q) {
                part[(2 * (int64_t)sp) * Q + qi] = fsum[k][t] + (double)s32[k];
                part[(2 * (int64_t)sp + 1) * Q + qi] = fsq[k][t] + (double)ss32[k];
            }
        }
    }
}

__global__ void k_fwd_finish(const double* __restrict__ part, int splits, int64_t Q,
                             int64_t n_paths, double* __restrict__ est, double* __restrict__ var,
                             const int* __restrict__ err)
{
    const bool bad = err && *err != 0;  // a path's line gave up
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < Q;
         q += (int64_t)gridDim.x * blockDim.x) {
        double sum = 0.0, sumsq = 0.0;
        for (int sp = 0; sp < splits; ++sp) {
            sum += part[(2 * (int64_t)sp) * Q + q];
            sumsq += part[(2 * (int64_t)sp + 1) * Q + q];
        }
        const double mean = sum / (double)n_paths;
        est[q] = bad ? __longlong_as_double(0x7FF8000000000000ll) : mean;
        var[q] = bad ? __longlong_as_double(0x7FF8000000000000ll)
                     : (n_paths > 1 ? fmax(sumsq - sum * mean, 0.0) / (double)(n_paths - 1)
                                    : 0.0);
    }
}

// Splits of the paths for k_fwd_connect: enough work items to fill every
// resident block slot, and a count of items close to a whole number of
// rounds of the persistent grid (the last round is the idle tail).
static int fwd_splits(int64_t q_blocks, int64_t max_splits, int64_t slots)
{
    int best = 1;
    double best_eff = -1.0;
    for (int s = 1; s <= 64 && s <= max_splits; ++s) {
        const int64_t items = q_blocks * s;
        const int64_t rounds = (items + slots - 1) / slots;
        const double eff = (double)items / (double)(rounds * slots);
        if (eff > best_eff + 0.02) {
            best_eff = eff;
            best = s;
        }
        if (eff >= 0.95) break;
    }
    return best;
}

// One warp per query: mean and unbiased variance in a fixed order.
// err (may be NULL): the solve's device check word; when a traversal check
// fired during the solve, every estimate of the call is NaN (the walk
// kernels themselves carry no per-walk check: it would cost registers in
// the traversal loop).
__device__ __forceinline__ bool solve_failed(const int* err) { return err && *err != 0; }

__global__ void k_reduce(const double* __restrict__ per_walk, int64_t Q, int32_t N,
                         double* __restrict__ est, double* __restrict__ var,
                         const int* __restrict__ err)
{
    const bool bad = solve_failed(err);
    const int lane = threadIdx.x & 31;
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t q = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5); q < Q;
         q += warps) {
        const double* v = per_walk + q * N;
        double s = 0.0;
        for (int i = lane; i < N; i += 32) s += v[i];
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
        const double mean = s / N;
        double ss = 0.0;
        for (int i = lane; i < N; i += 32) {
            const double e = v[i] - mean;
            ss = fma(e, e, ss);
        }
        for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xFFFFFFFFu, ss, o);
        if (lane == 0) {
            est[q] = bad ? __longlong_as_double(0x7FF8000000000000ll) : mean;
            var[q] = bad ? __longlong_as_double(0x7FF8000000000000ll)
                         : (N > 1 ? ss / (N - 1) : 0.0);
        }
    }
}

__global__ void k_reduce_accum(const double* __restrict__ per_walk, int64_t Q, int32_t N,
                               double* __restrict__ sum, double* __restrict__ sumsq,
                               const int* __restrict__ err)
{
    const double bad = solve_failed(err) ? __longlong_as_double(0x7FF8000000000000ll) : 0.0;
    const int lane = threadIdx.x & 31;
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t q = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5); q < Q;
         q += warps) {
        const double* v = per_walk + q * N;
        double s = 0.0, ss = 0.0;
        for (int i = lane; i < N; i += 32) {
            s += v[i];
            ss = fma(v[i], v[i], ss);
        }
        for (int o = 16; o > 0; o >>= 1) {
            s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
            ss += __shfl_xor_sync(0xFFFFFFFFu, ss, o);
        }
        if (lane == 0) {
            sum[q] += s + bad;
            sumsq[q] += ss + bad;
        }
    }
}

// One warp per query from the (sum, sum of squares) partials of its tpq
// 32-walk blocks: mean and unbiased variance, blocks combined in a fixed
// order (lane i takes blocks i, i + 32, ..., then a fixed shuffle tree).
__global__ void k_reduce_part(const double* __restrict__ part, int64_t Q, int32_t N, int32_t tpq,
                              double* __restrict__ est, double* __restrict__ var,
                              double* __restrict__ sum, double* __restrict__ sumsq,
                              const int* __restrict__ err)
{
    const bool bad = solve_failed(err);
    const int lane = threadIdx.x & 31;
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t q = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5); q < Q;
         q += warps) {
        const double2* pq = reinterpret_cast<const double2*>(part) + q * tpq;
        double s = 0.0, ss = 0.0;
        for (int i = lane; i < tpq; i += 32) {
            const double2 v = pq[i];
            s += v.x;
            ss += v.y;
        }
        for (int o = 16; o > 0; o >>= 1) {
            s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
            ss += __shfl_xor_sync(0xFFFFFFFFu, ss, o);
        }
        if (lane == 0) {
            const double nan = __longlong_as_double(0x7FF8000000000000ll);
            if (est) {
                const double mean = s / N;
                est[q] = bad ? nan : mean;
                var[q] = bad ? nan : (N > 1 ? fmax(ss - s * mean, 0.0) / (N - 1) : 0.0);
            }
            if (sum) {
                sum[q] += bad ? nan : s;
                sumsq[q] += bad ? nan : ss;
            }
        }
    }
}

__global__ void k_trace_lines(const float4* __restrict__ nodes, const float4* __restrict__ tv,
                              const int32_t* __restrict__ inv_order, int64_t n_tris,
                              int iter_limit, const double* __restrict__ o,
                              const double* __restrict__ d, const int32_t* __restrict__ exclude,
                              const uint32_t* __restrict__ keys, int64_t n, uint32_t key0,
                              uint32_t key1, float tauL, float edge_thr_L, int32_t* m,
                              int32_t* sum_s, int32_t* prim, int32_t* s_out, double* t_out,
                              double* y_out, uint8_t* flag, int* error_word)
{
    int err = 0;
    const StreamKey key{key0, key1};
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const double3 x = make_double3(o[3 * i], o[3 * i + 1], o[3 * i + 2]);
        const double3 dd = make_double3(d[3 * i], d[3 * i + 1], d[3 * i + 2]);
        const int ex = exclude ? exclude[i] : -1;
        const int self = (ex >= 0 && ex < n_tris) ? inv_order[ex] : -1;
        Trav t;
        const int pos = trace_line<true>(
            nodes, tv, make_float3((float)x.x, (float)x.y, (float)x.z),
            make_float3((float)dd.x, (float)dd.y, (float)dd.z), self, key, keys[3 * i],
            keys[3 * i + 1], keys[3 * i + 2], edge_thr_L, tauL, kGraze, t, err, iter_limit);
        m[i] = t.m;
        if (sum_s) sum_s[i] = t.sum_s;
        if (flag) flag[i] = (uint8_t)t.flag;
        int pr = -1, sg = 0;
        double tt = 0.0;
        double3 yy = make_double3(0.0, 0.0, 0.0);
        if (pos >= 0) {
            const Refined r = refine_hit(tv, pos, x, dd);
            pr = (int)prim_of(tv, pos);
            sg = r.s;
            yy = r.y;
            tt = (r.y.x - x.x) * dd.x + (r.y.y - x.y) * dd.y + (r.y.z - x.z) * dd.z;
        }
        if (prim) prim[i] = pr;
        if (s_out) s_out[i] = sg;
        if (t_out) t_out[i] = tt;
        if (y_out) {
            y_out[3 * i] = yy.x;
            y_out[3 * i + 1] = yy.y;
            y_out[3 * i + 2] = yy.z;
        }
    }
    if (err) atomicOr(error_word, err);
}

__global__ void k_line_axes(uint32_t key0, uint32_t key1, const uint32_t* __restrict__ qws,
                            int64_t n, double* __restrict__ d)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const double3 a = line_axis(StreamKey{key0, key1}, qws[3 * i], qws[3 * i + 1], qws[3 * i + 2]);
        d[3 * i] = a.x;
        d[3 * i + 1] = a.y;
        d[3 * i + 2] = a.z;
    }
}

__global__ void k_philox(const uint32_t* __restrict__ ctr, const uint32_t* __restrict__ keyv,
                         int64_t n, uint32_t* __restrict__ out)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const u32x4 r = philox4x32_10(ctr[4 * i], ctr[4 * i + 1], ctr[4 * i + 2], ctr[4 * i + 3],
                                      keyv[2 * i], keyv[2 * i + 1]);
        out[4 * i] = r.x;
        out[4 * i + 1] = r.y;
        out[4 * i + 2] = r.z;
        out[4 * i + 3] = r.w;
    }
}

}  // namespace

namespace {

// Launch a line-walk kernel (one lane per walk) with its traversal stacks in
// dynamic shared memory.
template <class K, class... Args>
int launch_lines(K kernel, const WalkParams& p, cudaStream_t s, Args... args)
{
    const size_t smem = line_stack_bytes(p.stack_levels, kLineThreads);
    kernel<<<grid_for((const void*)kernel, kLineThreads, smem, p.Q * (int64_t)p.N), kLineThreads,
             smem, s>>>(p, args...);
    WOB_CUDA_TRY(cudaGetLastError());
    return WOB_OK;
}

// The same for its form with kG lanes per walk.
template <class K, class... Args>
int launch_groups(K kernel, const WalkParams& p, cudaStream_t s, Args... args)
{
    const size_t smem = line_stack_bytes(p.stack_levels, kGroupThreads);
    kernel<<<grid_for((const void*)kernel, kGroupThreads, smem, kG * p.Q * (int64_t)p.N),
             kGroupThreads, smem, s>>>(p, args...);
    WOB_CUDA_TRY(cudaGetLastError());
    return WOB_OK;
}

// Too few walks to fill the GPU one lane each.
bool few_walks(const WalkParams& p)
{
    int dev = 0, sms = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return p.Q * (int64_t)p.N <= sms * kGroupWalksPerSm;
}

}  // namespace

int launch_dl_walks(const WalkParams& p, bool counted, bool debug, cudaStream_t s)
{
    if (p.per_walk_grad)
        return few_walks(p) ? launch_groups(k_dl_groups<true>, p, s)
                            : launch_lines(k_dl_lines<false, false, true>, p, s);
    if (counted) return launch_lines(k_dl_lines<true, true, false>, p, s);
    if (debug) return launch_lines(k_dl_lines<false, true, false>, p, s);
    return few_walks(p) ? launch_groups(k_dl_groups<false>, p, s)
                        : launch_lines(k_dl_lines<false, false, false>, p, s);
}

int launch_sl_walks(const WalkParams& p, bool debug, cudaStream_t s)
{
    const int threads = 128;
    static_assert(kRisThreads == threads, "one block size");
    const int64_t work = p.Q * (int64_t)p.N;
    if (p.ris > 1) {
        if (debug)
            k_sl_walks_ris<true><<<grid_for((const void*)k_sl_walks_ris<true>, threads, 0, work), threads, 0, s>>>(p, ris_units(p));
        else
            k_sl_walks_ris<false><<<grid_for((const void*)k_sl_walks_ris<false>, threads, 0, work), threads, 0, s>>>(p, ris_units(p));
    } else if (debug) {
        k_sl_walks_ff<true><<<grid_for((const void*)k_sl_walks_ff<true>, threads, 0, work), threads, 0, s>>>(p);
    } else {
        k_sl_walks_ff<false><<<grid_for((const void*)k_sl_walks_ff<false>, threads, 0, work), threads, 0, s>>>(p);
    }
    WOB_CUDA_TRY(cudaGetLastError());
    return WOB_OK;
}

int launch_nd_walks(const WalkParams& p, bool debug, cudaStream_t s)
{
    if (debug) return launch_lines(k_nd_lines<true>, p, s);
    return few_walks(p) ? launch_groups(k_nd_groups, p, s) : launch_lines(k_nd_lines<false>, p, s);
}

int launch_forward(const WalkParams& p, int64_t n_paths, int start_mode, double beta,
                   const float* queries, int64_t Q, double* zpos, double* zw, uint8_t* flags,
                   double* est, double* var, cudaStream_t s)
{
    double* buf = nullptr;  // aq, its sums, start weights, their sums: 4 x T doubles
    if (start_mode == 1) {
        WOB_CUDA_TRY(cudaMallocAsync((void**)&buf, 4 * p.T * sizeof(double), s));
        const int g = grid_for((const void*)k_fwd_qc, 256, 0, p.T);
        k_fwd_qc<<<g, 256, 0, s>>>(p, buf);
        int rc = inclusive_scan<double>(buf, buf + p.T, p.T, s);
        if (rc == WOB_OK) {
            k_fwd_mix<<<g, 256, 0, s>>>(p, buf + p.T, beta, buf + 2 * p.T);
            rc = inclusive_scan<double>(buf + 2 * p.T, buf + 3 * p.T, p.T, s);
        }
        if (rc != WOB_OK) {
            cudaFreeAsync(buf, s);
            return rc;
        }
    }
    const int threads = 128;
    WalkParams pp = p;  // the paths as the engine's walks
    pp.Q = 1;
    pp.N = (int32_t)n_paths;
    const double* start_cdf = buf ? buf + 3 * p.T : nullptr;
    int rc;
    if (few_walks(pp)) {
        rc = launch_groups(k_fwd_groups, pp, s, start_mode, start_cdf, zpos, zw, flags);
    } else {
        k_fwd_starts<<<grid_for((const void*)k_fwd_starts, threads, 0, n_paths), threads, 0, s>>>(
            pp, n_paths, start_mode, start_cdf, zpos, zw);
        rc = launch_lines(k_fwd_lines, pp, s, zpos, zw, flags);
    }
    if (buf) cudaFreeAsync(buf, s);
    if (rc == WOB_OK && Q > 0) {
        // packed records and live bytes, then (sum, sum of squares) per split and query
        const int64_t R = n_paths * p.M;
        const int64_t q_blocks = (Q + kFwdThreads * kFwdQ - 1) / (kFwdThreads * kFwdQ);
        const int ppt = kFwdTile / p.M;
        int dev = 0, sms = 1, per_sm = 1;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_fwd_connect, kFwdThreads,
                                                          0) != cudaSuccess ||
            per_sm < 1)
            per_sm = 1;
        const int64_t slots = (int64_t)sms * per_sm;
        const int splits = fwd_splits(q_blocks, (n_paths + ppt - 1) / ppt, slots);
        const int64_t per_split = (n_paths + splits - 1) / splits;
        const size_t rec_bytes = ((size_t)R * sizeof(float4) + 255) & ~(size_t)255;
        const size_t live_bytes = ((size_t)n_paths + 255) & ~(size_t)255;
        char* cb = nullptr;
        WOB_CUDA_TRY(cudaMallocAsync((void**)&cb,
                                     rec_bytes + live_bytes + 2 * splits * Q * sizeof(double), s));
        float4* rec = (float4*)cb;
        uint8_t* live = (uint8_t*)(cb + rec_bytes);
        double* part = (double*)(cb + rec_bytes + live_bytes);
        k_fwd_pack<<<grid_for((const void*)k_fwd_pack, threads, 0, n_paths), threads, 0, s>>>(
            zpos, zw, n_paths, p.M, rec, live);
        const int64_t items = q_blocks * splits;
        k_fwd_connect<<<(int)(items < slots ? items : slots), kFwdThreads, 0, s>>>(
            queries, Q, rec, live, n_paths, p.M, q_blocks, splits, per_split, part);
        k_fwd_finish<<<grid_for((const void*)k_fwd_finish, 256, 0, Q), 256, 0, s>>>(
            part, splits, Q, n_paths, est, var, p.error_word);
        if (cudaGetLastError() != cudaSuccess) rc = WOB_ERR_CUDA;
        cudaFreeAsync(cb, s);
    }
    if (rc != WOB_OK) set_error("forward paths failed");
    return rc;
}

int launch_reduce(const double* per_walk, int64_t Q, int32_t N, double* est, double* var,
                  cudaStream_t s, const int* err)
{
    const int threads = 256;
    k_reduce<<<grid_for((const void*)k_reduce, threads, 0, Q * 32), threads, 0, s>>>(
        per_walk, Q, N, est, var, err);
    WOB_CUDA_TRY(cudaGetLastError());
    return WOB_OK;
}

int launch_reduce_part(const double* part, int64_t Q, int32_t N, int32_t tpq, double* est,
                       double* var, double* sum, double* sumsq, cudaStream_t s, const int* err)
{
    const int threads = 256;
    k_reduce_part<<<grid_for((const void*)k_reduce_part, threads, 0, Q * 32), threads, 0, s>>>(
        part, Q, N, tpq, est, var, sum, sumsq, err);
    WOB_CUDA_TRY(cudaGetLastError());
    return WOB_OK;
}

int launch_reduce_accum(const double* per_walk, int64_t Q, int32_t N, double* sum, double* sumsq,
                        cudaStream_t s, const int* err)
{
    const int threads = 256;
    k_reduce_accum<<<grid_for((const void*)k_reduce_accum, threads, 0, Q * 32), threads, 0, s>>>(
        per_walk, Q, N, sum, sumsq, err);
    WOB_CUDA_TRY(cudaGetLastError());
    return WOB_OK;
}

int launch_trace_lines(const BvhDev& b, const double* o, const double* d, const int32_t* exclude,
                       const uint32_t* keys, int64_t n, uint32_t key0, uint32_t key1, float tauL,
                       float edge_thr_L, int32_t* m, int32_t* sum_s, int32_t* prim,
                       int32_t* s_out, double* t, double* y, uint8_t* flag, int* error_word,
                       cudaStream_t s)
{
    const int threads = 128;
    k_trace_lines<<<grid_for((const void*)k_trace_lines, threads, 0, n), threads, 0, s>>>(
        b.wnodes, b.tv, b.inv_order, b.mesh->T, (int)(4 * b.n_wide + 64), o, d,
        exclude, keys, n, key0, key1, tauL,
        edge_thr_L, m, sum_s, prim, s_out, t, y, flag, error_word);
    WOB_CUDA_TRY(cudaGetLastError());
    return WOB_OK;
}

int launch_line_axes(uint32_t key0, uint32_t key1, const uint32_t* qws, int64_t n, double* d,
                     cudaStream_t s)
{
    const int threads = 256;
    k_line_axes<<<grid_for((const void*)k_line_axes, threads, 0, n), threads, 0, s>>>(key0, key1, qws, n, d);
    WOB_CUDA_TRY(cudaGetLastError());
    return WOB_OK;
}

// Streaming read of n float4 (L1 bypassed), `passes` times; one atomic per
// warp keeps the loads.
__global__ void __launch_bounds__(256) k_probe_read(const float4* __restrict__ buf, int64_t n,
                                                    int passes, float* __restrict__ out)
{
    float acc = 0.f;
    for (int r = 0; r < passes; ++r)
        for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
             i += (int64_t)gridDim.x * blockDim.x) {
            const float4 v = __ldcg(buf + i);
            acc += (v.x + v.y) + (v.z + v.w);
        }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xFFFFFFFFu, acc, o);
    if ((threadIdx.x & 31) == 0) atomicAdd(out, acc);
}

int launch_probe_read(const float4* buf, int64_t n, int passes, float* out, cudaStream_t s)
{
    WOB_CUDA_TRY(cudaMemsetAsync(out, 0, sizeof(float), s));
    const int grid = grid_for((const void*)k_probe_read, 256, 0, (int64_t)1 << 40);
    k_probe_read<<<grid, 256, 0, s>>>(buf, n, passes, out);
    WOB_CUDA_TRY(cudaGetLastError());
    return WOB_OK;
}

int launch_philox(const uint32_t* ctr, const uint32_t* key, int64_t n, uint32_t* out,
                  cudaStream_t s)
{
    const int threads = 256;
    k_philox<<<grid_for((const void*)k_philox, threads, 0, n), threads, 0, s>>>(ctr, key, n, out);
    WOB_CUDA_TRY(cudaGetLastError());
    return WOB_OK;
}

}  // namespace wob
