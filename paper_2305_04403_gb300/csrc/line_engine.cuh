// line_engine.cuh -- the warp-level driver of the walks that follow lines.
//
// A walk is a serial chain of lines (axis, all-hits traversal, pick, refine),
// and lines take very different numbers of node visits (on the level-6 star
// 28.6 on average, up to about 60), so lanes that trace their k-th lines
// together wait for the longest of 32.  Here the lanes of a warp are
// decoupled: a warp alternates between phases that all 32 lanes reach
// together,
//   hand out   lanes without a walk take the next one of the warp's tiles;
//   axis       lanes that begin a line draw its axis;
//   nodes      lanes with nodes left visit them, one node per lane and turn,
//              until fewer than `need` lanes have work (line_busy_eighths);
//   leaves     the queued leaf triangles are tested;
//   land       lanes whose traversal is complete pick their hit, refine it
//              and add its term (the walk's own arithmetic, in the policy),
// and a lane that lands begins its next line while the others go on with
// theirs.  Waiting until most lanes have finished lets the landing phase
// (about 700 instructions) serve some two dozen lanes at a time, while the
// longest traversals go on beside the next lines.  Everything a lane does for
// its own walk is the same arithmetic in the same order whatever the other
// lanes do, so the values of the walks do not depend on the schedule.
//
// Tiles: a warp owns up to two tiles of 32 consecutive walks at a time (the
// one being handed out and the one whose last walks are still under way);
// values wait in shared memory until their tile is complete and are then
// summed in the fixed order of add_tile_partials.
//
// The state of a walk (point and axis as float-float pairs, the policy's
// accumulators, stream ids) and the traversal stack live in shared memory,
// structure of arrays; the node phase keeps only the six slab values of the
// line, the node, the queue and stack heights in registers.
//
// Measured against one thread per walk in lock step: the level-6 star slice
// (60.4 M lines: 7,374 queries x 512 walks x 16) 64.7 -> 39.5 ms, direct-BIE
// walks on the 200,000-triangle torus 40.1 -> 20.0 ms, 24 batched problems
// 31.3 -> 17.8 ms; 978 -> 532 warp instructions a line and 10.8 -> 17.3 lanes
// an instruction on the slice.  What bounds it now is the instruction issue
// (63% of cycles; L1 58%).  Earlier forms, on the slice: leaf references queued
// instead of (node, slots) entries 45.9 against 44.7 ms; 16-byte instead of
// 32-byte node loads 44.7 against 44.0 ms; 5 and 7 instead of 6 blocks per SM
// 46.6 and (values in local memory) 49.4 against 41.9 ms.
#pragma once

#include "node_stack.cuh"
#include "wob_device.cuh"

namespace wob {

constexpr unsigned kAllLanes = 0xFFFFFFFFu;
constexpr int kLineThreads = 128;  // threads of a block that runs the engine

constexpr int kNodeQ = 10;  // queued nodes with leaves to test, per lane

// Shared-memory slots of one walk (each array strided by S).
template <int S>
struct LaneMemT {
    volatile float* xd;      // 12: point hi, point lo, axis hi, axis lo
    volatile double* acc;    // the policy's accumulators
    volatile uint32_t* ids;  // 2: query and walk index of the lane's streams
    volatile int* lq;        // kNodeQ queued (node, leaf slots) entries
    volatile int* stack;     // one entry per level of the tree
    __device__ __forceinline__ float x_hi(int c) const { return xd[c * S]; }
    __device__ __forceinline__ float d_hi(int c) const { return xd[(6 + c) * S]; }
    __device__ __forceinline__ ff x(int c) const
    {
        return {xd[c * S], xd[(3 + c) * S]};
    }
    __device__ __forceinline__ ff d(int c) const
    {
        return {xd[(6 + c) * S], xd[(9 + c) * S]};
    }
    __device__ __forceinline__ void set_x(int c, ff v) const
    {
        xd[c * S] = v.hi;
        xd[(3 + c) * S] = v.lo;
    }
    __device__ __forceinline__ void set_d(int c, ff v) const
    {
        xd[(6 + c) * S] = v.hi;
        xd[(9 + c) * S] = v.lo;
    }
    __device__ __forceinline__ double get(int j) const { return acc[j * S]; }
    __device__ __forceinline__ void set(int j, double v) const { acc[j * S] = v; }
    __device__ __forceinline__ uint32_t q() const { return ids[0]; }
    __device__ __forceinline__ uint32_t w() const { return ids[S]; }
    __device__ __forceinline__ void set_ids(uint32_t q, uint32_t w) const
    {
        ids[0] = q;
        ids[S] = w;
    }
};

using LaneMem = LaneMemT<kLineThreads>;

// A block's shared memory: the accumulators of each thread and the values of
// each warp's two tiles.  The stack is dynamic shared memory.
struct LineShared {
    double acc[2 * kLineThreads];
    double vals[2 * kLineThreads];
    float xd[12 * kLineThreads];
    uint32_t ids[2 * kLineThreads];
    int lq[kNodeQ * kLineThreads];
    __device__ __forceinline__ LaneMem lane(int* stack)
    {
        const int t = threadIdx.x;
        return {xd + t, acc + t, ids + t, lq + t, stack + t};
    }
};

// Dynamic shared memory of a launch: a stack of one entry per level of the
// tree for each of a block's `threads`.  The deepest tree that is built (its binary
// tree has fewer than kStackSize levels) stays within the 48 KB that every
// kernel may use, so no launch changes a kernel's limit, which all threads share.
inline size_t line_stack_bytes(int levels, int threads) { return (size_t)levels * threads * sizeof(int); }
static_assert(sizeof(LineShared) + sizeof(int) * kStackSize * kLineThreads <= 48 * 1024,
              "static shared memory and the deepest tree's stacks");

// Header and quantised planes of a wide node, as two 32-byte loads (nodes are
// 96 bytes from an allocation's start: 32-byte aligned).
__device__ __forceinline__ void load_node(const float4* nd, float4& h, uint4& qx, uint4& qy, uint4& qz)
{
    uint32_t r[16];
#pragma unroll
    for (int i = 0; i < 2; ++i)
        asm("ld.global.nc.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
            : "=r"(r[8 * i]), "=r"(r[8 * i + 1]), "=r"(r[8 * i + 2]), "=r"(r[8 * i + 3]),
              "=r"(r[8 * i + 4]), "=r"(r[8 * i + 5]), "=r"(r[8 * i + 6]), "=r"(r[8 * i + 7])
            : "l"(nd + 2 * i));
    h = make_float4(__uint_as_float(r[0]), __uint_as_float(r[1]), __uint_as_float(r[2]),
                    __uint_as_float(r[3]));
    qx = make_uint4(r[4], r[5], r[6], r[7]);
    qy = make_uint4(r[8], r[9], r[10], r[11]);
    qz = make_uint4(r[12], r[13], r[14], r[15]);
}

// Registers of a lane's walk.
struct LaneWalk {
    int id;    // tile slot << 5 | walk of the tile
    int k;     // line of the walk (the step of its streams)
    int self;  // leaf position of the triangle the point lies on (-1: none)
    int flag;  // near-degenerate lines so far (debug solves)
};

// Where a line's traversal finds the geometry.
struct LineGeom {
    const float4* nodes;
    const float4* tv;
    float edge_thr_L, tauL, graze;
    int iter_limit;
};

// The hits of one line, by leaf position: hits[0 .. m-1] while m <= kMaxHits,
// afterwards hits[0] = the position of the smallest key so far, hits[1],
// hits[2] = that key.
__device__ __forceinline__ void add_hit(const float4* __restrict__ tv, int* hits, int& m, int pos,
                                        uint32_t prim, StreamKey key, uint32_t q, uint32_t w,
                                        uint32_t step)
{
    if (m < kMaxHits) {
        hits[m++] = pos;
        return;
    }
    uint64_t best = ~0ull;
    uint32_t bprim = 0xFFFFFFFFu;
    int bpos = -1;
    if (m == kMaxHits) {
        for (int i = 0; i < kMaxHits; ++i) {
            const uint32_t pr = prim_of(tv, hits[i]);
            keep_min(hit_key(key, q, w, step, pr), pr, hits[i], best, bprim, bpos);
        }
    } else {
        bpos = hits[0];
        bprim = prim_of(tv, bpos);
        best = ((uint64_t)(uint32_t)hits[1] << 32) | (uint32_t)hits[2];
    }
    keep_min(hit_key(key, q, w, step, prim), prim, pos, best, bprim, bpos);
    hits[0] = bpos;
    hits[1] = (int)(best >> 32);
    hits[2] = (int)best;
    ++m;
}

__device__ __forceinline__ int pick_hit(const float4* __restrict__ tv, const int* hits, int m,
                                        StreamKey key, uint32_t q, uint32_t w, uint32_t step)
{
    if (m == 1 || m > kMaxHits) return hits[0];
    uint64_t best = ~0ull;
    uint32_t bprim = 0xFFFFFFFFu;
    int bpos = -1;
    for (int i = 0; i < m; ++i) {
        const uint32_t pr = prim_of(tv, hits[i]);
        keep_min(hit_key(key, q, w, step, pr), pr, hits[i], best, bprim, bpos);
    }
    return bpos;
}

// The node phase goes on while this many eighths of the live lanes have nodes to
// visit: one (until the last lane is done) in trees of up to six levels, where a
// line's visits differ by little and the landing phase counts for more, two in
// deeper ones.  At four, with which lanes land sooner but fewer together, 1.05e6
// walks of four lines took 1.26, 1.09, 0.98, 0.93, 0.85 and 0.76 of the lock-step
// time on 2 to 7 levels (20 to 81,920 triangles), and take 1.04, 0.88, 0.83, 0.86,
// 0.79 and 0.70 with this rule.
__device__ __forceinline__ int line_busy_eighths(int levels) { return levels <= 6 ? 1 : 2; }

// Run the policy's walks to the end.  The policy P provides
//   bool fetch(int slot, int& cnt)     (whole warp) the next tile into slot
//   StreamKey key(const LaneWalk&)     streams of the lane's problem
//   LineGeom geom(const LaneWalk&)
//   void begin(mem, lw)                start the walk lw.id at its first vertex
//   bool depart(mem, lw)               at a vertex: true if the line lw.k leaves it
//   bool land(mem, lw, m, pos, flag)   the line lw.k ended (m hits, pos picked,
//                                      -1 if none); true: at the next vertex
//   double value(mem, lw)              the finished walk's value
//   void close(int slot, int cnt, double v)   (whole warp) a tile is complete
template <class P, bool COUNT>
__device__ __forceinline__ void run_lines(P& pol, const LaneMem mem, double* block_vals, int levels,
                                          int& err, WalkCount& c)
{
    const int busy_eighths = line_busy_eighths(levels);
    const int lane = threadIdx.x & 31;
    double* vals = block_vals + 2 * (threadIdx.x & ~31);  // of the warp's two tiles
    unsigned todo0 = 0, todo1 = 0;  // unfinished walks of the tile slots
    int cnt0 = 0, cnt1 = 0;
    int cur = 1, next = 0;          // walks cur .. of the slot being handed out
    bool more = true;
    // lane state
    LaneWalk lw{0, 0, -1, 0};
    bool live = false, trav = false, fresh = false;
    int node = 0, sp = 0, nq = 0, iters = 0, m = 0, flag = 0;
    int hits[kMaxHits];

    while (true) {
        // ---- hand out
        unsigned idle = __ballot_sync(kAllLanes, !live);
        while (idle && more) {
            const int have = cur ? cnt1 : cnt0;
            if (next >= have) {
                if ((cur ? todo0 : todo1) != 0u) break;  // both tiles under way
                int cnt = 0;
                more = pol.fetch(cur ^ 1, cnt);
                if (!more) break;
                cur ^= 1;
                next = 0;
                const unsigned all = cnt == 32 ? kAllLanes : (1u << cnt) - 1u;
                if (cur) {
                    cnt1 = cnt;
                    todo1 = all;
                } else {
                    cnt0 = cnt;
                    todo0 = all;
                }
                continue;
            }
            const int r = next + __popc(idle & ((1u << lane) - 1u));
            if (!live && r < have) {
                live = true;
                lw.id = (cur << 5) | r;
                pol.begin(mem, lw);
                fresh = true;
            }
            next += __popc(idle);
            idle = __ballot_sync(kAllLanes, !live);
        }
        const unsigned livem = __ballot_sync(kAllLanes, live);
        if (livem == 0u) break;
        const StreamKey key = pol.key(lw);
        const LineGeom g = pol.geom(lw);
        // ---- axis
        if (fresh) {
            trav = pol.depart(mem, lw);
            node = sp = nq = iters = flag = 0;
            m = trav ? 0 : -1;  // -1: the walk ends here, without a line
            if (trav) {
                ff d[3];
                line_axis_ff(key, mem.q(), mem.w(), (uint32_t)lw.k, d);
#pragma unroll
                for (int j = 0; j < 3; ++j) mem.set_d(j, d[j]);
            }
            fresh = false;
        }
        // (for every lane: a value kept for some would live through the landing)
        const float ix = guard_inv(mem.d_hi(0)), iy = guard_inv(mem.d_hi(1)),
                    iz = guard_inv(mem.d_hi(2));
        const float oix = mem.x_hi(0) * ix, oiy = mem.x_hi(1) * iy, oiz = mem.x_hi(2) * iz;
        // ---- nodes
        const int n_live = __popc(livem);
        const int need = (n_live * busy_eighths + 7) >> 3;
        while (true) {
            const bool can = trav && nq < kNodeQ;
            const unsigned busy = __ballot_sync(kAllLanes, can);
            if (__popc(busy) < need || busy == 0u) break;
            if (can) {
                if (++iters > g.iter_limit) {  // each node is visited at most once per line
                    err |= 2;
                    trav = false;
                } else {
                    const float4* nd = g.nodes + 6 * node;
                    float4 h;
                    uint4 qx, qy, qz;
                    load_node(nd, h, qx, qy, qz);
                    int base = __ldg(reinterpret_cast<const int*>(nd + 4));
                    const uint32_t hit = node_hits(h, qx, qy, qz, ix, iy, iz, oix, oiy, oiz);
                    const int nint = (__float_as_uint(h.w) >> 24) & 15;
                    uint32_t im = hit & ((1u << nint) - 1u);  // interior children
                    if (hit != im) {                          // leaf children: queue them
                        mem.lq[nq * kLineThreads] = (int)((uint32_t)node << 8 | (hit ^ im));
                        ++nq;
                    }
                    if (!im && sp > 0) {
                        const uint32_t e = (uint32_t)mem.stack[--sp * kLineThreads];
                        base = (int)(e & 0xFFFFFFu);
                        im = e >> 24;
                    }
                    if (im) {
                        node = base + __ffs(im) - 1;
                        im &= im - 1;
                        if (im) {
                            if (sp < levels) {
                                mem.stack[sp * kLineThreads] = base | (int)(im << 24);
                                ++sp;
                            } else {
                                err |= 1;
                            }
                        }
                    } else {
                        trav = false;
                    }
                }
            }
        }
        // ---- leaves
        if (nq > 0) {
            const LineShear L = line_shear(make_float3(mem.x_hi(0), mem.x_hi(1), mem.x_hi(2)),
                                           make_float3(mem.d_hi(0), mem.d_hi(1), mem.d_hi(2)));
            const float Tthr = g.edge_thr_L * fabsf(L.Sz);
            // the queue's (node, leaf slots) entries, one leaf at a time
            uint32_t slots = 0;
            const int* refs = nullptr;
            for (int i = 0; i < nq || slots;) {
                if (!slots) {
                    const uint32_t e = (uint32_t)mem.lq[i++ * kLineThreads];
                    slots = e & 255u;
                    refs = reinterpret_cast<const int*>(g.nodes + 6 * (e >> 8) + 4);
                }
                const int ref = __ldg(refs + __ffs(slots) - 1);
                slots &= slots - 1;
                const int first = leaf_first(ref), last = first + leaf_count(ref);
                for (int p = first; p < last; ++p) {
                    if (p == lw.self) continue;
                    const float4 a4 = __ldg(g.tv + 3 * p + 0);
                    const float4 b4 = __ldg(g.tv + 3 * p + 1);
                    const float4 c4 = __ldg(g.tv + 3 * p + 2);
                    if (COUNT) c.tris++;
                    float tl = 0.f;
                    if (line_tri(a4, b4, c4, L, Tthr, g.tauL, g.graze, flag, tl))
                        add_hit(g.tv, hits, m, p, __float_as_uint(a4.w), key, mem.q(), mem.w(),
                                (uint32_t)lw.k);
                }
            }
        }
        nq = 0;
        __syncwarp();
        // ---- land
        bool ended = false;
        if (live && !trav) {
            if (m >= 0) {
                if (COUNT) {
                    c.lines++;
                    c.nodes += iters;
                    c.hits += m;
                    c.flag += flag;
                }
                const int pos =
                    m > 0 ? pick_hit(g.tv, hits, m, key, mem.q(), mem.w(), (uint32_t)lw.k) : -1;
                fresh = pol.land(mem, lw, m, pos, flag);
                ended = !fresh;
            } else {
                ended = true;
            }
            if (ended) {
                vals[lw.id] = pol.value(mem, lw);
                live = false;
            }
        }
        // ---- complete tiles
        if (__any_sync(kAllLanes, ended)) {
            const unsigned bit = ended ? 1u << (lw.id & 31) : 0u;
            const unsigned e0 = __reduce_or_sync(kAllLanes, lw.id < 32 ? bit : 0u);
            const unsigned e1 = __reduce_or_sync(kAllLanes, lw.id >= 32 ? bit : 0u);
            __syncwarp();
            if (e0 && !(todo0 &= ~e0)) pol.close(0, cnt0, lane < cnt0 ? vals[lane] : 0.0);
            if (e1 && !(todo1 &= ~e1)) pol.close(1, cnt1, lane < cnt1 ? vals[32 + lane] : 0.0);
            __syncwarp();
        }
    }
}

// ---------------------------------------------------------------------------
// The same walks for calls with too few of them to fill the GPU: G lanes
// follow one line (lane j tests children j, j + G, ... of each wide node, and
// the queued triangles are tested G at a time), and a block of 32 G threads
// runs one tile of 32 walks.  A node visit is then a shorter chain of
// instructions and a call of a few thousand walks has G times the warps; the
// price is the landing phase, which runs on one lane of G.  Same box and
// triangle tests, same hits, same arithmetic per walk: the same values.
// 16,384 walks of 4 lines on 1,280 triangles take 90 us; with the stack shared
// by the group and a barrier between its pop and its push 97 us, and in that form
// without the barrier 92 us against 151 with a lane per walk, 100 with 2 lanes and
// 113 with 8 (two warps of four lanes each for every walk's warp, without
// splitting the nodes: 169 us).
// ---------------------------------------------------------------------------
constexpr int kG = 4;                       // lanes per walk: 2, 4 or 8
constexpr int kGroups = 32;                 // walks of a block: one tile
constexpr int kGroupThreads = kG * kGroups;
constexpr int kGroupQ = 40;                 // queued leaf references per walk
constexpr unsigned kGroupMask = (1u << kG) - 1u;
using GroupMem = LaneMemT<kGroups>;

struct GroupShared {
    double acc[2 * kGroups];
    double vals[kGroups];
    float xd[12 * kGroups];
    uint32_t ids[2 * kGroups];
    int lq[kGroupQ * kGroups];
    int hits[kGroups][kMaxHits];
    unsigned long long tile;
};
static_assert(sizeof(GroupShared) + sizeof(int) * kStackSize * kGroupThreads <= 48 * 1024,
              "static shared memory and the deepest tree's stacks");

template <class P>
__device__ __forceinline__ void run_line_groups(P& pol, GroupShared& sm, int* stack_base, int levels,
                                                int& err)
{
    const int lane = threadIdx.x & 31, j = lane & (kG - 1), gsh = lane & ~(kG - 1);
    const int grp = threadIdx.x / kG;  // the walk of the tile this lane works for
    // (the stack is this lane's: next_node)
    const GroupMem mem{sm.xd + grp, sm.acc + grp, sm.ids + grp, sm.lq + grp, stack_base + threadIdx.x};
    int* hits = sm.hits[grp];
    while (true) {
        int cnt = 0;
        if (!pol.fetch_block(&sm.tile, cnt)) break;
        LaneWalk lw{grp, 0, -1, 0};
        bool alive = grp < cnt;
        if (alive && j == 0) pol.begin(mem, lw);
        const StreamKey key = pol.key(lw);
        const LineGeom g = pol.geom(lw);
        while (__any_sync(kAllLanes, alive)) {
            // the leader's point and axis, read by its group
            int go = 0;
            if (alive && j == 0) {
                go = pol.depart(mem, lw);
                if (go) {
                    ff d[3];
                    line_axis_ff(key, mem.q(), mem.w(), (uint32_t)lw.k, d);
#pragma unroll
                    for (int c = 0; c < 3; ++c) mem.set_d(c, d[c]);
                }
            }
            __syncwarp();
            go = __shfl_sync(kAllLanes, go, gsh);
            lw.self = __shfl_sync(kAllLanes, lw.self, gsh);
            lw.k = __shfl_sync(kAllLanes, lw.k, gsh);
            const float3 o = make_float3(mem.x_hi(0), mem.x_hi(1), mem.x_hi(2));
            const float3 d = make_float3(mem.d_hi(0), mem.d_hi(1), mem.d_hi(2));
            bool trav = go != 0;
            int node = 0, sp = 0, nq = 0, iters = 0, m = 0, flag = 0;
            const float ix = guard_inv(trav ? d.x : 1.f), iy = guard_inv(trav ? d.y : 1.f),
                        iz = guard_inv(trav ? d.z : 1.f);
            const float oix = o.x * ix, oiy = o.y * iy, oiz = o.z * iz;
            while (true) {
                // nodes, until the lines have no more or a queue could run over
                while (__any_sync(kAllLanes, trav) && __all_sync(kAllLanes, nq <= kGroupQ - 8)) {
                    if (trav && ++iters > g.iter_limit) {
                        err |= 2;
                        trav = false;
                    }
                    uint32_t mine = 0;  // hit children of this lane, bit i: child j + kG i
                    int nint = 0, base = 0;
                    const float4* nd = g.nodes + 6 * node;
                    if (trav) {
                        float4 h;
                        uint4 qx, qy, qz;
                        load_node(nd, h, qx, qy, qz);
                        base = __ldg(reinterpret_cast<const int*>(nd + 4));  // first interior child
                        nint = (__float_as_uint(h.w) >> 24) & 15;
                        mine = lane_children<kG>(h, qx, qy, qz, j, ix, iy, iz, oix, oiy, oiz);
                    }
                    uint32_t hitm = 0;
#pragma unroll
                    for (int i = 0; i < 8 / kG; ++i)
                        hitm |= ((__ballot_sync(kAllLanes, (mine >> i) & 1u) >> gsh) & kGroupMask) << (kG * i);
                    if (trav) {
                        const uint32_t im = hitm & ((1u << nint) - 1u);
                        const uint32_t lm = hitm ^ im;
                        if (lm) {
#pragma unroll
                            for (int i = 0; i < 8 / kG; ++i) {
                                const int c = j + kG * i;
                                if ((lm >> c) & 1u)
                                    mem.lq[(nq + __popc(lm & ((1u << c) - 1u))) * kGroups] =
                                        __ldg(reinterpret_cast<const int*>(nd + 4) + c);
                            }
                            nq += __popc(lm);
                        }
                        trav = next_node(mem.stack, kGroupThreads, levels, base, im, sp, node, err);
                    }
                }
                __syncwarp();
                // the queued leaves, kG at a time
                // (point and axis read again: six registers fewer in the node phase)
                const LineShear L = line_shear(make_float3(mem.x_hi(0), mem.x_hi(1), mem.x_hi(2)),
                                               make_float3(mem.d_hi(0), mem.d_hi(1), mem.d_hi(2)));
                const float Tthr = g.edge_thr_L * fabsf(L.Sz);
                for (int i0 = 0; __any_sync(kAllLanes, i0 < nq); i0 += kG) {
                    const bool have = i0 + j < nq;
                    const int ref = have ? mem.lq[(i0 + j) * kGroups] : 0;
                    const int first = have ? leaf_first(ref) : 0, count = have ? leaf_count(ref) : 0;
                    for (int t = 0; __any_sync(kAllLanes, t < count); ++t) {
                        const int p = first + t;
                        bool hit = false;
                        uint32_t prim = 0;
                        if (t < count && p != lw.self) {
                            const float4 a4 = __ldg(g.tv + 3 * p + 0);
                            const float4 b4 = __ldg(g.tv + 3 * p + 1);
                            const float4 c4 = __ldg(g.tv + 3 * p + 2);
                            float tl = 0.f;
                            hit = line_tri(a4, b4, c4, L, Tthr, g.tauL, g.graze, flag, tl);
                            prim = __float_as_uint(a4.w);
                        }
                        uint32_t hm = (__ballot_sync(kAllLanes, hit) >> gsh) & kGroupMask;
                        if (m + __popc(hm) <= kMaxHits) {
                            if (hit) hits[m + __popc(hm & ((1u << j) - 1u))] = p;
                            m += __popc(hm);
                        } else {  // more hits than recorded: one after the other
                            __syncwarp(kGroupMask << gsh);
                            while (hm) {
                                const int from = __ffs(hm) - 1;
                                hm &= hm - 1;
                                if (j == from)
                                    add_hit(g.tv, hits, m, p, prim, key, mem.q(), mem.w(), (uint32_t)lw.k);
                                else
                                    ++m;
                                __syncwarp(kGroupMask << gsh);
                            }
                        }
                    }
                }
                __syncwarp();
                nq = 0;
                if (!__any_sync(kAllLanes, trav)) break;
            }
            flag = ((__ballot_sync(kAllLanes, flag != 0) >> gsh) & kGroupMask) != 0u;
            // land
            if (alive && j == 0) {
                bool more = false;
                if (go) {
                    const int pos =
                        m > 0 ? pick_hit(g.tv, hits, m, key, mem.q(), mem.w(), (uint32_t)lw.k) : -1;
                    more = pol.land(mem, lw, m, pos, flag);
                }
                if (!more) {
                    sm.vals[grp] = pol.value(mem, lw);
                    alive = false;
                }
            }
            __syncwarp();
            alive = __shfl_sync(kAllLanes, alive, gsh);
        }
        __syncthreads();
        if (threadIdx.x < 32) pol.close(0, cnt, lane < cnt ? sm.vals[lane] : 0.0);
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// The double-layer recursion (Sec. 4.1.1-4.1.2, ray sampling of Sec. 4.4.1)
// as the engine's vertex rules.  Accumulators: S (sum of terms) and P (phi x
// weight product) in FP64.
// ---------------------------------------------------------------------------
enum { kAccS = 0, kAccP };

// Start at x.  start_pos >= 0: x lies on that triangle (leaf position) and
// the walk estimates the density nu(x) (Eq. indirect_double_boundary_
// reordered2): x is vertex 1 with weight 1 and lines 1 .. M-1 follow.
template <class Mem>
__device__ __forceinline__ void dl_begin(const Mem& mem, LaneWalk& lw, float3 x, int start_pos,
                                         const DataDev& D, const float4* __restrict__ tv,
                                         double phi, int M)
{
    mem.set_x(0, {x.x, 0.f});
    mem.set_x(1, {x.y, 0.f});
    mem.set_x(2, {x.z, 0.f});
    mem.set(kAccS, 0.0);
    mem.set(kAccP, phi);
    lw.self = -1;
    lw.k = 0;
    lw.flag = 0;
    if (start_pos >= 0) {
        mem.set(kAccS, ((M == 1) ? phi : 2.0 * phi) * (double)dl_data_f(D, tv, start_pos, x));
        lw.self = start_pos;
        lw.k = 1;
    }
}

// The line lw.k landed on leaf position pos as one of m hits: refine in
// float-float and accumulate (weight product and sum in FP64).
template <class Mem>
__device__ __forceinline__ void dl_land(const Mem& mem, LaneWalk& lw, int m, int pos,
                                        const DataDev& D, const float4* __restrict__ tv,
                                        double phi, int M)
{
    const ff x[3] = {mem.x(0), mem.x(1), mem.x(2)};
    const ff d[3] = {mem.d(0), mem.d(1), mem.d(2)};
    ff y[3];
    const int ms = m * refine_hit_ff(tv, pos, x, d, y);
    // P: the weight times phi (k = 0: (m/2) s phi); a factor of one hit is a
    // change of sign, off the FP64 pipe
    const bool neg = lw.k == 0 ? (ms < 0) != (phi < 0.0) : (ms > 0) == (phi > 0.0);
    double P = lw.k == 0 ? 0.5 : mem.get(kAccP);
    if (m > 1) P *= (double)m;
    P = __hiloint2double(__double2hiint(P) ^ (neg ? 0x80000000 : 0), __double2loint(P));
    const double g = (double)dl_data_f(D, tv, pos, make_float3(y[0].hi, y[1].hi, y[2].hi));
    const double P2 = lw.k == M - 1 ? P : P + P;
    mem.set(kAccS, fma(P2, g, mem.get(kAccS)));
    mem.set(kAccP, P);
#pragma unroll
    for (int c = 0; c < 3; ++c) mem.set_x(c, y[c]);
    lw.self = pos;
    ++lw.k;
}

}  // namespace wob
