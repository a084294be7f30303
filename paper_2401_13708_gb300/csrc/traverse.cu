// traverse.cu -- Barnes-Hut repulsion (Sec. 4.2, Eq. CellApproximation) and
// the exact O(n^2) repulsion (Eq. KlGradientHyperbolicSplit, second sum).
//
// Warp-cooperative tree walk.  A warp takes 32 consecutive points in key
// order (neighbouring cells, so the lanes' walks overlap) and visits the
// pre-order node array with one warp-uniform cursor:
//   - at an internal cell every active lane tests its own criterion
//     r_cell / d(y_i, y_cell) < theta, written as delta_i,cell > thr_cell
//     with thr = cosh(r_cell / theta) - 1 (cosh is increasing, so the test is
//     exact and needs no transcendental);  a lane that accepts adds the cell
//     term N_cell w^2 d dd/dy_i and becomes inactive until the cursor leaves
//     the cell's subtree (pre-order index >= skip);
//   - the warp descends (cursor + 1) if any active lane rejected the cell,
//     otherwise it jumps to skip;
//   - leaves add the exact pair term for every active lane, except the lane
//     whose own point it is; depth-29 buckets add each of their points.
// Each lane therefore accumulates exactly the terms of its own depth-first
// walk; the warp visits the union of the 32 walks.  Node loads are
// warp-uniform (one sector, broadcast) and stay in L1/L2.
//
// Per lane the pair term is reduced to a scalar times (Delta, s) and a w
// for Z (see pair_terms_* in hts_internal.cuh); the result per point is
//   F_rep,i = 4 il_i (R_Delta + il_i R_s y_i),   Z_i = sum N w,
// written to the point's original index.
#include <limits.h>

#include <algorithm>

#include "hts_internal.cuh"

namespace hts {
namespace {

constexpr int kWalkBlock = 256;
#ifndef LB
#define LB 128
#endif
constexpr int kListBlock = LB;
constexpr int kExactBlock = 64;

// One node, read through the non-coherent path: a single 256-bit load (the
// node array comes from cudaMalloc and a node is 32 bytes, so every node is
// 32-byte aligned); two 128-bit loads measured 2% slower.
__device__ __forceinline__ NodeF load_node(const NodeF *__restrict__ nodes, int k)
{
    NodeF r;
    float skipf;
    asm("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=f"(r.xh), "=f"(r.yh), "=f"(r.xl), "=f"(r.yl), "=f"(r.il), "=f"(r.thr), "=f"(r.count), "=f"(skipf)
        : "l"(nodes + k));
    r.skip = __float_as_int(skipf);
    return r;
}

// Batched embeddings: the sorted points of segment s occupy positions
// [off[s], off[s+1]) (sorting keeps segments in order), so its tree is the
// pre-order range [pre[off[s]], pre[off[s+1]]).  A lane is active only inside
// its own segment's range; lanes of a warp that straddles two segments walk
// their own trees under the same cursor.
struct SegView {
    const uint64_t *keys;   // sorted keys (segment id in the top bits)
    const int64_t *off;     // segment offsets
    const int *pre;         // pre-order start position per first point
};

__device__ __forceinline__ void segment_range(const SegView &sv, int p, int m, int &root, int &end)
{
    const int sg = (int)(sv.keys[p] >> kSegShift);
    root = sv.pre[sv.off[sg]];
    end = min(sv.pre[sv.off[sg + 1]], m);
}

// Launch order of the walk's blocks.  A walk's chunks differ in cost (dense
// regions have longer walks), and a grid of several waves whose costliest
// blocks start last ends with a tail of few busy SMs.  Every walk therefore
// records, per logical block, the cycles its warps took, and
// walk_order_kernel turns them into the launch order of the next walk:
// costliest first, the cheap blocks filling the end (longest-processing-time
// first).  The mapping of chunks to warps is unchanged, so results do not
// depend on the order.
struct BlockOrder {
    const int *order;  // [0]: grid size the order was made for; [1 + k]: logical block launched k-th
    unsigned *cost;    // per logical block: summed cycles / 64 of its warps (nullptr: not recorded)
};

__device__ __forceinline__ int logical_block(const BlockOrder &bo)
{
    int b = blockIdx.x;
    if (bo.order && bo.order[0] == (int)gridDim.x) {
        const int o = bo.order[1 + blockIdx.x];
        if (o >= 0 && o < (int)gridDim.x) b = o;
    }
    return b;
}

__device__ __forceinline__ void record_cost(const BlockOrder &bo, int b, long long t0)
{
    if (bo.cost && (threadIdx.x & 31) == 0)
        atomicAdd(&bo.cost[b], (unsigned)min((clock64() - t0) >> 6, 0xFFFFFll));
}

// Cuts of the tree (one embedding).  The root is never accepted (every point
// lies inside it, and r_cell / d >= 1 > theta), so a walk is the union of the
// walks of the subtrees below any cut of the tree.  A warp that takes one
// 32-point chunk and one subtree first evaluates the criterion at the
// subtree root's ancestors -- a lane that accepts one is done with this
// subtree, and the interaction with that ancestor is counted by the first
// subtree below it only -- then walks the subtree: every lane gets exactly
// the interactions of its full walk, in the same order.
//   Sums:  a cut at depth D (walk_split_depth); one running sum per point and
//          subtree, added in subtree order by walk_combine_kernel.
//   Units: a finer cut (subtrees of at most about n / units points) that only
//          divides the work of listing the interactions (list_f32_kernel).
constexpr int kMaxSplitDepth = 3;
constexpr int kMaxFrontier = 64;           // 4^3
constexpr int64_t kSplitMaxN = 1 << 19;    // above: chunks alone fill the GPU (a cut measured slower at 1M)
constexpr int64_t kSplitEntries = 1 << 22; // partial-sum buffer: entries x points
constexpr int kMaxUnits = 256;
constexpr int kMaxAnc = 8;                 // ancestors of a unit (deeper subtrees are not cut further)

struct Cut {
    int node, end;     // subtree root and the index after the subtree
    int nanc;          // ancestors below the root
    int own;           // bit k: an accepted anc[k] is counted here
    int anc[kMaxAnc];
};

struct CutTables {
    Cut sums[kMaxFrontier];
    Cut units[kMaxUnits];
    int first[kMaxFrontier + 1];  // units of sum s: first[s] .. first[s + 1] - 1
    int nsums, nunits;
};

struct SplitView {
    const CutTables *cut;             // nullptr: the whole tree is one subtree
    void *part;                       // [sum][n] partial sums (float4 / double4); nullptr: one sum
};

struct NodesF {  // float32 nodes: cell test, points and skip index
    const NodeF *nodes;
    __device__ bool cell(int k) const { return nodes[k].count >= 2.0f; }
    __device__ int points(int k) const { return (int)nodes[k].count; }
    __device__ int skip(int k) const { return nodes[k].skip; }
};
struct NodesD {  // float64 nodes
    const NodeD *nodes;
    __device__ bool cell(int k) const { return nodes[k].count >= 2; }
    __device__ int points(int k) const { return nodes[k].count; }
    __device__ int skip(int k) const { return nodes[k].skip; }
};

// Interaction lists between list_f32_kernel and sum_f32_kernel: pages of up
// to 32 interactions (the node and the lanes of the chunk that take it).  The
// first page of every (chunk, unit) has a fixed place; further ones come from
// pools (chunk mod kListPools, so that the atomic counters are spread).  A
// chunk whose pool runs out is flagged and walked directly by sum_f32_kernel.
constexpr int kPage = 32;
constexpr int kListPools = 256;

struct ListView {
    uint2 *entries;    // [page][kPage]: node, lane mask
    int2 *head;        // per page: interactions held, next page (-1: none)
    int *taken;        // per pool: pages taken
    int *direct;       // per chunk: its pool ran out
    int units;         // first pages per chunk
    int chunks;
    int per_pool;      // further pages per pool
};

// Per-lane state of the float32 walk: the query point (sorted position p),
// its running sums, and the pre-order index from which the lane is open
// again (a lane that accepts a cell skips the cell's subtree).
struct LaneF {
    float2 qh, ql;  // position as hi / lo float pairs
    float twoil;
    int p;
    int own;          // position of the point's own leaf (-1 in a bucket)
    float2 rxy, rsz;  // sums of k Delta and of (k s, mult w)
    int resume;
    unsigned long long c_acc, c_pair, c_crit;  // counting walk only
};

// Adds mult times the pair term of (Delta, s, delta) with conformal factor il
// of the other point: a cell's N_cell-weighted term (Eq. CellApproximation)
// or one exact pair (mult = 1).
// (The sums are paired: (rx, ry) += k Delta and (rs, z) += (k, mult) (s, w),
// one fused multiply-add per pair, rounded as the scalar ones.)
template <int GF, bool SMALL = false>
__device__ __forceinline__ void add_pair_f32(LaneF &L, float2 d, float s, float delta, float mult, float il)
{
    const PairF t = SMALL ? pair_terms_small_f32<GF>(delta) : pair_terms_f32<GF>(delta);
    const float k = mult * t.rep * il;
    L.rxy = __ffma2_rn(make_float2(k, k), d, L.rxy);
    L.rsz = __ffma2_rn(make_float2(k, mult), make_float2(s, t.w), L.rsz);
}

// The compensated difference y_i - y_j of two hi/lo float pairs and |y_i - y_j|^2.
__device__ __forceinline__ float2 delta_f32(const LaneF &L, float2 h, float2 l, float &s)
{
    const float2 d = delta2(L.qh, L.ql, h, l);
    s = fmaf(d.x, d.x, d.y * d.y);
    return d;
}

// Accepted interactions are collected first and evaluated later, a batch of
// up to 32 at a time: lane e holds interaction e (the node and the lanes that
// take it) until the batch is evaluated.  The cursor then never waits for a
// pair term, and the pair terms of a batch are independent of each other and
// of the walk.
struct BatchF {
    int node;       // interaction `lane`: its node
    unsigned mask;  // and the lanes that take it
    int count;      // interactions held (the same on every lane)
};
constexpr int kBatchFull = 28;  // evaluated above this (a trip of the walk adds up to four)

// Node data of a batch, one array per field, so that the data of consecutive
// interactions are register pairs of one (broadcast) shared-memory load.
struct __align__(16) TileF {
    float xh[32], yh[32], xl[32], yl[32], il[32], count[32];
};

// One visit of the warp's cursor at `node`: the lanes that accept the cell
// (or take the leaf) are noted in the batch.  A leaf or bucket has threshold
// -1, so every open lane takes it but the one whose own point it is (`own`:
// the position of the lane's own leaf).  Returns the next cursor: node + 1 if
// some open lane did not accept (the warp descends; past a leaf, node + 1 is
// the index after it), otherwise the index after the node's subtree.
// A lane is open from its `resume` to its own `end`.
__device__ __forceinline__ int visit_f32(int node, int end, int lane, LaneF &L, BatchF &B,
                                         const NodeF *__restrict__ nodes)
{
    const NodeF c = load_node(nodes, node);
    float s;
    delta_f32(L, make_float2(c.xh, c.yh), make_float2(c.xl, c.yl), s);
    const float delta = s * L.twoil * c.il;
    const bool open = node >= L.resume && node < end;
    const bool acc = open && node != L.own && delta > c.thr;  // r_cell / d < theta  <=>  delta > thr
    const unsigned m = __ballot_sync(0xffffffffu, acc);
    const bool down = __any_sync(0xffffffffu, open && !acc);
    if (acc) L.resume = c.skip;
    if (lane == B.count) {
        B.node = node;
        B.mask = m;
    }
    B.count += m != 0u ? 1 : 0;
    // next > node always: every node slot's skip exceeds its index
    return down ? node + 1 : c.skip;
}

// The 32 x 32 bit matrix whose row `lane` is v, transposed: bit e of lane i's
// result is bit i of lane e's v.
__device__ __forceinline__ unsigned transpose_bits(unsigned v, int lane)
{
    unsigned m = 0x0000FFFFu;
#pragma unroll
    for (int j = 16; j > 0; j >>= 1) {
        const unsigned o = __shfl_xor_sync(0xffffffffu, v, j);
        v = (lane & j) ? (v & ~m) | ((o >> j) & m) : (v & m) | ((o << j) & ~m);
        m ^= m << (j >> 1);
    }
    return v;
}

// Two consecutive interactions of a batch: k (the weight of Delta and s in the
// sums) and w of both in paired FP32 arithmetic, each component rounded as the
// scalar operations of add_pair_f32.
template <int GF>
__device__ __forceinline__ void two_terms_f32(const LaneF &L, float2 xh, float2 yh, float2 xl, float2 yl, float2 il,
                                              float2 mult, float2 &k, float2 &w)
{
    const float2 dx = delta2(make_float2(L.qh.x, L.qh.x), make_float2(L.ql.x, L.ql.x), xh, xl);
    const float2 dy = delta2(make_float2(L.qh.y, L.qh.y), make_float2(L.ql.y, L.ql.y), yh, yl);
    const float2 s = __ffma2_rn(dx, dx, __fmul2_rn(dy, dy));
    float2 rep;
    pair_terms2_f32<GF>(__fmul2_rn(__fmul2_rn(s, make_float2(L.twoil, L.twoil)), il), w, rep);
    k = __fmul2_rn(__fmul2_rn(mult, rep), il);
}

// A depth-29 bucket: each of its points exactly (not the lane's own).
template <int GF, bool COUNT>
__device__ __forceinline__ void add_bucket_f32(LaneF &L, const NodeF &c, const PointF *__restrict__ spts, int n)
{
    const int lo = __float_as_int(c.il), cnt = (int)(-c.count);
    if (lo < 0 || cnt <= 0 || lo + cnt > n) return;
    for (int k = 0; k < cnt; ++k) {
        if (lo + k == L.p) continue;
        const PointF o = spts[lo + k];
        float s;
        const float2 d = delta_f32(L, make_float2(o.xh, o.yh), make_float2(o.xl, o.yl), s);
        add_pair_f32<GF>(L, d, s, s * L.twoil * o.il, 1.0f, o.il);
        if (COUNT) ++L.c_pair;
    }
}

// A batch that holds a bucket: interaction by interaction.
template <int GF>
__device__ __forceinline__ void add_with_buckets_f32(LaneF &L, int bnode, unsigned bmask, int count, int lane,
                                                     const NodeF *__restrict__ nodes,
                                                     const PointF *__restrict__ spts, int n)
{
    for (int e = 0; e < count; ++e) {
        const NodeF c = load_node(nodes, __shfl_sync(0xffffffffu, bnode, e));
        const bool take = (__shfl_sync(0xffffffffu, bmask, e) >> lane) & 1u;
        if (!take) continue;
        if (c.count < 0.0f) {
            add_bucket_f32<GF, false>(L, c, spts, n);
            continue;
        }
        float s;
        const float2 d = delta_f32(L, make_float2(c.xh, c.yh), make_float2(c.xl, c.yl), s);
        add_pair_f32<GF>(L, d, s, s * L.twoil * c.il, c.count, c.il);
    }
}

// The point of lane `lane` of a chunk (the last point again past the end).
__device__ __forceinline__ void load_lane(LaneF &L, int chunk, int lane, int n, const PointF *__restrict__ spts,
                                          const int *__restrict__ leaf)
{
    L.p = chunk * 32 + lane;
    const int k = min(L.p, n - 1);
    const PointF q = spts[k];
    L.qh = make_float2(q.xh, q.yh);
    L.ql = make_float2(q.xl, q.yl);
    L.twoil = 2.0f * q.il;
    L.own = leaf[k];
    L.rxy = L.rsz = make_float2(0.f, 0.f);
    L.c_acc = L.c_pair = L.c_crit = 0;
}

// The ancestors of a cut's subtree: a lane that accepts one is done (returns
// false); the interaction goes to the batch if it is counted here.
__device__ __forceinline__ bool visit_ancestors_f32(const Cut &F, bool live, int lane, LaneF &L, BatchF &B,
                                                    const NodeF *__restrict__ nodes)
{
    const int na = F.nanc, owned = F.own;
    for (int k = 0; k < na; ++k) {
        const int at = F.anc[k];
        const NodeF a = load_node(nodes, at);
        const bool own = (owned >> k) & 1;
        float s;
        delta_f32(L, make_float2(a.xh, a.yh), make_float2(a.xl, a.yl), s);
        const bool acc = live && s * L.twoil * a.il > a.thr;
        const unsigned m = __ballot_sync(0xffffffffu, acc && own);
        if (lane == B.count) {
            B.node = at;
            B.mask = m;
        }
        B.count += m != 0u ? 1 : 0;
        live = live && !acc;
    }
    return live;
}

// A chunk's sums into its points' results (or, split, into the partial sums
// of subtree `sum`).
__device__ __forceinline__ void store_lane(const LaneF &L, int sum, int n, const uint32_t *__restrict__ idx,
                                           double2 *frep, double *zi, void *part)
{
    if (L.p >= n) return;
    if (part) {
        reinterpret_cast<float4 *>(part)[(size_t)sum * n + L.p] = make_float4(L.rxy.x, L.rxy.y, L.rsz.x, L.rsz.y);
        return;
    }
    const uint32_t i = idx[L.p];
    double x = (double)L.qh.x + (double)L.ql.x, y = (double)L.qh.y + (double)L.ql.y;
    double il = 0.5 * (double)L.twoil;
    double rsd = il * (double)L.rsz.x;
    frep[i] = make_double2(4.0 * il * ((double)L.rxy.x + rsd * x), 4.0 * il * ((double)L.rxy.y + rsd * y));
    zi[i] = (double)L.rsz.y;
}

// One visit of the direct walk's cursor at `node`, whose data `c` are loaded:
// as visit_f32, but the pair term is added at once.  The next node's load is
// issued before it, so that the load's latency and the pair term's overlap:
// a walk of one wave of blocks lasts as long as its longest chunk's chain of
// visits (load, criterion, vote, pair term, next load), and the overlap cut a
// visit from ~420 to ~290 cycles (walk at N = 70,000: 520 -> 367 us; N =
// 131,071, theta = 0.2: 6.2 -> 4.4 ms).  At N = 1M, several waves, issue slots
// bound the walk (88% of them taken, counting the second slot of a paired
// FP32 instruction) and the overlap changes nothing.  Leaves take the cells'
// path (threshold -1), so a visit tests the kind of node only for buckets.
// The term runs on every lane when one takes it (no divergent branch); a lane
// that does not adds it with weight 0, which leaves its sums unchanged (every
// term is finite: delta is clamped).
template <int GF, bool COUNT, bool BOUNDED, bool SMALL>
__device__ __forceinline__ void visit_direct_f32(int &node, NodeF &c, int end, LaneF &L,
                                                 const NodeF *__restrict__ nodes, const PointF *__restrict__ spts,
                                                 int n)
{
    float s;
    const float2 d = delta_f32(L, make_float2(c.xh, c.yh), make_float2(c.xl, c.yl), s);
    const float delta = s * L.twoil * c.il;
    const bool open = node >= L.resume && (!BOUNDED || node < end);
    const bool acc = open && node != L.own && delta > c.thr;
    const bool some = __any_sync(0xffffffffu, acc), down = __any_sync(0xffffffffu, open && !acc);
    node = down ? node + 1 : c.skip;
    const NodeF next = load_node(nodes, node);
    if (COUNT) {
        L.c_crit += open && c.count >= 2.0f ? 1 : 0;
        L.c_acc += acc && c.count >= 2.0f ? 1 : 0;
        L.c_pair += acc && c.count == 1.0f ? 1 : 0;
    }
    if (some) {
        L.resume = acc ? c.skip : L.resume;
        if (c.count >= 0.0f)
            add_pair_f32<GF, SMALL>(L, d, s, delta, acc ? c.count : 0.0f, c.il);
        else if (acc)
            add_bucket_f32<GF, COUNT>(L, c, spts, n);
    }
    c = next;
}

// Largest disk radius of each segment's points (the root annulus of its tree).
struct AnnulusView {
    const unsigned long long *bounds;  // [2s + 1]: largest split coordinate of segment s (float64 bits)
    const uint64_t *keys;              // sorted keys (segment id in the top bits); nullptr: one segment
    int rule, last;                    // split rule; last sorted position
};

// Whether every delta of the warp's points is below the series limit of
// pair_terms_f32, by the radii alone: |y_i - c| <= |y_i| + R and il_c <=
// 1 / (1 - R^2) for every point and midpoint c of a tree whose points lie
// within radius R (a midpoint lies in the hull of its points).  The same on
// every lane; a warp that straddles segments takes the larger R for all lanes,
// so that the terms of lanes that are not open stay finite too.
__device__ __forceinline__ bool all_small(const LaneF &L, int lane, const AnnulusView &an)
{
    const int p0 = __shfl_sync(0xffffffffu, L.p, 0);
    const int s = an.keys ? (int)(an.keys[p0 + min(lane, an.last - p0)] >> kSegShift) : 0;
    const float v = (float)__longlong_as_double((long long)an.bounds[2 * s + 1]);
    const float R2 = an.rule == HTS_EQUAL_AREA ? (v - 1.0f) / (v + 1.0f) : v * v;
    const float R = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(sqrtf(fmaxf(R2, 0.0f)))));
    const float r = sqrtf(L.qh.x * L.qh.x + L.qh.y * L.qh.y) + R;
    // (1% below the limit: far more than the roundings above)
    return __all_sync(0xffffffffu, R < 0.5f && r * r * L.twoil < 0.0198f * (1.0f - R * R));
}

// One warp walks for a chunk (sum `sum` of the cut when there are partial
// sums).  kWalkTrip visits per trip and one test of the cursor: the loop-back
// branch and the cursor tests cost (8 visits per trip against 4, walk at
// N = 131,071, theta = 0.2: 4.57 against 4.78 ms; at N = 1M, spread: 6.11
// against 6.32).  The cursor may run up to kWalkTrip - 1 nodes past `stop`
// (and the load one further): past the last node the tree build leaves empty
// slots (visited as no-ops), and below it every lane's own bound `end` closes
// it (BOUNDED).
// The first iterations, while the embedding is within a radius of ~0.05, take
// the loop without the logarithm (all_small; walk at N = 1M from Y0: 2.58 ->
// 2.30 ms, 64 embeddings: 0.74 -> 0.65 ms).
template <int GF, bool COUNT, bool SEG, bool SPLIT>
__device__ __forceinline__ void walk_f32_chunk(LaneF &L, int n, int lane, const NodeF *__restrict__ nodes,
                                                const int *__restrict__ n_nodes, const PointF *__restrict__ spts,
                                                unsigned long long *counters, const SegView sv, const CutTables *cut,
                                                int sum, const AnnulusView &an)
{
    const bool valid = L.p < n;
    unsigned long long c_visit = 0;
    const int m = min(*n_nodes, 2 * n);
    int root = 0, end = m;
    if (SEG) segment_range(sv, valid ? L.p : n - 1, m, root, end);
    bool live = valid;
    if (SPLIT) {  // ancestors first, then the subtree [node, end)
        const Cut &F = cut->sums[sum];
        const int na = F.nanc, owned = F.own;
        for (int k = 0; k < na; ++k) {
            const NodeF a = load_node(nodes, F.anc[k]);
            const bool own = (owned >> k) & 1;
            float s;
            const float2 d = delta_f32(L, make_float2(a.xh, a.yh), make_float2(a.xl, a.yl), s);
            const float delta = s * L.twoil * a.il;
            if (COUNT) L.c_crit += (live && own) ? 1 : 0;
            if (live && delta > a.thr) {
                if (own) {
                    add_pair_f32<GF>(L, d, s, delta, a.count, a.il);
                    if (COUNT) ++L.c_acc;
                }
                live = false;
            }
        }
        root = F.node;
        end = F.end;
    }
    L.resume = live ? root : INT_MAX;
    int node = SEG ? __shfl_sync(0xffffffffu, root, 0) : root;  // lane 0 holds the first segment
    const int stop = SEG ? __reduce_max_sync(0xffffffffu, valid ? end : 0) : end;
    NodeF c = load_node(nodes, node);
    if (!COUNT && all_small(L, lane, an)) {
        while (node < stop) {
#pragma unroll
            for (int k = 0; k < kWalkTrip; ++k)
                visit_direct_f32<GF, false, SEG || SPLIT, true>(node, c, end, L, nodes, spts, n);
        }
        return;
    }
    while (node < stop) {
#pragma unroll
        for (int k = 0; k < kWalkTrip; ++k) {
            if (COUNT && lane == 0 && node < stop) ++c_visit;  // (counted: visits below stop)
            visit_direct_f32<GF, COUNT, SEG || SPLIT, false>(node, c, end, L, nodes, spts, n);
        }
    }
    if (COUNT) {
        unsigned long long c_acc = L.c_acc, c_pair = L.c_pair, c_crit = L.c_crit;
        for (int o = 16; o > 0; o >>= 1) {
            c_acc += __shfl_xor_sync(0xffffffffu, c_acc, o);
            c_pair += __shfl_xor_sync(0xffffffffu, c_pair, o);
            c_crit += __shfl_xor_sync(0xffffffffu, c_crit, o);
        }
        if (lane == 0) {
            atomicAdd(&counters[0], c_acc);
            atomicAdd(&counters[1], c_pair);
            atomicAdd(&counters[2], c_visit);
            atomicAdd(&counters[3], (unsigned long long)min(32, n - L.p));
            atomicAdd(&counters[4], c_crit);
        }
    }
}

// Direct walk: one warp per chunk of 32 sorted points (and, split, per sum:
// grid.y); the warps of a block (blockDim.x / 32 <= kWalkBlock / 32, picked by
// the autotuner) take consecutive chunks, so their walks share node data in
// L1.  The block size does not change results.
template <int GF, bool COUNT, bool SEG, bool SPLIT>
__global__ void __launch_bounds__(kWalkBlock) walk_f32_kernel(int n, const NodeF *__restrict__ nodes,
                                                              const int *__restrict__ n_nodes,
                                                              const PointF *__restrict__ spts,
                                                              const int *__restrict__ leaf,
                                                              const uint32_t *__restrict__ idx, double2 *frep,
                                                              double *zi, unsigned long long *counters,
                                                              const SegView sv, const SplitView sp, const AnnulusView an,
                                                              const BlockOrder bo)
{
    const int b = logical_block(bo);
    const int chunk = (b * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (chunk * 32 >= n) return;
    if (SPLIT && (int)blockIdx.y >= sp.cut->nsums) return;
    const long long t0 = clock64();
    LaneF L;
    load_lane(L, chunk, lane, n, spts, leaf);
    walk_f32_chunk<GF, COUNT, SEG, SPLIT>(L, n, lane, nodes, n_nodes, spts, counters, sv, sp.cut, blockIdx.y, an);
    store_lane(L, blockIdx.y, n, idx, frep, zi, SPLIT ? sp.part : nullptr);
    record_cost(bo, b, t0);
}

// Lists the interactions of a chunk (grid.x: chunks, a warp each; the warps of
// a block take consecutive chunks, so their walks share node data in L1) with
// one unit of the tree (grid.y).
__global__ void __launch_bounds__(kListBlock, 6) list_f32_kernel(int n, const NodeF *__restrict__ nodes,
                                                                 const PointF *__restrict__ spts,
                                                                 const int *__restrict__ leaf,
                                                                 const CutTables *__restrict__ cut, const ListView lv)
{
    const int chunk = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (chunk >= lv.chunks || (int)blockIdx.y >= cut->nunits) return;
    LaneF L;
    load_lane(L, chunk, lane, n, spts, leaf);
    BatchF B;
    B.node = 0;
    B.mask = 0u;
    B.count = 0;
    const Cut &F = cut->units[blockIdx.y];
    const bool live = visit_ancestors_f32(F, L.p < n, lane, L, B, nodes);
    int node = F.node;
    const int end = F.end;
    L.resume = live ? node : INT_MAX;
    if (!__any_sync(0xffffffffu, live)) node = end;
    int page = chunk * lv.units + (int)blockIdx.y;
    const int pool = chunk & (kListPools - 1);
    while (node < end) {  // (a page holds what a trip can add to kBatchFull)
#pragma unroll
        for (int k = 0; k < kPage - kBatchFull; ++k) node = visit_f32(node, end, lane, L, B, nodes);
        if (B.count > kBatchFull) {  // the page is full: write it, take another
            if (lane < B.count) lv.entries[(size_t)page * kPage + lane] = make_uint2((unsigned)B.node, B.mask);
            int next = 0;
            if (lane == 0) {
                next = atomicAdd(&lv.taken[pool], 1);
                next = next < lv.per_pool ? lv.chunks * lv.units + pool * lv.per_pool + next : -1;
                lv.head[page] = make_int2(B.count, next);
                if (next < 0) lv.direct[chunk] = 1;
            }
            next = __shfl_sync(0xffffffffu, next, 0);
            if (next < 0) return;
            page = next;
            B.count = 0;
        }
    }
    if (lane < B.count) lv.entries[(size_t)page * kPage + lane] = make_uint2((unsigned)B.node, B.mask);
    if (lane == 0) lv.head[page] = make_int2(B.count, -1);
}

// A block evaluates the listed interactions of a chunk (grid.x; grid.y: the
// sum).  The interactions of consecutive pages make batches of up to 32, dealt
// to the block's kSumWarps warps in turn: the pair terms of different batches
// run beside each other, and only the running sums go from warp to warp in
// batch order, so every sum is taken in the order of the walk.  With one warp
// per chunk the longest chunk takes most of the kernel (N = 20,011, 2,500
// (chunk, sum) pairs: 180 us with one warp each, 133 us with four).
constexpr int kSumWarps = 4;

struct SumShared {
    TileF tile[kSumWarps];
    float2 term[kSumWarps][32][32];  // [warp][interaction][lane]: k, w (0 where the lane does not take it)
    float4 sums[32];                 // running sums of the lanes' points after the last finished batch
};

// Waits for / passes on the running sums: barrier 1 + w pairs the warp w that
// waits with the warp before it.
__device__ __forceinline__ void sums_wait(int w)
{
    asm volatile("bar.sync %0, 64;" ::"r"(1 + w) : "memory");
}
__device__ __forceinline__ void sums_pass(int w)
{
    __threadfence_block();
    asm volatile("bar.arrive %0, 64;" ::"r"(1 + (w + 1 == kSumWarps ? 0 : w + 1)) : "memory");
}

// One batch of a warp (its `batch`-th in the block's order): terms, then, in
// turn, the sums.
template <int GF>
__device__ __forceinline__ void sum_batch_f32(LaneF &L, const BatchF &B, int batch, int w, int lane, SumShared &S,
                                              const NodeF *__restrict__ nodes, const PointF *__restrict__ spts, int n)
{
    TileF &T = S.tile[w];
    const bool have = lane < B.count;
    const unsigned mask = have ? B.mask : 0u;
    const NodeF c = load_node(nodes, have ? B.node : 0);
    const bool bucket = __any_sync(0xffffffffu, have && c.count < 0.0f);
    if (!bucket) {
        __syncwarp();  // the warp's previous batch has been read
        T.xh[lane] = c.xh;
        T.yh[lane] = c.yh;
        T.xl[lane] = c.xl;
        T.yl[lane] = c.yl;
        T.il[lane] = c.il;
        T.count[lane] = c.count;
        unsigned bits = transpose_bits(mask, lane);
        __syncwarp();
        for (int e = 0; e < B.count; e += 4) {  // (slots past the count: no lane takes them)
            const float4 xh = *reinterpret_cast<const float4 *>(&T.xh[e]), yh = *reinterpret_cast<const float4 *>(&T.yh[e]);
            const float4 xl = *reinterpret_cast<const float4 *>(&T.xl[e]), yl = *reinterpret_cast<const float4 *>(&T.yl[e]);
            const float4 il = *reinterpret_cast<const float4 *>(&T.il[e]);
            const float4 ct = *reinterpret_cast<const float4 *>(&T.count[e]);
            const bool t0 = bits & 1u, t1 = bits & 2u, t2 = bits & 4u, t3 = bits & 8u;
            float2 k, v;
            two_terms_f32<GF>(L, make_float2(xh.x, xh.y), make_float2(yh.x, yh.y), make_float2(xl.x, xl.y),
                              make_float2(yl.x, yl.y), make_float2(il.x, il.y),
                              make_float2(t0 ? ct.x : 0.0f, t1 ? ct.y : 0.0f), k, v);
            S.term[w][e][lane] = make_float2(k.x, t0 ? v.x : 0.0f);
            S.term[w][e + 1][lane] = make_float2(k.y, t1 ? v.y : 0.0f);
            two_terms_f32<GF>(L, make_float2(xh.z, xh.w), make_float2(yh.z, yh.w), make_float2(xl.z, xl.w),
                              make_float2(yl.z, yl.w), make_float2(il.z, il.w),
                              make_float2(t2 ? ct.z : 0.0f, t3 ? ct.w : 0.0f), k, v);
            S.term[w][e + 2][lane] = make_float2(k.x, t2 ? v.x : 0.0f);
            S.term[w][e + 3][lane] = make_float2(k.y, t3 ? v.y : 0.0f);
            bits >>= 4;
        }
    }
    if (batch > 0) {
        sums_wait(w);
        const float4 r = S.sums[lane];
        L.rxy = make_float2(r.x, r.y);
        L.rsz = make_float2(r.z, r.w);
    }
    if (!bucket) {
        for (int e = 0; e < B.count; e += 4) {
            const float4 xh = *reinterpret_cast<const float4 *>(&T.xh[e]), yh = *reinterpret_cast<const float4 *>(&T.yh[e]);
            const float4 xl = *reinterpret_cast<const float4 *>(&T.xl[e]), yl = *reinterpret_cast<const float4 *>(&T.yl[e]);
            const float4 ct = *reinterpret_cast<const float4 *>(&T.count[e]);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float2 t = S.term[w][e + q][lane];
                float s;
                const float2 d = delta_f32(L, make_float2((&xh.x)[q], (&yh.x)[q]), make_float2((&xl.x)[q], (&yl.x)[q]), s);
                L.rxy = __ffma2_rn(make_float2(t.x, t.x), d, L.rxy);
                L.rsz = __ffma2_rn(make_float2(t.x, (&ct.x)[q]), make_float2(s, t.y), L.rsz);
            }
        }
    } else {
        add_with_buckets_f32<GF>(L, B.node, mask, B.count, lane, nodes, spts, n);
        __syncwarp();
    }
    S.sums[lane] = make_float4(L.rxy.x, L.rxy.y, L.rsz.x, L.rsz.y);
    sums_pass(w);
}

template <int GF, bool SPLIT>
__global__ void __launch_bounds__(32 * kSumWarps, 6) sum_f32_kernel(int n, const NodeF *__restrict__ nodes,
                                                                    const int *__restrict__ n_nodes,
                                                                    const PointF *__restrict__ spts,
                                                                    const int *__restrict__ leaf,
                                                                    const uint32_t *__restrict__ idx, double2 *frep,
                                                                    double *zi, const SplitView sp, const ListView lv,
                                                                    const AnnulusView an)
{
    __shared__ SumShared S;
    const int chunk = blockIdx.x, w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int sum = SPLIT ? (int)blockIdx.y : 0;
    if (sum >= sp.cut->nsums) return;
    LaneF L;
    load_lane(L, chunk, lane, n, spts, leaf);
    if (lv.direct[chunk]) {
        if (w > 0) return;
        walk_f32_chunk<GF, false, false, SPLIT>(L, n, lane, nodes, n_nodes, spts, nullptr, SegView{}, sp.cut, sum, an);
        store_lane(L, sum, n, idx, frep, zi, SPLIT ? sp.part : nullptr);
        return;
    }
    BatchF B;
    B.node = 0;
    B.mask = 0u;
    B.count = 0;
    int batch = 0, turn = 0;  // the batch being gathered, and its warp: batch mod kSumWarps
    const int u0 = sp.cut->first[sum], u1 = sp.cut->first[sum + 1];
    for (int ub = u0; ub < u1; ub += 32) {
        const int2 h = ub + lane < u1 ? lv.head[chunk * lv.units + ub + lane] : make_int2(0, -1);
        unsigned todo = __ballot_sync(0xffffffffu, h.x > 0);
        while (todo) {
            const int j = __ffs((int)todo) - 1;
            todo &= todo - 1;
            int page = chunk * lv.units + ub + j;
            int count = __shfl_sync(0xffffffffu, h.x, j), next = __shfl_sync(0xffffffffu, h.y, j);
            while (true) {
                if (B.count + count > 32) {
                    if (turn == w) sum_batch_f32<GF>(L, B, batch, w, lane, S, nodes, spts, n);
                    ++batch;
                    turn = turn + 1 == kSumWarps ? 0 : turn + 1;
                    B.count = 0;
                }
                if (turn == w && lane >= B.count && lane < B.count + count) {
                    const uint2 e = lv.entries[(size_t)page * kPage + lane - B.count];
                    B.node = (int)e.x;
                    B.mask = e.y;
                }
                B.count += count;
                if (next < 0) break;
                page = next;
                const int2 g = lv.head[page];
                count = g.x;
                next = g.y;
            }
        }
    }
    if (B.count > 0) {
        if (turn == w) sum_batch_f32<GF>(L, B, batch, w, lane, S, nodes, spts, n);
        ++batch;
        turn = turn + 1 == kSumWarps ? 0 : turn + 1;
    }
    if (turn != w) return;
    if (batch > 0) {  // the warp after the last batch's takes the sums
        sums_wait(w);
        const float4 r = S.sums[lane];
        L.rxy = make_float2(r.x, r.y);
        L.rsz = make_float2(r.z, r.w);
    }
    store_lane(L, sum, n, idx, frep, zi, SPLIT ? sp.part : nullptr);
}

template <int GF, bool COUNT, bool SEG, bool SPLIT>
__device__ __forceinline__ void walk_f64_chunk(int warp, int n, const NodeD *__restrict__ nodes,
                                                const int *__restrict__ n_nodes,
                                                const PointD *__restrict__ spts,
                                                const uint32_t *__restrict__ idx, double2 *frep, double *zi,
                                                unsigned long long *counters, const SegView sv,
                                                const SplitView sp, int fi)
{
    const int lane = threadIdx.x & 31;
    const int p = warp * 32 + lane;
    const bool valid = p < n;
    const PointD q = spts[valid ? p : n - 1];
    const double twoil = 2.0 * q.il;
    double rx = 0, ry = 0, rs = 0, z = 0;
    const int m = min(*n_nodes, 2 * n);
    int root = 0, end = m;
    if (SEG) segment_range(sv, valid ? p : n - 1, m, root, end);
    unsigned long long c_acc = 0, c_pair = 0, c_visit = 0;
    bool live = valid;
    if (SPLIT) {  // as in the float32 walk
        const Cut &F = sp.cut->sums[fi];
        for (int k = 0; k < F.nanc; ++k) {
            const NodeD a = nodes[F.anc[k]];
            double dx = q.x - a.x, dy = q.y - a.y;
            double s = fma(dx, dx, dy * dy);
            double delta = s * twoil * a.il;
            if (live && delta > a.thr) {
                if ((F.own >> k) & 1) {
                    PairD t = pair_terms_f64<GF>(delta);
                    double mult = (double)a.count;
                    double kk = mult * t.rep * a.il;
                    rx = fma(kk, dx, rx);
                    ry = fma(kk, dy, ry);
                    rs = fma(kk, s, rs);
                    z = fma(mult, t.w, z);
                    if (COUNT) ++c_acc;
                }
                live = false;
            }
        }
        root = F.node;
        end = F.end;
    }
    int resume = live ? root : INT_MAX;
    int node = SEG ? __shfl_sync(0xffffffffu, root, 0) : root;
    const int stop = SEG ? __reduce_max_sync(0xffffffffu, valid ? end : 0) : end;
    while (node < stop) {
        const NodeD c = nodes[node];
        const bool active = node >= resume && (!SEG || node < end);
        int next = node + 1;
        if (c.count >= 2) {
            double dx = q.x - c.x, dy = q.y - c.y;
            double s = fma(dx, dx, dy * dy);
            double delta = s * twoil * c.il;
            bool acc = active && delta > c.thr;
            if (acc) {
                PairD t = pair_terms_f64<GF>(delta);
                double mult = (double)c.count;
                double k = mult * t.rep * c.il;
                rx = fma(k, dx, rx);
                ry = fma(k, dy, ry);
                rs = fma(k, s, rs);
                z = fma(mult, t.w, z);
                resume = c.skip;
                if (COUNT) ++c_acc;
            }
            if (!__any_sync(0xffffffffu, active && !acc)) next = c.skip;
        } else if (c.count == 1) {
            if (active && c.pos != p) {
                double dx = q.x - c.x, dy = q.y - c.y;
                double s = fma(dx, dx, dy * dy);
                PairD t = pair_terms_f64<GF>(s * twoil * c.il);
                double k = t.rep * c.il;
                rx = fma(k, dx, rx);
                ry = fma(k, dy, ry);
                rs = fma(k, s, rs);
                z += t.w;
                if (COUNT) ++c_pair;
            }
        } else {
            const int lo = c.pos, cnt = -c.count;
            if (active && lo >= 0 && cnt > 0 && lo + cnt <= n) {
                for (int k2 = 0; k2 < cnt; ++k2) {
                    if (lo + k2 == p) continue;
                    PointD o = spts[lo + k2];
                    double dx = q.x - o.x, dy = q.y - o.y;
                    double s = fma(dx, dx, dy * dy);
                    PairD t = pair_terms_f64<GF>(s * twoil * o.il);
                    double k = t.rep * o.il;
                    rx = fma(k, dx, rx);
                    ry = fma(k, dy, ry);
                    rs = fma(k, s, rs);
                    z += t.w;
                    if (COUNT) ++c_pair;
                }
            }
        }
        if (COUNT && lane == 0) ++c_visit;
        node = next;  // as in the float32 walk
    }
    if (SPLIT && valid) {
        reinterpret_cast<double4_32a *>(sp.part)[(size_t)fi * n + p] = make_double4_32a(rx, ry, rs, z);
    } else if (valid) {
        const uint32_t i = idx[p];
        double rsd = q.il * rs;
        frep[i] = make_double2(4.0 * q.il * (rx + rsd * q.x), 4.0 * q.il * (ry + rsd * q.y));
        zi[i] = z;
    }
    if (COUNT) {
        for (int o = 16; o > 0; o >>= 1) {
            c_acc += __shfl_xor_sync(0xffffffffu, c_acc, o);
            c_pair += __shfl_xor_sync(0xffffffffu, c_pair, o);
        }
        if (lane == 0) {
            atomicAdd(&counters[0], c_acc);
            atomicAdd(&counters[1], c_pair);
            atomicAdd(&counters[2], c_visit);
            atomicAdd(&counters[3], (unsigned long long)min(32, n - warp * 32));
        }
    }
}

// As walk_f32_kernel, in float64.
template <int GF, bool COUNT, bool SEG, bool SPLIT>
__global__ void __launch_bounds__(kWalkBlock) walk_f64_kernel(int n, const NodeD *__restrict__ nodes,
                                                              const int *__restrict__ n_nodes,
                                                              const PointD *__restrict__ spts,
                                                              const int *__restrict__ leaf,
                                                              const uint32_t *__restrict__ idx, double2 *frep,
                                                              double *zi, unsigned long long *counters,
                                                              const SegView sv, const SplitView sp,
                                                              const BlockOrder bo)
{
    const int b = logical_block(bo);
    const int warp = (b * blockDim.x + threadIdx.x) >> 5;
    if (warp * 32 >= n) return;
    if (SPLIT && (int)blockIdx.y >= sp.cut->nsums) return;
    const long long t0 = clock64();
    walk_f64_chunk<GF, COUNT, SEG, SPLIT>(warp, n, nodes, n_nodes, spts, idx, frep, zi, counters, sv, sp, blockIdx.y);
    record_cost(bo, b, t0);
}

// The next launch order from the recorded costs: a counting sort on 256
// levels of cost / (max + 1), costliest first (the order inside a level is
// arbitrary); then the costs are cleared for the next walk.  One block.
__global__ void __launch_bounds__(1024) walk_order_kernel(unsigned *cost, int nb, int *order)
{
    __shared__ unsigned hist[256];
    __shared__ unsigned smax;
    if (threadIdx.x < 256) hist[threadIdx.x] = 0;
    if (threadIdx.x == 0) smax = 0;
    __syncthreads();
    unsigned m = 0;
    for (int b = threadIdx.x; b < nb; b += blockDim.x) m = max(m, cost[b]);
    for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) atomicMax(&smax, m);
    __syncthreads();
    const unsigned long long top = (unsigned long long)smax + 1ull;
    for (int b = threadIdx.x; b < nb; b += blockDim.x)
        atomicAdd(&hist[255 - (int)((unsigned long long)cost[b] * 256ull / top)], 1u);
    __syncthreads();
    if (threadIdx.x == 0) {  // exclusive scan over the 256 levels
        unsigned run = 0;
        for (int k = 0; k < 256; ++k) {
            const unsigned h = hist[k];
            hist[k] = run;
            run += h;
        }
    }
    __syncthreads();
    for (int b = threadIdx.x; b < nb; b += blockDim.x) {
        const unsigned pos = atomicAdd(&hist[255 - (int)((unsigned long long)cost[b] * 256ull / top)], 1u);
        order[1 + pos] = b;
        cost[b] = 0;
    }
    __syncthreads();
    if (threadIdx.x == 0) order[0] = nb;
}

// Both cuts (one block): level by level from the root, one thread per subtree,
// every cell above `depth` into its children, then every cell of more than
// `grain` points, while the subtrees fit `cap`; in pre-order throughout.  A
// cell with more than 4 children or a skip that does not advance is a broken
// tree: status bit 2, no subtrees (the walk then does no work and the error is
// reported).
template <typename NV>
__global__ void __launch_bounds__(kMaxUnits) cut_kernel(const NV nodes, const int *__restrict__ n_nodes, int n,
                                                        int depth, int grain, int cap, CutTables *ct, int *status)
{
    __shared__ Cut sub[2][kMaxUnits];
    __shared__ int sum_of[2][kMaxUnits];
    __shared__ int wtot[kMaxUnits / 32];
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    const int m = min(*n_nodes, 2 * n);
    int cur = 0, count = 1, nsums = 1;
    if (t == 0) {
        sub[0][0] = Cut{0, m, 0, 0, {0, 0, 0, 0, 0, 0, 0, 0}};
        sum_of[0][0] = 0;
    }
    __syncthreads();
    int bad = m <= 0 ? 1 : 0;
    for (int lev = 0; lev < depth + kMaxAnc && !bad; ++lev) {
        Cut U;
        int kids = 0, ch[4] = {0, 0, 0, 0};
        bool expand = false;
        if (t < count) {
            U = sub[cur][t];
            expand = nodes.cell(U.node) && (lev < depth || (nodes.points(U.node) > grain && U.nanc < kMaxAnc));
            kids = expand ? 0 : 1;
            if (expand) {
                for (int c = U.node + 1; c < U.end && !bad;) {
                    const int nx = nodes.skip(c);
                    if (kids == 4 || nx <= c) {
                        bad = 1;
                        break;
                    }
                    ch[kids++] = c;
                    c = nx;
                }
            }
        }
        int incl = kids;
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
        }
        if (lane == 31) wtot[w] = incl;
        bad = __syncthreads_or(bad);
        const int grown = __syncthreads_or(expand ? 1 : 0);
        int at = incl - kids, total = 0;
        for (int k = 0; k < kMaxUnits / 32; ++k) {
            if (k < w) at += wtot[k];
            total += wtot[k];
        }
        if (bad || (lev >= depth && !grown) || total > cap) {
            bad |= lev < depth && total > cap ? 1 : 0;
            break;
        }
        if (t < count) {
            const int s = sum_of[cur][t];
            if (!expand) {
                sub[cur ^ 1][at] = U;
                sum_of[cur ^ 1][at] = s;
            } else {
                const int na = U.nanc;
                const bool below = U.node != 0;  // an ancestor of its children, unless it is the root
                for (int k = 0; k < kids; ++k) {
                    Cut F = U;
                    F.node = ch[k];
                    F.end = k + 1 < kids ? ch[k + 1] : U.end;
                    F.own = k == 0 ? U.own | (below ? 1 << na : 0) : 0;
                    if (below) {
                        for (int q = 0; q < kMaxAnc; ++q)
                            if (q == na) F.anc[q] = U.node;
                        F.nanc = na + 1;
                    }
                    sub[cur ^ 1][at + k] = F;
                    sum_of[cur ^ 1][at + k] = s;
                }
            }
        }
        __syncthreads();
        cur ^= 1;
        count = total;
        if (lev + 1 == depth) {
            if (t < count) {
                ct->sums[t] = sub[cur][t];
                sum_of[cur][t] = t;
            }
            nsums = count;
            __syncthreads();
        }
    }
    if (bad) {
        if (t == 0) atomicOr(status, 2);
        count = nsums = 0;
    }
    if (t < count) {
        ct->units[t] = sub[cur][t];
        const int s = sum_of[cur][t];
        if (t == 0 || sum_of[cur][t - 1] != s) ct->first[s] = t;
    }
    if (t == 0) {
        ct->first[nsums] = count;
        if (bad) ct->first[0] = ct->first[1] = 0;
        ct->nsums = nsums;
        ct->nunits = count;
    }
}

// Sorted point p: the partial sums of the cut's subtrees in subtree order,
// then the per-point factors.  Four lanes per point, one per quantity, in
// blocks of one warp: the float64 adds and conversions (4 x 64 of each at the
// deepest cut) go to a pipe of two lanes a cycle per SM, so a small problem
// wants them on as many SMs as possible (N = 2000: 38 us with 8 blocks of 256
// points' threads, 6 us with 250 warps).
constexpr int kCombineBlock = 32;

template <typename PT, typename T>
__global__ void __launch_bounds__(kCombineBlock) walk_combine_kernel(int n, const PT *__restrict__ spts,
                                                                     const uint32_t *__restrict__ idx,
                                                                     const T *__restrict__ part,
                                                                     const int *__restrict__ count, double2 *frep,
                                                                     double *zi)
{
    const int p = (blockIdx.x * kCombineBlock + threadIdx.x) >> 2, q = threadIdx.x & 3;
    const int k = min(p, n - 1), nf = *count;
    const T *__restrict__ v = part + 4 * (size_t)k + q;
    double a = 0;
#pragma unroll 8
    for (int e = 0; e < nf; ++e) a += (double)v[4 * (size_t)e * n];
    const double rx = __shfl_sync(0xffffffffu, a, 0, 4), ry = __shfl_sync(0xffffffffu, a, 1, 4);
    const double rs = __shfl_sync(0xffffffffu, a, 2, 4), z = __shfl_sync(0xffffffffu, a, 3, 4);
    if (p >= n || q > 0) return;
    double x, y, il;
    point_xy_il(spts[p], x, y, il);
    const double rsd = il * rs;
    const uint32_t i = idx[p];
    frep[i] = make_double2(4.0 * il * (rx + rsd * x), 4.0 * il * (ry + rsd * y));
    zi[i] = z;
}

// Exact repulsion: one thread per point i, tiles of kExactBlock points j
// staged in shared memory, every pair j != i of the same segment.  A small
// problem has too few i-blocks to fill the GPU, so the j range of each
// i-block is cut into `split` chunks (grid.y): with split == 1 the block
// writes the finished force and Z_i, otherwise raw sums per chunk go to
// `part` and exact_combine_kernel adds them in chunk order (deterministic).
struct ExactArgs {
    int n, split;
    double2 *frep;
    double *zi;
    double4_32a *part;  // [split][n]: sums of k Delta_x, k Delta_y, k s, w
    const unsigned char *seg_of;
    const int64_t *seg_off;
};

__device__ __forceinline__ void exact_ranges(const ExactArgs &A, int i, int &jlo, int &jhi, int &cbeg, int &cend)
{
    // own segment [jlo, jhi); the union over the block's threads, cut into chunks
    int blo = 0, bhi = A.n;
    jlo = 0;
    jhi = A.n;
    if (A.seg_of) {
        const int first = blockIdx.x * kExactBlock, last = min(first + kExactBlock, A.n) - 1;
        const int si = A.seg_of[i < A.n ? i : A.n - 1];
        jlo = (int)A.seg_off[si];
        jhi = (int)A.seg_off[si + 1];
        blo = (int)A.seg_off[A.seg_of[first]];
        bhi = (int)A.seg_off[A.seg_of[last] + 1];
    }
    const int tiles = (bhi - blo + kExactBlock - 1) / kExactBlock;
    const int per = (tiles + A.split - 1) / A.split;
    cbeg = min(bhi, blo + (int)blockIdx.y * per * kExactBlock);
    cend = min(bhi, cbeg + per * kExactBlock);
}

template <int GF>
__global__ void __launch_bounds__(kExactBlock) exact_f32_kernel(const PointF *__restrict__ pts, ExactArgs A)
{
    __shared__ PointF tile[kExactBlock];
    const int n = A.n;
    const int i = blockIdx.x * kExactBlock + threadIdx.x;
    int jlo, jhi, cbeg, cend;
    exact_ranges(A, i, jlo, jhi, cbeg, cend);
    const PointF q = pts[i < n ? i : n - 1];
    const float2 qh = make_float2(q.xh, q.yh), ql = make_float2(q.xl, q.yl);
    const float twoil = 2.0f * q.il;
    float2 rxy = make_float2(0.f, 0.f), rsz = make_float2(0.f, 0.f);  // paired sums, as in the walk
    for (int base = cbeg; base < cend; base += kExactBlock) {
        int j = base + threadIdx.x;
        if (j < cend) tile[threadIdx.x] = pts[j];
        __syncthreads();
        const int cnt = min(kExactBlock, cend - base);
        for (int k = 0; k < cnt; ++k) {
            const int jj = base + k;
            if (jj == i || jj < jlo || jj >= jhi) continue;
            const PointF o = tile[k];
            const float2 d = delta2(qh, ql, make_float2(o.xh, o.yh), make_float2(o.xl, o.yl));
            const float s = fmaf(d.x, d.x, d.y * d.y);
            const PairF t = pair_terms_f32<GF>(s * twoil * o.il);
            const float kk = t.rep * o.il;
            rxy = __ffma2_rn(make_float2(kk, kk), d, rxy);
            rsz = __ffma2_rn(make_float2(kk, 1.0f), make_float2(s, t.w), rsz);
        }
        __syncthreads();
    }
    if (i >= n) return;
    if (A.split > 1) {
        A.part[(size_t)blockIdx.y * n + i] = make_double4_32a(rxy.x, rxy.y, rsz.x, rsz.y);
        return;
    }
    double x = (double)q.xh + (double)q.xl, y = (double)q.yh + (double)q.yl;
    double il = (double)q.il;
    double rsd = il * (double)rsz.x;
    A.frep[i] = make_double2(4.0 * il * ((double)rxy.x + rsd * x), 4.0 * il * ((double)rxy.y + rsd * y));
    A.zi[i] = (double)rsz.y;
}

template <int GF>
__global__ void __launch_bounds__(kExactBlock) exact_f64_kernel(const PointD *__restrict__ pts, ExactArgs A)
{
    __shared__ PointD tile[kExactBlock];
    const int n = A.n;
    const int i = blockIdx.x * kExactBlock + threadIdx.x;
    int jlo, jhi, cbeg, cend;
    exact_ranges(A, i, jlo, jhi, cbeg, cend);
    const PointD q = pts[i < n ? i : n - 1];
    const double twoil = 2.0 * q.il;
    double rx = 0, ry = 0, rs = 0, z = 0;
    for (int base = cbeg; base < cend; base += kExactBlock) {
        int j = base + threadIdx.x;
        if (j < cend) tile[threadIdx.x] = pts[j];
        __syncthreads();
        const int cnt = min(kExactBlock, cend - base);
        for (int k = 0; k < cnt; ++k) {
            const int jj = base + k;
            if (jj == i || jj < jlo || jj >= jhi) continue;
            const PointD o = tile[k];
            double dx = q.x - o.x, dy = q.y - o.y;
            double s = fma(dx, dx, dy * dy);
            PairD t = pair_terms_f64<GF>(s * twoil * o.il);
            double kk = t.rep * o.il;
            rx = fma(kk, dx, rx);
            ry = fma(kk, dy, ry);
            rs = fma(kk, s, rs);
            z += t.w;
        }
        __syncthreads();
    }
    if (i >= n) return;
    if (A.split > 1) {
        A.part[(size_t)blockIdx.y * n + i] = make_double4_32a(rx, ry, rs, z);
        return;
    }
    double rsd = q.il * rs;
    A.frep[i] = make_double2(4.0 * q.il * (rx + rsd * q.x), 4.0 * q.il * (ry + rsd * q.y));
    A.zi[i] = z;
}

// Sums of the chunks of each point in chunk order, then the per-point factors.
template <typename PT>
__global__ void exact_combine_kernel(const PT *__restrict__ pts, ExactArgs A)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= A.n) return;
    double rx = 0, ry = 0, rs = 0, z = 0;
    for (int c = 0; c < A.split; ++c) {
        const double4_32a v = A.part[(size_t)c * A.n + i];
        rx += v.x;
        ry += v.y;
        rs += v.z;
        z += v.w;
    }
    const PT q = pts[i];
    double x, y, il;
    point_xy_il(q, x, y, il);
    const double rsd = il * rs;
    A.frep[i] = make_double2(4.0 * il * (rx + rsd * x), 4.0 * il * (ry + rsd * y));
    A.zi[i] = z;
}

}  // namespace

int walk_split_capacity(int64_t n)
{
    // subtrees x points of the partial-sum buffer (0: no split)
    if (n <= 0 || n > kSplitMaxN) return 0;
    return (int)std::min<int64_t>(kMaxFrontier, kSplitEntries / n);
}

// Listed or direct: up to kListMaxN points (1,024 chunks) the direct walk's
// few chains of visits leave the GPU idle (N = 20,011: 412 us direct against
// 142 us to list and 133 us to sum); above, its chunks are enough and listing
// costs more instructions than it saves time (N = 70,000: 363 us direct,
// 173 + 172 us listed; list_units 0).  The tree is divided into enough units
// for about kListWarps (chunk, unit) warps (N = 20,011, list kernel: 20,000 /
// 40,000 / 100,000 warps 183 / 142 / 205 us).
#ifndef LW
#define LW 40000
#endif
#ifndef LMAX
#define LMAX 128
#endif
constexpr int64_t kListWarps = LW;
constexpr int64_t kListMaxN = 1 << 15;

static int list_target(int64_t n)
{
    const int64_t chunks = std::max<int64_t>((n + 31) / 32, 1);
    return (int)std::max<int64_t>(2, std::min<int64_t>(kListWarps / chunks, LMAX));
}

// First pages per chunk: the cap of the cut into units (a cut by point counts
// overshoots its target; a cut at depth D has up to 4^D subtrees).
int list_units(int64_t n)
{
    if (n > kListMaxN) return 0;
    return std::min(kMaxUnits, std::max(4 * list_target(n), walk_split_capacity(n)));
}

// Further pages per pool: 512 pages a chunk (16,384 interactions; theta = 0.5
// lists about 1,000 to 4,000 a chunk), 134 MB at kListMaxN points.
static int list_per_pool(int64_t n) { return (int)((n + 31) / 32 * 512 / kListPools + 1); }

int64_t list_pages(int64_t n)
{
    return n > kListMaxN ? 0 : (n + 31) / 32 * list_units(n) + (int64_t)list_per_pool(n) * kListPools;
}
size_t list_page_bytes() { return sizeof(uint2) * kPage; }
int64_t list_flags(int64_t n) { return kListPools + (n + 31) / 32; }

// Cut depth for n points: the shallowest that gives about 2048 warps, within
// the buffer; `want` >= 0 overrides (clamped), -1 chooses.  (A deeper cut for
// the float64 walk measured slower at N = 20,000: there the float64 pipe, not
// the warp count, is the limit.)
int walk_split_depth(int64_t n, int want, bool fp64)
{
    (void)fp64;
    const int cap = walk_split_capacity(n);
    int dmax = 0;
    while (dmax < kMaxSplitDepth && (1 << (2 * (dmax + 1))) <= cap) ++dmax;
    if (want >= 0) return std::min(want, dmax);
    const int64_t chunks = (n + 31) / 32, target = 2048;
    int d = 0;
    while (d < dmax && chunks * (1 << (2 * d)) < target) ++d;
    return d;
}

void launch_walk(hts_ctx *c)
{
    const int n = (int)c->n;
    const int warps = (n + 31) / 32;
    const int wb = c->walk_block;  // 32 .. kWalkBlock threads, a multiple of 32
    const bool cnt = c->counters_on != 0;  // counters accumulate while enabled
    const bool seg = c->nseg > 1;
    const SegView sv{c->keys, c->seg_off, c->pre};
    const bool fp64 = c->cfg.precision == HTS_FP64;
    const int depth = seg ? 0 : walk_split_depth(n, c->walk_split, fp64);
    const bool list = !fp64 && !seg && !cnt && list_units(n) > 0;
    SplitView sp{nullptr, nullptr};
    const AnnulusView an{c->minmax, seg ? c->keys : nullptr, c->cfg.split_rule, n - 1};
    dim3 grid((unsigned)((warps * 32 + wb - 1) / wb), 1);
    if (list || depth > 0) {
        CutTables *ct = reinterpret_cast<CutTables *>(c->split_frontier);
        const int grain = list ? std::max(32, n / list_target(n)) : INT_MAX, cap = list ? list_units(n) : kMaxFrontier;
        if (!fp64)
            cut_kernel<<<1, kMaxUnits, 0, c->stream>>>(NodesF{c->nodes32}, c->n_nodes, n, depth, grain, cap, ct,
                                                       c->status);
        else
            cut_kernel<<<1, kMaxUnits, 0, c->stream>>>(NodesD{c->nodes64}, c->n_nodes, n, depth, grain, cap, ct,
                                                       c->status);
        c->launches += 1;
        sp = SplitView{ct, c->split_part};
        grid.y = 1u << (2 * depth);
    }
    c->launches += 1;
    // blocks in order of their cost in the previous walk, when the grid is
    // more than one wave (resident threads per SM: 2048)
    const bool balance = !list && depth == 0 && (int64_t)grid.x > (int64_t)c->sm_count * (2048 / wb);
    const BlockOrder bo{balance ? c->walk_order : nullptr, balance ? c->walk_cost : nullptr};
#define HTS_WALK(P, NODES, SPTS, GF, CT, SG, SPL)                                                    \
    walk_##P##_kernel<GF, CT, SG, SPL><<<grid, wb, 0, c->stream>>>(n, NODES, c->n_nodes, SPTS, c->cnt, c->idx, \
                                                                   c->frep, c->zi, c->counters, sv, sp HTS_X##P, bo)
#define HTS_Xf32 , an
#define HTS_Xf64
#define HTS_WALK_GF(P, NODES, SPTS, GF)                                                                   \
    if (depth > 0) {                                                                                       \
        if (cnt) HTS_WALK(P, NODES, SPTS, GF, true, false, true); else HTS_WALK(P, NODES, SPTS, GF, false, false, true); \
    } else if (cnt) {                                                                                      \
        if (seg) HTS_WALK(P, NODES, SPTS, GF, true, true, false); else HTS_WALK(P, NODES, SPTS, GF, true, false, false); \
    } else {                                                                                               \
        if (seg) HTS_WALK(P, NODES, SPTS, GF, false, true, false); else HTS_WALK(P, NODES, SPTS, GF, false, false, false); \
    }
#define HTS_SUM(GF, SPL)                                                                                          \
    sum_f32_kernel<GF, SPL><<<dim3((unsigned)warps, grid.y), 32 * kSumWarps, 0, c->stream>>>(n, c->nodes32, c->n_nodes, c->spts32, c->cnt, c->idx, c->frep, \
                                                        c->zi, sp, lv, an)
#define HTS_WALK_ALL(P, NODES, SPTS)                                \
    if (c->cfg.grad_form == HTS_EXACT_KL) {                          \
        HTS_WALK_GF(P, NODES, SPTS, 0)                               \
    } else {                                                         \
        HTS_WALK_GF(P, NODES, SPTS, 1)                               \
    }
    if (list) {
        const ListView lv{c->list_entries, c->list_head, c->list_flags, c->list_flags + kListPools, list_units(n),
                          warps, list_per_pool(n)};
        cudaMemsetAsync(c->list_flags, 0, sizeof(int) * (size_t)list_flags(n), c->stream);
        list_f32_kernel<<<dim3((unsigned)((warps * 32 + kListBlock - 1) / kListBlock), (unsigned)lv.units), kListBlock,
                          0, c->stream>>>(n, c->nodes32, c->spts32, c->cnt, sp.cut, lv);
        c->launches += 1;
        if (c->cfg.grad_form == HTS_EXACT_KL) {
            if (depth > 0) HTS_SUM(0, true); else HTS_SUM(0, false);
        } else {
            if (depth > 0) HTS_SUM(1, true); else HTS_SUM(1, false);
        }
    } else if (!fp64) {
        HTS_WALK_ALL(f32, c->nodes32, c->spts32)
    } else {
        HTS_WALK_ALL(f64, c->nodes64, c->spts64)
    }
    if (balance) {
        walk_order_kernel<<<1, 1024, 0, c->stream>>>(c->walk_cost, (int)grid.x, c->walk_order);
        c->launches += 1;
    }
#undef HTS_WALK_ALL
#undef HTS_SUM
#undef HTS_WALK
#undef HTS_WALK_GF
    if (depth > 0) {
        const unsigned cb = (unsigned)(((int64_t)n * 4 + kCombineBlock - 1) / kCombineBlock);
        const int *nsums = &reinterpret_cast<const CutTables *>(c->split_frontier)->nsums;
        if (!fp64)
            walk_combine_kernel<PointF, float><<<cb, kCombineBlock, 0, c->stream>>>(
                n, c->spts32, c->idx, reinterpret_cast<const float *>(c->split_part), nsums, c->frep, c->zi);
        else
            walk_combine_kernel<PointD, double><<<cb, kCombineBlock, 0, c->stream>>>(
                n, c->spts64, c->idx, reinterpret_cast<const double *>(c->split_part), nsums, c->frep, c->zi);
        c->launches += 1;
    }
}

size_t walk_split_frontier_bytes() { return sizeof(CutTables); }

int exact_split(int64_t n)
{
    constexpr int64_t kTargetBlocks = 1216;  // 8 blocks of 64 threads on each of 152 SMs
    const int64_t blocks = (n + kExactBlock - 1) / kExactBlock;
    if (blocks <= 0 || blocks >= kTargetBlocks) return 1;
    return (int)std::min<int64_t>(blocks, (kTargetBlocks + blocks - 1) / blocks);
}

void launch_exact(hts_ctx *c)
{
    ExactArgs A;
    A.n = (int)c->n;
    A.split = exact_split(c->n);
    A.frep = c->frep;
    A.zi = c->zi;
    A.part = reinterpret_cast<double4_32a *>(c->exact_part);
    A.seg_of = c->nseg > 1 ? c->seg_of : nullptr;
    A.seg_off = c->seg_off;
    const dim3 grid((unsigned)((A.n + kExactBlock - 1) / kExactBlock), (unsigned)A.split);
    const int cb = (A.n + 255) / 256;
    c->launches += A.split > 1 ? 2 : 1;
    if (c->cfg.precision == HTS_FP32_MIXED) {
        if (c->cfg.grad_form == HTS_EXACT_KL)
            exact_f32_kernel<0><<<grid, kExactBlock, 0, c->stream>>>(c->pts32, A);
        else
            exact_f32_kernel<1><<<grid, kExactBlock, 0, c->stream>>>(c->pts32, A);
        if (A.split > 1) exact_combine_kernel<PointF><<<cb, 256, 0, c->stream>>>(c->pts32, A);
    } else {
        if (c->cfg.grad_form == HTS_EXACT_KL)
            exact_f64_kernel<0><<<grid, kExactBlock, 0, c->stream>>>(c->pts64, A);
        else
            exact_f64_kernel<1><<<grid, kExactBlock, 0, c->stream>>>(c->pts64, A);
        if (A.split > 1) exact_combine_kernel<PointD><<<cb, 256, 0, c->stream>>>(c->pts64, A);
    }
}

}  // namespace hts
