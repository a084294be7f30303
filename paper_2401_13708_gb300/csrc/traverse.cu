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
// Two forms: direct (walk_*: the terms are added as the cursor goes) and listed
// (list_*: many warps per chunk, one per subtree, write down which interactions
// each lane takes; sum_*: the terms of the listed ones, in the order of the walk
// in float32).  launch_walk chooses by size and precision.
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
constexpr int kListBlock = 128;
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

struct NodesF {  // cell test, points and skip index
    const NodeF *nodes;
    __device__ bool cell(int k) const { return nodes[k].count >= 2.0f; }
    __device__ int points(int k) const { return (int)nodes[k].count; }
    __device__ int skip(int k) const { return nodes[k].skip; }
};

// Interaction lists between list_f32_kernel and sum_f32_kernel: pages of up
// to 32 interactions (the node and the lanes of the chunk that take it).  The
// first page of every (chunk, unit) has a fixed place; further ones come from
// pools (chunk mod kListPools, so that the atomic counters are spread).  Where
// a pool runs out, float32 chunks that found it empty are flagged and walked
// directly by sum_f32_kernel (the same sums).  Direct float64 sums differ in
// their last bits, and which chunk finds the pool empty depends on timing: there
// all chunks of the pool are walked directly (ran_out).
constexpr int kPage = 32;
constexpr int kListPools = 256;

struct ListView {
    uint2 *entries;    // [page][kPage]: node, lane mask
    int2 *head;        // per page: interactions held, next page (-1: none)
    int *taken;        // per pool: pages taken
    int *direct;       // per chunk: it found its pool empty
    int units;         // first pages per chunk
    int chunks;
    int per_pool;      // further pages per pool
    // more pages were asked for than the pool has: the same in every run (a
    // warp asks until it is done or is refused)
    __device__ bool ran_out(int chunk) const { return taken[chunk & (kListPools - 1)] > per_pool; }
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

// Notes an interaction that some lane takes.
__device__ __forceinline__ void batch_add(BatchF &B, int lane, int node, unsigned m)
{
    if (lane == B.count) {
        B.node = node;
        B.mask = m;
    }
    B.count += m != 0u ? 1 : 0;
}

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
    batch_add(B, lane, node, m);
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
        batch_add(B, lane, at, __ballot_sync(0xffffffffu, acc && own));
        live = live && !acc;
    }
    return live;
}

// 0, or NaN for a point that is not finite.  No criterion and so no other point
// takes such a point's leaf; through its Z_i the embedding's Z is NaN, and with
// it the gradient of every point (as the exact one).
__device__ __forceinline__ double zero_if_finite(double x, double y) { return (x - x) + (y - y); }

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
    zi[i] = (double)L.rsz.y + zero_if_finite(x, y);
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

// The page a (chunk, unit) warp writes its batches to.
struct ListPage {
    int page;
    __device__ ListPage(const ListView &lv, int chunk, int unit) : page(chunk * lv.units + unit) {}
    __device__ __forceinline__ void write(const ListView &lv, int lane, const BatchF &B) const
    {
        if (lane < B.count) lv.entries[(size_t)page * kPage + lane] = make_uint2((unsigned)B.node, B.mask);
    }
    // The batch fills the page: writes it and takes another (false: none left).
    __device__ __forceinline__ bool next(const ListView &lv, int chunk, int lane, BatchF &B)
    {
        write(lv, lane, B);
        const int pool = chunk & (kListPools - 1);
        int to = 0;
        if (lane == 0) {
            to = atomicAdd(&lv.taken[pool], 1);
            to = to < lv.per_pool ? lv.chunks * lv.units + pool * lv.per_pool + to : -1;
            lv.head[page] = make_int2(B.count, to);
            if (to < 0) lv.direct[chunk] = 1;
        }
        to = __shfl_sync(0xffffffffu, to, 0);
        page = to;
        B.count = 0;
        return to >= 0;
    }
    __device__ __forceinline__ void last(const ListView &lv, int lane, const BatchF &B) const
    {
        write(lv, lane, B);
        if (lane == 0) lv.head[page] = make_int2(B.count, -1);
    }
};

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
    ListPage page(lv, chunk, (int)blockIdx.y);
    while (node < end) {  // (a page holds what a trip can add to kBatchFull)
#pragma unroll
        for (int k = 0; k < kPage - kBatchFull; ++k) node = visit_f32(node, end, lane, L, B, nodes);
        if (B.count > kBatchFull && !page.next(lv, chunk, lane, B)) return;
    }
    page.last(lv, lane, B);
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
        T.il[lane] = have ? c.il : 0.0f;  // (past the count: weight 0 times a term that must be finite)
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

// ---- float64 walk ---------------------------------------------------------
// The float64 pipe (two lanes a cycle per SM) bounds it, so float64 is spent
// on the pair terms alone, on lanes that need them:
//   - the criterion is decided in float32 from the float32 nodes, whose
//     positions are hi/lo pairs, wherever the float32 delta is further from
//     the threshold than its error; otherwise (about one test in 10^5) in
//     float64, so every decision is the float64 one;
//   - accepted interactions go to a ring of four groups of 32, and every lane
//     takes its own ones in order: a lane that takes few in one group goes on
//     to the next while the others catch up (a lane takes about 70% of its
//     warp's interactions).
// Walk at N = 70,000, theta = 0.5: 15.1 ms visit by visit, 10.1 ms with whole
// batches of 128, 8.2 ms with the ring; 21.6 ms before the pair terms of
// f64math.cuh.
constexpr int kWalkBlockD = 128;
constexpr float kSureF32 = 3.8146973e-6f;   // 2^-18
constexpr float kNearF32 = 8.8817842e-16f;  // 2^-50

struct __align__(16) TileD {
    double2 xy[128];
    double2 ic[128];   // conformal factor; points (negative: a bucket)
    int node[128];
    unsigned mask[128];
};

struct LaneD {
    double x, y, twoil;
    double rx, ry, rs, z;
    float2 qh, ql;  // the position as hi / lo float pairs
    float twoilf;
    int p, own, resume;
};

__device__ __forceinline__ void load_lane(LaneD &L, int chunk, int lane, int n, const PointD *__restrict__ spts,
                                          const int *__restrict__ leaf)
{
    L.p = chunk * 32 + lane;
    const int k = min(L.p, n - 1);
    const PointD q = spts[k];
    L.x = q.x;
    L.y = q.y;
    L.twoil = 2.0 * q.il;
    split_f32(q.x, L.qh.x, L.ql.x);
    split_f32(q.y, L.qh.y, L.ql.y);
    L.twoilf = (float)L.twoil;
    L.own = leaf[k];
    L.rx = L.ry = L.rs = L.z = 0.0;
}

template <int GF>
__device__ __forceinline__ void add_pair_f64(LaneD &L, double x, double y, double il, double mult)
{
    const double dx = L.x - x, dy = L.y - y;
    const double s = fma(dx, dx, dy * dy);
    const PairD t = pair_terms_f64<GF>(s * L.twoil * il);
    const double k = mult * t.rep * il;
    L.rx = fma(k, dx, L.rx);
    L.ry = fma(k, dy, L.ry);
    L.rs = fma(k, s, L.rs);
    L.z = fma(mult, t.w, L.z);
}

// A depth-29 bucket: each of its points (not the lane's own).
template <int GF>
__device__ __forceinline__ void add_bucket_f64(LaneD &L, int node, const NodeD *__restrict__ nodes64,
                                               const PointD *__restrict__ spts, int n, unsigned &pairs)
{
    const NodeD c = nodes64[node];
    const int lo = c.pos, cnt = -c.count;
    if (lo < 0 || cnt <= 0 || lo + cnt > n) return;
    for (int k = 0; k < cnt; ++k) {
        if (lo + k == L.p) continue;
        const PointD o = spts[lo + k];
        add_pair_f64<GF>(L, o.x, o.y, o.il, 1.0);
        ++pairs;
    }
}

// A lane's criterion at a node (r_cell / d < theta  <=>  delta > thr); `ask`:
// the lane is open there.  The float32 delta is off by less than 2^-20 of
// itself where |Delta| > 2^-25: the compensated difference by 3 x 2^-24 of
// itself and 2^-47, il, thr and the products by a few 2^-24 more; 2^-18 is
// allowed.  Leaves and buckets have threshold -1.
__device__ __forceinline__ bool accepts_f64(const LaneD &L, bool ask, const NodeF &c, int node,
                                            const NodeD *__restrict__ nodes64)
{
    const float2 d = delta2(L.qh, L.ql, make_float2(c.xh, c.yh), make_float2(c.xl, c.yl));
    const float s = fmaf(d.x, d.x, d.y * d.y);
    const float delta = s * L.twoilf * c.il, margin = c.thr * kSureF32;
    bool acc = delta > c.thr;
    const bool unsure = ask && c.count >= 2.0f && (fabsf(delta - c.thr) <= margin || s < kNearF32) && c.thr < 3e38f;
    if (__any_sync(0xffffffffu, unsure)) {
        if (unsure) {
            const NodeD e = nodes64[node];
            const double dx = L.x - e.x, dy = L.y - e.y;
            acc = fma(dx, dx, dy * dy) * L.twoil * e.il > e.thr;
        }
        __syncwarp();
    }
    return ask && acc;
}

// One visit (as visit_f32); `m`: the lanes that take the node's interaction.
__device__ __forceinline__ int visit_f64(int node, int end, LaneD &L, unsigned &m, const NodeF *__restrict__ nodes,
                                         const NodeD *__restrict__ nodes64)
{
    const NodeF c = load_node(nodes, node);
    const bool open = node >= L.resume && node < end;
    const bool acc = accepts_f64(L, open && node != L.own, c, node, nodes64);
    m = __ballot_sync(0xffffffffu, acc);
    const bool down = __any_sync(0xffffffffu, open && !acc);
    if (acc) L.resume = c.skip;
    return down ? node + 1 : c.skip;
}

// The ring: group i of those held (0: the oldest) is at (head + i) mod 4 of the
// warp's tile; bit e of b_i: the lane has interaction e of group i to add.
struct RingD {
    unsigned b0, b1, b2, b3;
    int head, held;
};

// The nodes and masks of `count` interactions of the next group are in the
// tile: fetches their data.
__device__ __forceinline__ void ring_push(RingD &R, int count, int lane, TileD &T, const NodeD *__restrict__ nodes64)
{
    __syncwarp();
    const int e = ((R.head + R.held) & 3) * 32 + lane;
    const bool have = lane < count;
    if (have) {
        const NodeD c = nodes64[T.node[e]];
        T.xy[e] = make_double2(c.x, c.y);
        T.ic[e] = make_double2(c.il, (double)c.count);
    }
    const unsigned b = transpose_bits(have ? T.mask[e] : 0u, lane);
    R.b0 = R.held == 0 ? b : R.b0;
    R.b1 = R.held == 1 ? b : R.b1;
    R.b2 = R.held == 2 ? b : R.b2;
    R.b3 = R.held == 3 ? b : R.b3;
    ++R.held;
    __syncwarp();
}

// Adds interactions until every lane is done with the oldest group, and frees it.
template <int GF>
__device__ __forceinline__ void ring_drain(RingD &R, LaneD &L, TileD &T, const NodeD *__restrict__ nodes64,
                                           const PointD *__restrict__ spts, int n, unsigned &pairs)
{
    while (__any_sync(0xffffffffu, R.b0 != 0u)) {
        int e = -1;  // the lane's next interaction
        if (R.b0) {
            e = __ffs((int)R.b0) - 1;
            R.b0 &= R.b0 - 1u;
        } else if (R.b1) {
            e = __ffs((int)R.b1) + 31;
            R.b1 &= R.b1 - 1u;
        } else if (R.b2) {
            e = __ffs((int)R.b2) + 63;
            R.b2 &= R.b2 - 1u;
        } else if (R.b3) {
            e = __ffs((int)R.b3) + 95;
            R.b3 &= R.b3 - 1u;
        }
        __syncwarp();
        if (e >= 0) {
            e = (e + 32 * R.head) & 127;
            const double2 xy = T.xy[e], ic = T.ic[e];
            if ((long long)bits_of(ic.y) > 0) {
                add_pair_f64<GF>(L, xy.x, xy.y, ic.x, ic.y);
            } else {
                add_bucket_f64<GF>(L, T.node[e], nodes64, spts, n, pairs);
            }
        }
        __syncwarp();
    }
    R.b0 = R.b1;
    R.b1 = R.b2;
    R.b2 = R.b3;
    R.b3 = 0u;
    R.head = (R.head + 1) & 3;
    --R.held;
}

__device__ __forceinline__ void store_lane(const LaneD &L, int sum, int n, const uint32_t *__restrict__ idx,
                                           double2 *frep, double *zi, void *part)
{
    if (L.p >= n) return;
    if (part) {
        reinterpret_cast<double4_32a *>(part)[(size_t)sum * n + L.p] = make_double4_32a(L.rx, L.ry, L.rs, L.z);
        return;
    }
    const uint32_t i = idx[L.p];
    const double il = 0.5 * L.twoil, rsd = il * L.rs;
    frep[i] = make_double2(4.0 * il * (L.rx + rsd * L.x), 4.0 * il * (L.ry + rsd * L.y));
    zi[i] = L.z + zero_if_finite(L.x, L.y);
}

// One warp walks for a chunk (sum `sum` of the cut when there are partial sums).
template <int GF, bool COUNT, bool SEG, bool SPLIT>
__device__ __forceinline__ void walk_f64_chunk(LaneD &L, int n, int lane, const NodeF *__restrict__ nodes,
                                                const NodeD *__restrict__ nodes64, const int *__restrict__ n_nodes,
                                                const PointD *__restrict__ spts, unsigned long long *counters,
                                                const SegView sv, const CutTables *cut, int sum, TileD &T)
{
    unsigned long long c_visit = 0, c_acc = 0, c_pair = 0;
    const bool valid = L.p < n;
    const int m = min(*n_nodes, 2 * n);
    int root = 0, end = m, count = 0;
    if (SEG) segment_range(sv, valid ? L.p : n - 1, m, root, end);
    bool live = valid;
    RingD R{0u, 0u, 0u, 0u, 0, 0};
    if (SPLIT) {  // ancestors first, then the subtree [node, end)
        const Cut &F = cut->sums[sum];
        const int na = F.nanc, owned = F.own;
        for (int k = 0; k < na; ++k) {
            const int at = F.anc[k];
            const bool own = (owned >> k) & 1;
            const bool acc = accepts_f64(L, live, load_node(nodes, at), at, nodes64);
            const unsigned am = __ballot_sync(0xffffffffu, acc && own);
            if (am != 0u) {
                if (lane == 0) {
                    T.node[count] = at;
                    T.mask[count] = am;
                }
                ++count;
            }
            if (COUNT) c_acc += (acc && own) ? 1 : 0;
            live = live && !acc;
        }
        root = F.node;
        end = F.end;
    }
    L.resume = live ? root : INT_MAX;
    int node = SEG ? __shfl_sync(0xffffffffu, root, 0) : root;  // lane 0 holds the first segment
    int stop = SEG ? __reduce_max_sync(0xffffffffu, valid ? end : 0) : end;
    if (!__any_sync(0xffffffffu, live)) stop = node;
    unsigned pairs = 0;
    while (true) {
        while (R.held < 4 && node < stop) {  // fill the next group
            const int base = ((R.head + R.held) & 3) * 32;
            while (count < 32 && node < stop) {
                unsigned am;
                const int at = node;
                if (COUNT && lane == 0) ++c_visit;
                node = visit_f64(node, end, L, am, nodes, nodes64);
                if (am != 0u) {
                    if (lane == 0) {
                        T.node[base + count] = at;
                        T.mask[base + count] = am;
                    }
                    ++count;
                    if (COUNT && ((am >> lane) & 1u)) {
                        const float ct = nodes[at].count;
                        c_acc += ct >= 2.0f ? 1 : 0;
                        c_pair += ct == 1.0f ? 1 : 0;
                    }
                }
            }
            if (count == 32) {
                ring_push(R, 32, lane, T, nodes64);
                count = 0;
            }
        }
        if (count > 0 && R.held < 4) {  // the last interactions
            ring_push(R, count, lane, T, nodes64);
            count = 0;
        }
        if (R.held == 0) break;
        ring_drain<GF>(R, L, T, nodes64, spts, n, pairs);
    }
    if (COUNT) {
        c_pair += pairs;
        for (int o = 16; o > 0; o >>= 1) {
            c_acc += __shfl_xor_sync(0xffffffffu, c_acc, o);
            c_pair += __shfl_xor_sync(0xffffffffu, c_pair, o);
        }
        if (lane == 0) {
            atomicAdd(&counters[0], c_acc);
            atomicAdd(&counters[1], c_pair);
            atomicAdd(&counters[2], c_visit);
            atomicAdd(&counters[3], (unsigned long long)min(32, n - L.p));
        }
    }
}

// Direct walk: one warp per chunk of 32 sorted points (grid.x) and sum (grid.y).
template <int GF, bool COUNT, bool SEG, bool SPLIT>
__global__ void __launch_bounds__(kWalkBlockD) walk_f64_kernel(int n, const NodeF *__restrict__ nodes,
                                                               const NodeD *__restrict__ nodes64,
                                                               const int *__restrict__ n_nodes,
                                                               const PointD *__restrict__ spts,
                                                               const int *__restrict__ leaf,
                                                               const uint32_t *__restrict__ idx, double2 *frep,
                                                               double *zi, unsigned long long *counters,
                                                               const SegView sv, const SplitView sp,
                                                               const BlockOrder bo)
{
    __shared__ TileD tile[kWalkBlockD / 32];
    const int b = logical_block(bo);
    const int chunk = (b * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (chunk * 32 >= n) return;
    if (SPLIT && (int)blockIdx.y >= sp.cut->nsums) return;
    const long long t0 = clock64();
    LaneD L;
    load_lane(L, chunk, lane, n, spts, leaf);
    walk_f64_chunk<GF, COUNT, SEG, SPLIT>(L, n, lane, nodes, nodes64, n_nodes, spts, counters, sv, sp.cut, blockIdx.y,
                                          tile[threadIdx.x >> 5]);
    store_lane(L, blockIdx.y, n, idx, frep, zi, SPLIT ? sp.part : nullptr);
    record_cost(bo, b, t0);
}

// Small problems: lists the interactions of a chunk with one unit of the tree,
// as list_f32_kernel.
__global__ void __launch_bounds__(kListBlock, 6) list_f64_kernel(int n, const NodeF *__restrict__ nodes,
                                                                 const NodeD *__restrict__ nodes64,
                                                                 const PointD *__restrict__ spts,
                                                                 const int *__restrict__ leaf,
                                                                 const CutTables *__restrict__ cut, const ListView lv)
{
    const int chunk = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (chunk >= lv.chunks || (int)blockIdx.y >= cut->nunits) return;
    LaneD L;
    load_lane(L, chunk, lane, n, spts, leaf);
    BatchF B;
    B.node = 0;
    B.mask = 0u;
    B.count = 0;
    const Cut &F = cut->units[blockIdx.y];
    bool live = L.p < n;
    const int na = F.nanc, owned = F.own;
    for (int k = 0; k < na; ++k) {
        const int at = F.anc[k];
        const bool own = (owned >> k) & 1;
        const bool acc = accepts_f64(L, live, load_node(nodes, at), at, nodes64);
        batch_add(B, lane, at, __ballot_sync(0xffffffffu, acc && own));
        live = live && !acc;
    }
    int node = F.node;
    const int end = F.end;
    L.resume = live ? node : INT_MAX;
    if (!__any_sync(0xffffffffu, live)) node = end;
    ListPage page(lv, chunk, (int)blockIdx.y);
    while (node < end) {
#pragma unroll 1
        for (int k = 0; k < kPage - kBatchFull; ++k) {
            unsigned m;
            const int at = node;
            node = visit_f64(node, end, L, m, nodes, nodes64);
            batch_add(B, lane, at, m);
        }
        if (B.count > kBatchFull && !page.next(lv, chunk, lane, B)) return;
    }
    page.last(lv, lane, B);
}

// Blocks evaluate the listed interactions of a chunk (grid.x), a window of up
// to kWindow at a time: in every window a point's interactions are divided
// evenly among the lanes that hold the point, one in each of the warps of the
// chunk's blocks (grid.y), so that the float64 pipe sees full warps whatever
// the lists look like (it is busy 87% of the kernel at N = 70,000; one pair
// term is 39 float64 operations).  The lanes' sums are added in warp order (of several
// blocks: by walk_combine_kernel), so the result is reproducible.
constexpr int kSumBlockD = 192;
constexpr int kWindow = 320;  // (256 - 768 interactions and 4 - 8 warps: within 5% of each other)

struct WindowD {
    double2 xy[kWindow];
    double2 ic[kWindow];                 // conformal factor; points (negative: a bucket)
    int node[kWindow];
    unsigned take[kWindow / 32][32];     // [batch][lane]: the interactions of the batch that the lane's point takes
    double4_32a sums[kSumBlockD / 32][32];
};

template <int GF>
__device__ __forceinline__ void sum_window_f64(LaneD &L, int batches, int share, int shares, int lane, const WindowD &W,
                                               const NodeD *__restrict__ nodes64, const PointD *__restrict__ spts, int n)
{
    int total = 0;
    for (int b = 0; b < batches; ++b) total += __popc(W.take[b][lane]);
    int at = total * share / shares, left = total * (share + 1) / shares - at;  // the lane's share of the point's
    int b = -1;
    unsigned bits = 0u;
    while (__any_sync(0xffffffffu, left > 0)) {
        if (left > 0) {
            while (true) {  // to the next interaction
                const int here = __popc(bits);
                if (at < here) break;
                at -= here;
                bits = W.take[++b][lane];
            }
            for (; at > 0; --at) bits &= bits - 1u;
            const int e = 32 * b + __ffs((int)bits) - 1;
            bits &= bits - 1u;
            --left;
            const double2 xy = W.xy[e], ic = W.ic[e];
            if ((long long)bits_of(ic.y) > 0) {
                add_pair_f64<GF>(L, xy.x, xy.y, ic.x, ic.y);
            } else {
                unsigned pairs = 0;
                add_bucket_f64<GF>(L, W.node[e], nodes64, spts, n, pairs);
            }
        }
        __syncwarp();
    }
}

template <int GF>
__global__ void __launch_bounds__(kSumBlockD) sum_f64_kernel(int n, const NodeF *__restrict__ nodes,
                                                             const NodeD *__restrict__ nodes64,
                                                             const int *__restrict__ n_nodes,
                                                             const PointD *__restrict__ spts,
                                                             const int *__restrict__ leaf,
                                                             const uint32_t *__restrict__ idx, double2 *frep,
                                                             double *zi, const SplitView sp, const ListView lv)
{
    constexpr int kWarps = kSumBlockD / 32, kBatches = kWindow / 32;
    __shared__ union { WindowD window; TileD tile; } S;
    WindowD &W = S.window;
    const int chunk = blockIdx.x, w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int shares = kWarps * (int)gridDim.y, share = (int)blockIdx.y * kWarps + w;
    LaneD L;
    load_lane(L, chunk, lane, n, spts, leaf);
    if (lv.ran_out(chunk)) {  // (the same for all the chunk's blocks)
        if (w > 0) return;
        if (blockIdx.y == 0)  // (the other blocks' sums are zero: every block's are added)
            walk_f64_chunk<GF, false, false, false>(L, n, lane, nodes, nodes64, n_nodes, spts, nullptr, SegView{},
                                                    nullptr, 0, S.tile);
        store_lane(L, blockIdx.y, n, idx, frep, zi, gridDim.y > 1 ? sp.part : nullptr);
        return;
    }
    // batches of up to 32 interactions from consecutive pages, dealt to the
    // warps to fetch; every warp follows the same pages
    int slot = 0, fill = 0;
    const int units = sp.cut->nunits;
    unsigned mask = 0u;
    auto done = [&]() {
        if (slot % kWarps == w) {
            __syncwarp();
            const int e = 32 * slot + lane;
            if (lane < fill) {
                const NodeD c = nodes64[W.node[e]];
                W.xy[e] = make_double2(c.x, c.y);
                W.ic[e] = make_double2(c.il, (double)c.count);
            }
            W.take[slot][lane] = transpose_bits(lane < fill ? mask : 0u, lane);
        }
        ++slot;
        fill = 0;
    };
    auto flush = [&]() {
        __syncthreads();
        sum_window_f64<GF>(L, slot, share, shares, lane, W, nodes64, spts, n);
        __syncthreads();
        slot = 0;
    };
    for (int ub = 0; ub < units; ub += 32) {
        const int2 h = ub + lane < units ? lv.head[chunk * lv.units + ub + lane] : make_int2(0, -1);
        unsigned todo = __ballot_sync(0xffffffffu, h.x > 0);
        while (todo) {
            const int j = __ffs((int)todo) - 1;
            todo &= todo - 1;
            int page = chunk * lv.units + ub + j;
            int count = __shfl_sync(0xffffffffu, h.x, j), next = __shfl_sync(0xffffffffu, h.y, j);
            while (true) {
                if (fill + count > 32) {
                    done();
                    if (slot == kBatches) flush();
                }
                if (slot % kWarps == w && lane >= fill && lane < fill + count) {
                    const uint2 e = lv.entries[(size_t)page * kPage + lane - fill];
                    W.node[32 * slot + lane] = (int)e.x;
                    mask = e.y;
                }
                fill += count;
                if (next < 0) break;
                page = next;
                const int2 g = lv.head[page];
                count = g.x;
                next = g.y;
            }
        }
    }
    if (fill > 0) done();
    if (slot > 0) flush();
    W.sums[w][lane] = make_double4_32a(L.rx, L.ry, L.rs, L.z);
    __syncthreads();
    if (w > 0) return;
    for (int k = 1; k < kWarps; ++k) {
        const double4_32a v = W.sums[k][lane];
        L.rx += v.x;
        L.ry += v.y;
        L.rs += v.z;
        L.z += v.w;
    }
    store_lane(L, blockIdx.y, n, idx, frep, zi, gridDim.y > 1 ? sp.part : nullptr);
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
__global__ void __launch_bounds__(kMaxUnits) cut_kernel(const NodesF nodes, const int *__restrict__ n_nodes, int n,
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

// The partial sums of a point in order (the cut's subtrees, or the chunks of
// the exact kernel), then the per-point factors.  Four lanes per point, one per quantity, in
// blocks of one warp: the float64 adds and conversions (4 x 64 of each at the
// deepest cut) go to a pipe of two lanes a cycle per SM, so a small problem
// wants them on as many SMs as possible (N = 2000: 38 us with 8 blocks of 256
// points' threads, 6 us with 250 warps).
constexpr int kCombineBlock = 32;

template <typename PT, typename T>
__global__ void __launch_bounds__(kCombineBlock) walk_combine_kernel(int n, const PT *__restrict__ spts,
                                                                     const uint32_t *__restrict__ idx,
                                                                     const T *__restrict__ part,
                                                                     const int *__restrict__ count, int fixed,
                                                                     double2 *frep, double *zi)
{
    const int p = (blockIdx.x * kCombineBlock + threadIdx.x) >> 2, q = threadIdx.x & 3;
    const int k = min(p, n - 1), nf = count ? *count : fixed;
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
    const uint32_t i = idx ? idx[p] : (uint32_t)p;  // sorted positions, or points
    frep[i] = make_double2(4.0 * il * (rx + rsd * x), 4.0 * il * (ry + rsd * y));
    zi[i] = z + zero_if_finite(x, y);
}

// Exact repulsion: one thread per point i, tiles of kExactBlock points j
// staged in shared memory, every pair j != i of the same segment.  A small
// problem has too few i-blocks to fill the GPU, so the j range of each
// i-block is cut into `split` chunks (grid.y): with split == 1 the block
// writes the finished force and Z_i, otherwise raw sums per chunk go to
// `part` and walk_combine_kernel adds them in chunk order (deterministic).
struct ExactArgs {
    int n, split;
    double2 *frep;
    double *zi;
    double4_32a *part;  // [split][n]: sums of k Delta_x, k Delta_y, k s, w
    const unsigned char *seg_of;
    const int64_t *seg_off;
};

// Own segment [jlo, jhi); the union over the block's threads, cut into chunks
// [cbeg, cend).  Returns whether the block's points share one segment.
__device__ __forceinline__ bool exact_ranges(const ExactArgs &A, int i, int &jlo, int &jhi, int &cbeg, int &cend)
{
    int blo = 0, bhi = A.n;
    bool one = true;
    jlo = 0;
    jhi = A.n;
    if (A.seg_of) {
        const int first = blockIdx.x * kExactBlock, last = min(first + kExactBlock, A.n) - 1;
        const int si = A.seg_of[i < A.n ? i : A.n - 1];
        jlo = (int)A.seg_off[si];
        jhi = (int)A.seg_off[si + 1];
        blo = (int)A.seg_off[A.seg_of[first]];
        bhi = (int)A.seg_off[A.seg_of[last] + 1];
        one = A.seg_of[first] == A.seg_of[last];
    }
    const int tiles = (bhi - blo + kExactBlock - 1) / kExactBlock;
    const int per = (tiles + A.split - 1) / A.split;
    cbeg = min(bhi, blo + (int)blockIdx.y * per * kExactBlock);
    cend = min(bhi, cbeg + per * kExactBlock);
    return one;
}

// Adds one exact pair.
template <int GF>
__device__ __forceinline__ void add_exact_f32(float2 qh, float2 ql, float twoil, const PointF &o, float2 &rxy, float2 &rsz)
{
    const float2 d = delta2(qh, ql, make_float2(o.xh, o.yh), make_float2(o.xl, o.yl));
    const float s = fmaf(d.x, d.x, d.y * d.y);
    const PairF t = pair_terms_f32<GF>(s * twoil * o.il);
    const float kk = t.rep * o.il;
    rxy = __ffma2_rn(make_float2(kk, kk), d, rxy);
    rsz = __ffma2_rn(make_float2(kk, 1.0f), make_float2(s, t.w), rsz);
}

template <int GF>
__global__ void __launch_bounds__(kExactBlock) exact_f32_kernel(const PointF *__restrict__ pts, ExactArgs A)
{
    __shared__ PointF tile[kExactBlock];
    const int n = A.n;
    const int i = blockIdx.x * kExactBlock + threadIdx.x;
    int jlo, jhi, cbeg, cend;
    const bool one = exact_ranges(A, i, jlo, jhi, cbeg, cend);
    const PointF q = pts[i < n ? i : n - 1];
    const float2 qh = make_float2(q.xh, q.yh), ql = make_float2(q.xl, q.yl);
    const float twoil = 2.0f * q.il;
    float2 rxy = make_float2(0.f, 0.f), rsz = make_float2(0.f, 0.f);  // paired sums, as in the walk
    for (int base = cbeg; base < cend; base += kExactBlock) {
        int j = base + threadIdx.x;
        if (j < cend) tile[threadIdx.x] = pts[j];
        __syncthreads();
        const int cnt = min(kExactBlock, cend - base);
        // every pair of a full tile off the diagonal counts where the block's
        // points share one segment: no tests.  Otherwise the sums keep their
        // values where a pair does not count (with weight 0 a point that is not
        // finite would reach other segments: 0 x NaN is NaN).  Four pairs in
        // flight either way: a block on a boundary passes over both segments and
        // decides the kernel's time (two segments of 30,000 points: 4.9 ms with a
        // branch around the pair)
        const bool plain = cnt == kExactBlock && one && (base + cnt <= blockIdx.x * kExactBlock ||
                                                               base >= (blockIdx.x + 1) * kExactBlock);
        if (plain) {
#pragma unroll 4
            for (int k = 0; k < kExactBlock; ++k) add_exact_f32<GF>(qh, ql, twoil, tile[k], rxy, rsz);
        } else {
#pragma unroll 4
            for (int k = 0; k < cnt; ++k) {
                const int jj = base + k;
                const bool take = jj != i && jj >= jlo && jj < jhi;
                float2 u = rxy, v = rsz;
                add_exact_f32<GF>(qh, ql, twoil, tile[k], u, v);
                rxy = make_float2(take ? u.x : rxy.x, take ? u.y : rxy.y);
                rsz = make_float2(take ? v.x : rsz.x, take ? v.y : rsz.y);
            }
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
// 40,000 / 100,000 warps 183 / 142 / 205 us).  In float64 the pair terms are
// most of the walk and the listed ones fill the float64 pipe better (N =
// 70,000: 8.2 ms direct, 0.5 + 7.3 ms listed), so the limit is the lists' size.
constexpr int64_t kListWarps = 40000, kListTargetMax = 128;
constexpr int64_t kListMaxN = 1 << 15, kListMaxN64 = 1 << 18;

static int list_target(int64_t n)
{
    const int64_t chunks = std::max<int64_t>((n + 31) / 32, 1);
    return (int)std::max<int64_t>(2, std::min<int64_t>(kListWarps / chunks, kListTargetMax));
}

// First pages per chunk: the cap of the cut into units (a cut by point counts
// overshoots its target; a cut at depth D has up to 4^D subtrees).
int list_units(int64_t n, bool fp64)
{
    if (n > (fp64 ? kListMaxN64 : kListMaxN)) return 0;
    return std::min(kMaxUnits, std::max(4 * list_target(n), walk_split_capacity(n)));
}

// Further pages per pool: 512 pages a chunk (16,384 interactions; theta = 0.5
// lists about 1,000 to 4,000 a chunk), 134 MB at kListMaxN points; above, 256
// a chunk, 537 MB at kListMaxN64.
static int list_per_pool(int64_t n) { return (int)((n + 31) / 32 * (n > kListMaxN ? 256 : 512) / kListPools + 1); }

int64_t list_pages(int64_t n, bool fp64)
{
    const int u = list_units(n, fp64);
    return u ? (n + 31) / 32 * u + (int64_t)list_per_pool(n) * kListPools : 0;
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

// Blocks per chunk that sum a listed float64 walk: four blocks on each of 152
// SMs while there are fewer chunks than SMs (N = 2,000, two / four / six per SM:
// 124 / 108 / 132 us).  The number decides the order of the sums, so it follows
// from the size alone, not from the SMs of the device at hand.
static int f64_sum_blocks(int64_t n)
{
    constexpr int64_t kTargetBlocks = 4 * 152;
    const int64_t chunks = std::max<int64_t>((n + 31) / 32, 1);
    return (int)std::max<int64_t>(1, std::min<int64_t>(kTargetBlocks / chunks, std::min(16, walk_split_capacity(n))));
}

// Whether launch_walk lists the interactions first, given the buffers (float64: a
// depth that was asked for is the cut of the direct walk; float32: the counting
// walk is direct, with the same bits).
bool walk_wants_lists(const hts_ctx *c)
{
    const bool fp64 = c->cfg.precision == HTS_FP64;
    return c->nseg == 1 && (fp64 ? c->walk_split < 0 : !c->counters_on) && list_units(c->n, fp64) > 0;
}

bool walk_lists(const hts_ctx *c) { return c->list_entries && walk_wants_lists(c); }

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
    const bool list = walk_lists(c);
    const int blocks64 = fp64 && list ? f64_sum_blocks(n) : 1;
    const bool split = fp64 && list ? blocks64 > 1 : depth > 0;
    SplitView sp{nullptr, nullptr};
    const AnnulusView an{c->minmax, seg ? c->keys : nullptr, c->cfg.split_rule, n - 1};
    const int wbd = std::min(wb, kWalkBlockD);
    const int block = fp64 ? wbd : wb;
    dim3 grid((unsigned)((warps * 32 + block - 1) / block), 1);
    CutTables *ct = reinterpret_cast<CutTables *>(c->split_frontier);
    if (list || split) {
        const int grain = list ? std::max(32, n / list_target(n)) : INT_MAX, cap = list ? list_units(n, fp64) : kMaxFrontier;
        cut_kernel<<<1, kMaxUnits, 0, c->stream>>>(NodesF{c->nodes32}, c->n_nodes, n, depth, grain, cap, ct, c->status);
        c->launches += 1;
        sp = SplitView{ct, c->split_part};
        grid.y = 1u << (2 * depth);
    }
    c->launches += 1;
    // blocks in order of their cost in the previous walk, when the grid is
    // more than one wave (resident threads per SM: 2048)
    const bool balance = !list && !split && (int64_t)grid.x > (int64_t)c->sm_count * (2048 / block);
    const BlockOrder bo{balance ? c->walk_order : nullptr, balance ? c->walk_cost : nullptr};
#define HTS_WALK32(GF, CT, SG, SPL)                                                                                  \
    walk_f32_kernel<GF, CT, SG, SPL><<<grid, block, 0, c->stream>>>(n, c->nodes32, c->n_nodes, c->spts32, c->cnt, \
                                                                    c->idx, c->frep, c->zi, c->counters, sv, sp, an, bo)
#define HTS_WALK64(GF, CT, SG, SPL)                                                                             \
    walk_f64_kernel<GF, CT, SG, SPL><<<grid, block, 0, c->stream>>>(n, c->nodes32, c->nodes64, c->n_nodes,   \
                                                                    c->spts64, c->cnt, c->idx, c->frep, c->zi, \
                                                                    c->counters, sv, sp, bo)
#define HTS_SUM(GF, CT, SG, SPL)                                                                                     \
    sum_f32_kernel<GF, SPL><<<dim3((unsigned)warps, grid.y), 32 * kSumWarps, 0, c->stream>>>(                        \
        n, c->nodes32, c->n_nodes, c->spts32, c->cnt, c->idx, c->frep, c->zi, sp, lv, an)
#define HTS_WALK_GF(K, GF)                                                                       \
    if (split) {                                                                                 \
        if (cnt) K(GF, true, false, true); else K(GF, false, false, true);                       \
    } else if (cnt) {                                                                            \
        if (seg) K(GF, true, true, false); else K(GF, true, false, false);                       \
    } else {                                                                                     \
        if (seg) K(GF, false, true, false); else K(GF, false, false, false);                     \
    }
#define HTS_WALK(K)                                \
    if (c->cfg.grad_form == HTS_EXACT_KL) {        \
        HTS_WALK_GF(K, 0)                          \
    } else {                                       \
        HTS_WALK_GF(K, 1)                          \
    }
    if (list) {
        const ListView lv{c->list_entries, c->list_head, c->list_flags, c->list_flags + kListPools, list_units(n, fp64),
                          warps, list_per_pool(n)};
        cudaMemsetAsync(c->list_flags, 0, sizeof(int) * (size_t)list_flags(n), c->stream);
        const dim3 lgrid((unsigned)((warps * 32 + kListBlock - 1) / kListBlock), (unsigned)lv.units);
        c->launches += 1;
        if (fp64) {
            if (cnt) {  // (the direct walk's float64 sums differ in their last bits: it only counts)
                if (c->cfg.grad_form == HTS_EXACT_KL)
                    walk_f64_kernel<0, true, false, false><<<dim3(grid.x), block, 0, c->stream>>>(
                        n, c->nodes32, c->nodes64, c->n_nodes, c->spts64, c->cnt, c->idx, c->frep, c->zi, c->counters, sv,
                        SplitView{nullptr, nullptr}, bo);
                else
                    walk_f64_kernel<1, true, false, false><<<dim3(grid.x), block, 0, c->stream>>>(
                        n, c->nodes32, c->nodes64, c->n_nodes, c->spts64, c->cnt, c->idx, c->frep, c->zi, c->counters, sv,
                        SplitView{nullptr, nullptr}, bo);
                c->launches += 1;
            }
            list_f64_kernel<<<lgrid, kListBlock, 0, c->stream>>>(n, c->nodes32, c->nodes64, c->spts64, c->cnt, sp.cut, lv);
            const dim3 sgrid((unsigned)warps, (unsigned)blocks64);
            if (c->cfg.grad_form == HTS_EXACT_KL)
                sum_f64_kernel<0><<<sgrid, kSumBlockD, 0, c->stream>>>(n, c->nodes32, c->nodes64, c->n_nodes, c->spts64,
                                                                        c->cnt, c->idx, c->frep, c->zi, sp, lv);
            else
                sum_f64_kernel<1><<<sgrid, kSumBlockD, 0, c->stream>>>(n, c->nodes32, c->nodes64, c->n_nodes, c->spts64,
                                                                        c->cnt, c->idx, c->frep, c->zi, sp, lv);
        } else {
            list_f32_kernel<<<lgrid, kListBlock, 0, c->stream>>>(n, c->nodes32, c->spts32, c->cnt, sp.cut, lv);
            HTS_WALK(HTS_SUM)
        }
    } else if (fp64) {
        HTS_WALK(HTS_WALK64)
    } else {
        HTS_WALK(HTS_WALK32)
    }
    if (balance) {
        walk_order_kernel<<<1, 1024, 0, c->stream>>>(c->walk_cost, (int)grid.x, c->walk_order);
        c->launches += 1;
    }
#undef HTS_WALK
#undef HTS_WALK_GF
#undef HTS_SUM
#undef HTS_WALK64
#undef HTS_WALK32
    if (split) {
        const unsigned cb = (unsigned)(((int64_t)n * 4 + kCombineBlock - 1) / kCombineBlock);
        if (!fp64)
            walk_combine_kernel<PointF, float><<<cb, kCombineBlock, 0, c->stream>>>(
                n, c->spts32, c->idx, reinterpret_cast<const float *>(c->split_part), &ct->nsums, 0, c->frep, c->zi);
        else
            walk_combine_kernel<PointD, double><<<cb, kCombineBlock, 0, c->stream>>>(
                n, c->spts64, c->idx, reinterpret_cast<const double *>(c->split_part), list ? nullptr : &ct->nsums, blocks64,
                c->frep, c->zi);
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
    const unsigned cb = (unsigned)(((int64_t)A.n * 4 + kCombineBlock - 1) / kCombineBlock);
    c->launches += A.split > 1 ? 2 : 1;
    if (c->cfg.precision == HTS_FP32_MIXED) {
        if (c->cfg.grad_form == HTS_EXACT_KL)
            exact_f32_kernel<0><<<grid, kExactBlock, 0, c->stream>>>(c->pts32, A);
        else
            exact_f32_kernel<1><<<grid, kExactBlock, 0, c->stream>>>(c->pts32, A);
        if (A.split > 1)
            walk_combine_kernel<PointF, double><<<cb, kCombineBlock, 0, c->stream>>>(A.n, c->pts32, nullptr, c->exact_part,
                                                                                     nullptr, A.split, A.frep, A.zi);
    } else {
        if (c->cfg.grad_form == HTS_EXACT_KL)
            exact_f64_kernel<0><<<grid, kExactBlock, 0, c->stream>>>(c->pts64, A);
        else
            exact_f64_kernel<1><<<grid, kExactBlock, 0, c->stream>>>(c->pts64, A);
        if (A.split > 1)
            walk_combine_kernel<PointD, double><<<cb, kCombineBlock, 0, c->stream>>>(A.n, c->pts64, nullptr, c->exact_part,
                                                                                     nullptr, A.split, A.frep, A.zi);
    }
}

}  // namespace hts
