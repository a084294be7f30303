// sort.cu -- sort of (key, index) pairs (by ranks, or an LSD radix sort) and an
// exclusive int scan.
//
// The tree of Sec. 4.1 is a hierarchy over the keys, so sorting the points
// by key puts every cell's points in one contiguous run.  Up to kRankMax keys
// they are sorted by ranks (sort_by_rank); above, eight stable passes of 8
// bits each (58 key bits + 6 segment bits), one kernel per pass:
//   digit_hist  once per sort: the global histograms of all eight digits
//               (they do not depend on the order of the keys; shared-memory
//               atomics per key and digit), then an exclusive scan of each
//               gives every digit its first slot;
//   onesweep    per pass, one tile per block (1024, 2048 or 4096 keys of
//               256 threads, or 8192 keys of 512 threads, by problem size:
//               tile_keys), tiles taken in launch
//               order from an atomic counter: warp histograms (the lanes
//               sharing a digit from eight ballots, one per digit bit), the
//               tile's per-digit counts published to a status word, and a
//               decoupled look-back over earlier tiles (thread d for digit
//               d, kLookBack status words per round trip) adds up the keys
//               of digit d before this tile; then each key is ranked among
//               equal digits in order and written out.  Look-back spins are
//               bounded: a timeout sets a status bit (reported as an
//               error), and out-of-range positions are never written.
// Traffic per pass: 12 B read + 12 B write per key (+ 8 B read once for the
// histograms).
#include <cuda/atomic>

#include <algorithm>

#include "hts_internal.cuh"

namespace hts {
namespace {

// Sorted tiles and ranks (sort_by_rank) up to kRankMax keys, with larger tiles
// for more keys: the tile sort grows with the tile, the rank search with their
// number.  Measured (tile sort + ranks, us; radix sort's kernels, without the
// gaps between its 11 launches):
//   keys       512-key tiles  1024        2048         4096         radix
//   2,000      4.1 + 4.3      7.1 + 4.1   13.7                      39.9
//   8,192      4.2 + 8.4      7.2 + 5.6   14.0 + 5.0   31.7 + 4.1   42.1
//   20,011     4.2 + 19.1     7.2 + 11.9  14.0 + 8.2   31.8 + 6.0   47.0
//   40,000     4.3 + 37.2     7.2 + 21.1  14.0 + 13.7
//   70,000                    7.3 + 49.5  14.1 + 29.0  31.8 + 18.1  55.9
//   131,071                               14.1 + 48.2  31.7 + 26.9  60.8
//   262,144                               14.1 + 177   31.8 + 95.5  76.4
constexpr int64_t kRankMax = 150000, kRank512 = 8192, kRank1024 = 32768, kRank2048 = 90000;
constexpr int kWaitTestFrom = 4096;  // (hts_set_wait_test)
constexpr int kMinTile = 1024;     // one-sweep tiles hold 1024, 2048, 4096 or 8192 keys (tile_keys)
constexpr int kSortThreads = 256;
constexpr int kScanThreads = 1024;
constexpr int kScanItems = 4;
constexpr int kScanBlock = kScanThreads * kScanItems;

constexpr int kPasses = 8;
constexpr unsigned long long kFlagAgg = 1ull << 62;   // tile count published
constexpr unsigned long long kFlagPre = 2ull << 62;   // inclusive prefix published
constexpr unsigned long long kValMask = (1ull << 62) - 1ull;
constexpr int kSpinLimit = 1 << 22;
constexpr int kLookBack = 8;  // status words loaded per look-back round trip
// above this, 8192-key tiles of 512 threads (4096-key tiles of 256 threads
// serve sizes between 524,288 and this bound when it is raised)
constexpr int64_t kBigTileFrom = 524288;

// Keys per one-sweep tile.  A pass is latency-bound: one block ranks and
// writes its tile in kTile / 256 sequential rounds, so smaller tiles finish
// sooner while there are SMs to spare; large problems take larger tiles
// (fewer look-back steps and status words: every tile of a pass is resident
// at once, so the last tile looks back over nearly all of them).  Measured
// sort times per iteration: 20,000 keys 156 / 110 / 87 us with 4096 / 2048 /
// 1024-key tiles, 262,145 keys 174 / 143 / 152 us, 1,000,000 keys 283 / 295 /
// 301 us (before the ballot ranking and the batched look-back); with them,
// 1,000,000 keys 198 us with 4096-key tiles and 185 us with 8192 keys of 512
// threads (700,000 keys: 181 / 180 us).
int tile_keys(int64_t n)
{
    return n <= 196608 ? 1024 : n <= 524288 ? 2048 : n <= kBigTileFrom ? 4096 : 8192;
}

// The lanes of the warp whose 8-bit digit equals this lane's, from eight
// ballots (one per digit bit); a lane that is not `ok` matches only itself.
// Every lane of the warp makes the call.
__device__ __forceinline__ unsigned digit_peers(int dg, bool ok, int lane)
{
    const unsigned valid = __ballot_sync(0xffffffffu, ok);
    unsigned m = ok ? valid : (1u << lane);
#pragma unroll
    for (int b = 0; b < 8; ++b) {
        const unsigned bb = __ballot_sync(0xffffffffu, (dg >> b) & 1);
        m &= ((dg >> b) & 1) ? bb : ~bb;
    }
    return m;
}

// Global histograms of all eight digits; hist[pass][digit] (2048 ints).
template <int kTile>
__global__ void __launch_bounds__(kSortThreads) digit_hist_kernel(const uint64_t *__restrict__ keys, int n,
                                                                  int *hist)
{
    __shared__ int h[kPasses][256];
    for (int k = threadIdx.x; k < kPasses * 256; k += kSortThreads) (&h[0][0])[k] = 0;
    __syncthreads();
    const int base = blockIdx.x * kTile;
    for (int r = 0; r < kTile / kSortThreads; ++r) {
        const int i = base + r * kSortThreads + threadIdx.x;
        const bool ok = i < n;
        const uint64_t key = ok ? keys[i] : 0ull;
#pragma unroll
        for (int p = 0; p < kPasses; ++p) {
            if (ok) atomicAdd(&h[p][(int)((key >> (8 * p)) & 0xFFu)], 1);
        }
    }
    __syncthreads();
    for (int k = threadIdx.x; k < kPasses * 256; k += kSortThreads) {
        const int v = (&h[0][0])[k];
        if (v) atomicAdd(&hist[k], v);
    }
}

// hist[pass][digit] -> exclusive prefix over digits (in place), one warp per pass.
__global__ void digit_offsets_kernel(int *hist)
{
    const int p = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (p >= kPasses) return;
    int *h = hist + p * 256;
    int v[8], local = 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        v[k] = h[lane * 8 + k];
        local += v[k];
    }
    int incl = local;
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    int run = incl - local;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        h[lane * 8 + k] = run;
        run += v[k];
    }
}

template <int kTile, int kThreads = kSortThreads>
__global__ void __launch_bounds__(kThreads) onesweep_kernel(const uint64_t *__restrict__ kin,
                                                                const uint32_t *__restrict__ vin,
                                                                uint64_t *__restrict__ kout,
                                                                uint32_t *__restrict__ vout, int n, int shift,
                                                                const int *__restrict__ digit_off,
                                                                unsigned long long *tile_status, int *tile_ctr,
                                                                int *status, int spin_limit, int withhold_first)
{
    constexpr int kW = kThreads / 32;  // warps per tile
    constexpr int kPerWarp = kTile / kW;
    constexpr int kRounds = kPerWarp / 32;
    __shared__ int wh[kW][256];
    __shared__ int s_tile;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int k = threadIdx.x; k < kW * 256; k += kThreads) (&wh[0][0])[k] = 0;
    if (threadIdx.x == 0) s_tile = atomicAdd(tile_ctr, 1);  // tiles in launch order
    __syncthreads();
    const int tile = s_tile;

    const int base = tile * kTile + w * kPerWarp;
    const unsigned lt = (1u << lane) - 1u;
    uint64_t key[kRounds];
    uint32_t val[kRounds];
    unsigned peers[kRounds];  // lanes of the round with the same digit (kept for the scatter)
#pragma unroll
    for (int r = 0; r < kRounds; ++r) {
        int i = base + r * 32 + lane;
        bool ok = i < n;
        key[r] = ok ? kin[i] : 0ull;
        val[r] = ok ? vin[i] : 0u;
        const int dg = (int)((key[r] >> shift) & 0xFFu);
        const unsigned m = digit_peers(dg, ok, lane);
        peers[r] = m;
        if (ok && (m & lt) == 0u) wh[w][dg] += __popc(m);
        __syncwarp();
    }
    __syncthreads();
    if (threadIdx.x < 256) {
        const int d = threadIdx.x;  // the first 256 threads: one digit each
        int cnt = 0;
#pragma unroll
        for (int k = 0; k < kW; ++k) {
            const int t = wh[k][d];
            wh[k][d] = cnt;  // exclusive prefix over the warps of this tile
            cnt += t;
        }
        cuda::atomic_ref<unsigned long long, cuda::thread_scope_device> mine(tile_status[(size_t)tile * 256 + d]);
        long long excl = 0;
        if (tile == 0) {
            // (withhold_first: the wait test of hts_set_wait_test; the later
            // tiles' waits then run out)
            if (!withhold_first) mine.store(kFlagPre | (unsigned long long)cnt, cuda::memory_order_relaxed);
        } else {
            mine.store(kFlagAgg | (unsigned long long)cnt, cuda::memory_order_relaxed);
            // decoupled look-back: add tile counts until an inclusive prefix,
            // kLookBack earlier tiles per round trip (their loads are
            // independent; a tile whose word is not yet published is waited
            // for in order).  Tile 0 always holds an inclusive prefix, so the
            // walk ends there at the latest.
            bool done = false;
            for (int t = tile - 1; t >= 0 && !done; t -= kLookBack) {
                unsigned long long v[kLookBack];
#pragma unroll
                for (int j = 0; j < kLookBack; ++j)
                    v[j] = t - j >= 0 ? cuda::atomic_ref<unsigned long long, cuda::thread_scope_device>(
                                            tile_status[(size_t)(t - j) * 256 + d])
                                            .load(cuda::memory_order_relaxed)
                                      : 0ull;
#pragma unroll
                for (int j = 0; j < kLookBack; ++j) {
                    if (done || t - j < 0) break;
                    unsigned long long vj = v[j];
                    int spins = 0;
                    while ((vj >> 62) == 0ull && ++spins < spin_limit) {
                        __nanosleep(64);
                        vj = cuda::atomic_ref<unsigned long long, cuda::thread_scope_device>(
                                 tile_status[(size_t)(t - j) * 256 + d])
                                 .load(cuda::memory_order_relaxed);
                    }
                    if ((vj >> 62) == 0ull) {  // gave up: report (HTS_ETIMEOUT), positions invalid
                        atomicOr(status, 128);
                        excl = (long long)n;
                        done = true;
                        break;
                    }
                    excl += (long long)(vj & kValMask);
                    done = (vj & kFlagPre) && !(vj & kFlagAgg);
                }
            }
            mine.store(kFlagPre | (unsigned long long)(excl + cnt), cuda::memory_order_relaxed);
        }
        const int off = digit_off[d] + (int)min(excl, (long long)n);
#pragma unroll
        for (int k = 0; k < kW; ++k) wh[k][d] += off;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kRounds; ++r) {
        int i = base + r * 32 + lane;
        bool ok = i < n;
        const int dg = (int)((key[r] >> shift) & 0xFFu);
        int pos = 0;
        if (ok) pos = wh[w][dg] + __popc(peers[r] & lt);
        __syncwarp();
        if (ok && (peers[r] & lt) == 0u) wh[w][dg] += __popc(peers[r]);
        __syncwarp();
        if (ok) {
            if (pos >= 0 && pos < n) {
                kout[pos] = key[r];
                vout[pos] = val[r];
            } else {
                atomicOr(status, 4);
            }
        }
    }
}

// ---- exclusive scan --------------------------------------------------------

// kCount: the input is the number of tree nodes that start at each sorted point
// (CountArgs), which is also stored.
template <bool kCount>
__global__ void __launch_bounds__(kScanThreads) scan_block_kernel(const int *in, const CountArgs counts, int *out,
                                                                  int64_t len, int *block_sums)
{
    __shared__ int warp_tot[kScanThreads / 32];
    int64_t base = (int64_t)blockIdx.x * kScanBlock + (int64_t)threadIdx.x * kScanItems;
    int v[kScanItems];
    int local = 0;
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
        int64_t i = base + k;
        if (kCount) {
            v[k] = 0;
            if (i < counts.n) {
                const bool leaf = counts.n == 1 || quad_level(counts.pref[counts.leaf_parent[i]]) < kLevels;
                v[k] = __popc(counts.mask[i]) + (leaf ? 1 : 0);
            }
            if (i < len) counts.cnt[i] = v[k];
        } else {
            v[k] = i < len ? in[i] : 0;
        }
        local += v[k];
    }
    int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int incl = local;
    for (int o = 1; o < 32; o <<= 1) {
        int t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) warp_tot[w] = incl;
    __syncthreads();
    if (w == 0) {
        int t = lane < kScanThreads / 32 ? warp_tot[lane] : 0;
        int s = t;
        for (int o = 1; o < 32; o <<= 1) {
            int u = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += u;
        }
        if (lane < kScanThreads / 32) warp_tot[lane] = s - t;  // exclusive warp offsets
        if (lane == 31 && block_sums) block_sums[blockIdx.x] = s;
    }
    __syncthreads();
    int run = warp_tot[w] + incl - local;
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
        int64_t i = base + k;
        if (i < len) out[i] = run;
        run += v[k];
    }
}

__global__ void add_offsets_kernel(int *out, int64_t len, const int *__restrict__ offs)
{
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < len) out[i] += offs[i / kScanBlock];
}

}  // namespace

int64_t scan_tmp_size(int64_t len)
{
    int64_t total = 0;
    while (len > kScanBlock) {
        len = (len + kScanBlock - 1) / kScanBlock;
        total += len + 1;
    }
    return total + 1;
}

// Exclusive scan of len ints (in and out may alias only if equal).
// Returns the number of kernels launched.
static int scan_exclusive(const int *in, int *out, int64_t len, int *tmp, cudaStream_t s)
{
    if (len <= 0) return 0;
    int64_t blocks = (len + kScanBlock - 1) / kScanBlock;
    if (blocks == 1) {
        scan_block_kernel<false><<<1, kScanThreads, 0, s>>>(in, CountArgs{}, out, len, nullptr);
        return 1;
    }
    int *sums = tmp;
    scan_block_kernel<false><<<(unsigned)blocks, kScanThreads, 0, s>>>(in, CountArgs{}, out, len, sums);
    int k = scan_exclusive(sums, sums, blocks, tmp + blocks + 1, s);
    add_offsets_kernel<<<(unsigned)((len + 255) / 256), 256, 0, s>>>(out, len, sums);
    return k + 2;
}

// Exclusive scan of the node counts of n sorted points (out: n + 1 entries).
int scan_counts(const CountArgs &counts, int *out, int *tmp, cudaStream_t s)
{
    const int64_t len = (int64_t)counts.n + 1, blocks = (len + kScanBlock - 1) / kScanBlock;
    int *sums = tmp;
    scan_block_kernel<true><<<(unsigned)blocks, kScanThreads, 0, s>>>(nullptr, counts, out, len,
                                                                     blocks > 1 ? sums : nullptr);
    if (blocks == 1) return 1;
    const int k = scan_exclusive(sums, sums, blocks, tmp + blocks + 1, s);
    add_offsets_kernel<<<(unsigned)((len + 255) / 256), 256, 0, s>>>(out, len, sums);
    return k + 2;
}

namespace {

// ---- sort by ranks ------------------------------------------------------------
// Up to kRankMax keys the eight dependent passes of the radix sort are latency
// (11 launches), and comparing is cheaper.  A block
// sorts a tile of kTile keys in shared memory: runs of 64 by counting the
// smaller keys of the run, then runs of 512 and the tile by counting, for every
// key, the smaller keys of each other run (binary searches).  One more kernel
// finds every key's place among all tiles the same way, the first steps of
// each search in a sample of every 32nd key.  Equal keys stay in index order:
// runs and tiles hold consecutive indices, so an earlier one's equal keys come
// before and a later one's after.  The tail of the last tile is filled with
// 2^64 - 1, which a point can have as its key too (segment 63, outermost, angle
// just below a full turn): it is told from the points by its place alone, after
// all of them, where the same counting leaves it.  (A bitonic sort of a
// 2,048-key tile: 22 us.)
constexpr int kRun = 64, kRun2 = 512, kSample = 32;
template <int kTile> constexpr int kTileThreads = kTile < 1024 ? kTile : 1024;

// Keys of a sorted run (kLen, a power of two) that go before `key`: those below
// it and, in a run of earlier indices, those equal to it (below key + 1, or all
// of them where that wraps).
template <int kLen>
__device__ __forceinline__ int count_before(const uint64_t *run, uint64_t key, bool earlier)
{
    const uint64_t lim = key + (earlier ? 1ull : 0ull);
    int c = 0;
#pragma unroll
    for (int s = kLen >> 1; s > 0; s >>= 1)
        if (run[c + s - 1] < lim) c += s;
    c += run[c] < lim ? 1 : 0;
    return earlier && key == ~0ull ? kLen : c;
}

// Merges groups of kLen-key runs (kGroup keys each) of `k` into `ko`.
template <int kTile, int kLen, int kGroup>
__device__ __forceinline__ void merge_runs(const uint64_t *k, const uint16_t *v, uint64_t *ko, uint16_t *vo)
{
#pragma unroll
    for (int q = 0; q < kTile / kTileThreads<kTile>; ++q) {
        const int e = threadIdx.x + q * kTileThreads<kTile>;
        const uint64_t key = k[e];
        const int group = e & ~(kGroup - 1), own = (e & (kGroup - 1)) / kLen;
        int pos = e & (kLen - 1);
#pragma unroll
        for (int r = 0; r < kGroup / kLen; ++r) {
            const int c = count_before<kLen>(k + group + r * kLen, key, r < own);
            pos += r == own ? 0 : c;
        }
        ko[group + pos] = key;
        vo[group + pos] = v[e];
    }
}

template <int kTile>
__global__ void __launch_bounds__(kTileThreads<kTile>) tile_sort_kernel(const uint64_t *kin, int n, uint64_t *kout,
                                                                 uint32_t *vout, uint64_t *sample)
{
    constexpr int kPer = kTile / kTileThreads<kTile>;
    extern __shared__ uint64_t sort_shared[];
    uint64_t *ka = sort_shared, *kb = ka + kTile;
    uint16_t *va = reinterpret_cast<uint16_t *>(kb + kTile), *vb = va + kTile;
    const int base = blockIdx.x * kTile, lane = threadIdx.x & 31;
    uint64_t key[kPer];
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
        const int e = threadIdx.x + q * kTileThreads<kTile>;
        key[q] = base + e < n ? kin[base + e] : ~0ull;
        ka[e] = key[q];
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < kPer; ++q) {  // runs of 64: 32 keys of the other half of the run, 32 of this warp's
        const int e = threadIdx.x + q * kTileThreads<kTile>;
        const uint64_t *run = ka + (e & ~(kRun - 1));
        const int half = e & 32;
        const uint64_t next = key[q] + 1ull, other = half ? next : key[q];
        int rank = 0;
#pragma unroll 8
        for (int j = 0; j < 32; ++j) {
            rank += run[(half ^ 32) + j] < other ? 1 : 0;
            rank += run[half + j] < (j < lane ? next : key[q]) ? 1 : 0;
        }
        if (key[q] == ~0ull) rank += e & (kRun - 1);  // (`next` wrapped: all the earlier ones)
        kb[(e & ~(kRun - 1)) + rank] = key[q];
        vb[(e & ~(kRun - 1)) + rank] = (uint16_t)e;
    }
    __syncthreads();
    merge_runs<kTile, kRun, kRun2>(kb, vb, ka, va);
    __syncthreads();
    if (kTile > kRun2) {
        merge_runs<kTile, kRun2, kTile>(ka, va, kb, vb);
        __syncthreads();
    }
    const uint64_t *ks = kTile > kRun2 ? kb : ka;
    const uint16_t *vs = kTile > kRun2 ? vb : va;
    for (int e = threadIdx.x; e < kTile; e += kTileThreads<kTile>) {
        if (base + e < n) {
            kout[base + e] = ks[e];
            vout[base + e] = (uint32_t)(base + vs[e]);
        }
        if (sample && (e & (kSample - 1)) == kSample - 1) sample[(base + e) / kSample] = ks[e];
    }
}

// Every key's place among all tiles: its place in its own tile plus, for each
// other tile, the number of smaller keys there.
template <int kTile>
__global__ void __launch_bounds__(1024) rank_scatter_kernel(const uint64_t *__restrict__ kin,
                                                            const uint32_t *__restrict__ vin,
                                                            const uint64_t *__restrict__ sample, int n, int tiles,
                                                            uint64_t *__restrict__ kout, uint32_t *__restrict__ vout,
                                                            int *status)
{
    constexpr int kAtOnce = 8, kPerTile = kTile / kSample;
    extern __shared__ uint64_t sort_shared[];
    for (int e = threadIdx.x; e < tiles * kPerTile; e += blockDim.x) sort_shared[e] = sample[e];
    __syncthreads();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint64_t key = kin[i];
    const int own = i / kTile;
    int pos = i - own * kTile;
    for (int t0 = 0; t0 < tiles; t0 += kAtOnce) {
        int at[kAtOnce];  // first key of the sampled group that holds the place (n: none)
#pragma unroll
        for (int q = 0; q < kAtOnce; ++q) {
            const int t = t0 + q;
            at[q] = n;
            if (t < tiles && t != own) {
                const int c = count_before<kPerTile>(sort_shared + t * kPerTile, key, t < own);
                pos += c * kSample;
                if (c < kPerTile) at[q] = t * kTile + c * kSample;
            }
        }
#pragma unroll
        for (int s = kSample >> 1; s > 0; s >>= 1) {
#pragma unroll
            for (int q = 0; q < kAtOnce; ++q) {  // (fewer than kSample smaller keys in the group)
                const int p = at[q] + s - 1;
                // (key + 1 wraps only where every key of the tile goes before: at[q] == n)
                if (p < n && __ldg(kin + p) < key + (t0 + q < own ? 1ull : 0ull)) {
                    at[q] += s;
                    pos += s;
                }
            }
        }
    }
    if (pos >= 0 && pos < n) {
        kout[pos] = key;
        vout[pos] = vin[i];
    } else {
        atomicOr(status, 4);
    }
}

template <int kTile>
void sort_by_rank(hts_ctx *c)
{
    const int n = (int)c->n, tiles = (n + kTile - 1) / kTile;
    constexpr size_t kShared = 2 * kTile * (sizeof(uint64_t) + sizeof(uint16_t));
    const size_t samples = sizeof(uint64_t) * (size_t)tiles * (kTile / kSample);
    if (kShared > 48 * 1024)
        cudaFuncSetAttribute(tile_sort_kernel<kTile>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kShared);
    uint64_t *ko = tiles > 1 ? c->keys_alt : c->keys;
    uint32_t *vo = tiles > 1 ? c->idx_alt : c->idx;
    uint64_t *sample = tiles > 1 ? reinterpret_cast<uint64_t *>(c->sort_scratch) : nullptr;
    tile_sort_kernel<kTile><<<tiles, kTileThreads<kTile>, kShared, c->stream>>>(c->keys, n, ko, vo, sample);
    c->launches += 1;
    if (tiles == 1) return;
    static_assert(kRankMax / kSample * 8 + kTile / kSample * 8 <= 48 * 1024, "the sample fits shared memory");
    const int block = n <= 65536 ? 256 : 1024;  // (every block reads the whole sample)
    rank_scatter_kernel<kTile><<<(n + block - 1) / block, block, samples, c->stream>>>(
        c->keys_alt, c->idx_alt, sample, n, tiles, c->keys, c->idx, c->status);
    c->launches += 1;
}

}  // namespace

size_t sort_status_words(int64_t n)
{
    const int64_t tiles = (n + kMinTile - 1) / kMinTile;  // the most tiles any size up to n uses
    return (size_t)kPasses * 256 * (size_t)std::max<int64_t>(tiles, 1);
}

void launch_sort_pairs(hts_ctx *c)
{
    const int n = (int)c->n;
    const int tile = tile_keys(n);
    const int tiles = (n + tile - 1) / tile;
    // (the wait test is about the look-back, which up to kWaitTestFrom keys is never asked for)
    if (n <= kRankMax && (c->wait_test == 0 || n <= kWaitTestFrom)) {
        if (n <= kRank512)
            sort_by_rank<512>(c);
        else if (n <= kRank1024)
            sort_by_rank<1024>(c);
        else if (n <= kRank2048)
            sort_by_rank<2048>(c);
        else
            sort_by_rank<4096>(c);
        return;
    }
    // scratch: 2048 ints of digit offsets, 8 tile counters, then the status words
    int *hist = reinterpret_cast<int *>(c->sort_scratch);
    int *ctr = hist + kPasses * 256;
    unsigned long long *stat = reinterpret_cast<unsigned long long *>(c->sort_scratch + (kPasses * 256 + 64) / 2);
    cudaMemsetAsync(c->sort_scratch, 0, sizeof(unsigned long long) * ((kPasses * 256 + 64) / 2 +
                                                                      (size_t)kPasses * 256 * tiles), c->stream);
    // (the histograms do not depend on the pass tiles: at most 4096 keys per
    // block keeps enough blocks in flight)
    const int hblocks = (n + 4095) / 4096;
    if (tile == 1024)
        digit_hist_kernel<1024><<<tiles, kSortThreads, 0, c->stream>>>(c->keys, n, hist);
    else if (tile == 2048)
        digit_hist_kernel<2048><<<tiles, kSortThreads, 0, c->stream>>>(c->keys, n, hist);
    else
        digit_hist_kernel<4096><<<hblocks, kSortThreads, 0, c->stream>>>(c->keys, n, hist);
    digit_offsets_kernel<<<1, 32 * kPasses, 0, c->stream>>>(hist);
    c->launches += 2 + kPasses;
    uint64_t *ka = c->keys, *kb = c->keys_alt;
    uint32_t *va = c->idx, *vb = c->idx_alt;
    const int spin = c->wait_test > 0 ? c->wait_test : kSpinLimit;
    const int hold = c->wait_test > 0 ? 1 : 0;
    for (int p = 0; p < kPasses; ++p) {
        unsigned long long *sp = stat + (size_t)p * 256 * tiles;
        if (tile == 1024)
            onesweep_kernel<1024><<<tiles, kSortThreads, 0, c->stream>>>(ka, va, kb, vb, n, 8 * p, hist + p * 256,
                                                                         sp, ctr + p, c->status, spin, hold);
        else if (tile == 2048)
            onesweep_kernel<2048><<<tiles, kSortThreads, 0, c->stream>>>(ka, va, kb, vb, n, 8 * p, hist + p * 256,
                                                                         sp, ctr + p, c->status, spin, hold);
        else if (tile == 4096)
            onesweep_kernel<4096><<<tiles, kSortThreads, 0, c->stream>>>(ka, va, kb, vb, n, 8 * p, hist + p * 256,
                                                                         sp, ctr + p, c->status, spin, hold);
        else
            onesweep_kernel<8192, 2 * kSortThreads><<<tiles, 2 * kSortThreads, 0, c->stream>>>(
                ka, va, kb, vb, n, 8 * p, hist + p * 256, sp, ctr + p, c->status, spin, hold);
        uint64_t *tk = ka; ka = kb; kb = tk;
        uint32_t *tv = va; va = vb; vb = tv;
    }
    // eight passes: the sorted pairs are back in c->keys / c->idx
}

}  // namespace hts
