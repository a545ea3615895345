// sort.cu -- binning and the (tile, depth) key sort (the "Sort" kernel of
// the paper's App. B timing table; keys as in 3DGS, Sec. 3.2).
//
// Order of work (all on the device; the pair count reaches the host through
// pinned words that step 3 writes, in capacity mode not at all; steps 1 to 3 of a
// scene of at most 4096 Gaussians are one block, k_depth_small):
//   1. compact the Gaussians that survived projection into (depth bits, id)
//      pairs, in id order, counting the radix digits as it goes;
//   2. stable LSD radix sort of those pairs by depth (4 passes of 8 bits):
//      ties keep id order, so the order is (depth, id);
//   3. scan their tile counts, in that order, into pair offsets;
//   4. bin: every Gaussian writes (tile, id) for each tile of its range, so
//      the pair list is in (depth, id) order;
//   5. stable LSD radix sort of the pairs by tile id only (2 passes for up
//      to 65536 tiles), which yields (tile, depth, id) order;
//   6. per-tile [start, end) ranges.
// Sorting the N Gaussians by depth once and the K pairs by tile alone moves
// 2 passes over K instead of the 6 a 64-bit (tile, depth) key needs.
#include "internal.h"

namespace sg {

// ------------------------------------------------------------------ scan
__device__ __forceinline__ uint32_t warp_incl_scan(uint32_t v)
{
    int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t t = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += t;
    }
    return v;
}

// ------------------------------------------------------------------ radix sort
// Stable LSD radix sort of (key, value) pairs, digits of at most 8 bits, one
// kernel per digit pass with decoupled look-back (the "onesweep" scheme):
//   1. the kernel that writes the keys counts the digits of every pass
//      (k_compact_depth, k_bin) into scratch zeroed before;
//   2. per pass, the exclusive scan of its digit counts gives the first
//      output position of each digit (every block of the pass scans them);
//   3. k_onesweep, per pass: a block takes the next tile of kRadixTile pairs
//      (an atomic ticket, so tiles are taken in order), ranks them stably
//      (each warp owns kRadixItems x 32 consecutive pairs), publishes its
//      per-digit counts, orders its pairs by digit in shared memory, and walks back over
//      earlier tiles' published counts until it meets an inclusive prefix;
//      then it publishes its own and writes its pairs out.
// A tile only waits for tiles taken before it, whose blocks are running and
// which publish their counts before they wait themselves; every such wait is
// bounded, and a wait that runs out sets *err.
//
// A pass moves 16 bytes a pair, all in L2 at the sizes of a frame: it is
// bound by the latency of its stages and by L2 transactions.  Hence
//   - tiles of 4096 pairs (512 threads, two blocks an SM: three spill), so
//     that 0.7M pairs fill the chip;
//   - equal digits found by an atomicOr of lane bits into the digit's word
//     (8 ballots a pair took the six passes of a 1M view from 89 to 97 us);
//   - a look-back that reads 32 tiles' words a round, four digits a load, in
//     eight groups of threads: the tiles of a launch all publish at about the
//     same time, so a walk of 8 words a round was a chain of tiles / 8 rounds
//     of L2 latency.  More words a round cost more than they save (64: 103
//     us): reading words that are not yet published delays their writers;
//   - pairs written from shared memory in digit order, consecutive threads to
//     consecutive addresses within a digit (a scattered 4-byte write is an L2
//     transaction of its own).
// Measured, the six passes of a frame (four over the visible Gaussians, two
// over the pairs), against tiles of 8192 ranked by ballots, eight words a
// round and scattered writes: 150k Gaussians 85 -> 45 us, 1M (1.5M pairs) 120
// -> 87 us, 2M (3.9M pairs) 242 -> 149 us.
#ifndef SG_RADIX_THREADS
#define SG_RADIX_THREADS 512
#endif
constexpr int kRadixThreads = SG_RADIX_THREADS;
constexpr int kRadixItems = kRadixTile / kRadixThreads;
constexpr int kRadixWarps = kRadixThreads / 32;
constexpr int kLbGroups = kRadixThreads / 64;        // threads per four digits in the look-back
#ifndef SG_LB_BATCH
#define SG_LB_BATCH 4
#endif
constexpr int kLbBatch = SG_LB_BATCH;                // earlier tiles a thread reads a round
static_assert(kRadixThreads % 256 == 0 && kRadixItems * kRadixThreads == kRadixTile &&
                  kRadixTile <= 65535 && kRadixWarps * 256 <= kRadixTile, "radix tile layout");
static_assert(kLbGroups * 256 * sizeof(uint32_t) <= kRadixWarps * 256 * sizeof(uint16_t),
              "look-back sums in the counts' place");
constexpr uint32_t kLbAgg = 1u << 30, kLbPre = 2u << 30, kLbCount = (1u << 30) - 1u;
// Polling rounds a look-back wait makes before it gives up (about a second
// on an idle GPU).  Test hook: the tile whose look-back words the kernels
// of one site never publish (-1: none), so that the next tile's wait runs
// out.  Both live in device memory, where sg_debug_lookback sets them, so
// that replays of captured launch sequences see them too.
constexpr uint32_t kLbSpinsDefault = 1u << 20;
__device__ uint32_t g_lb_spins = kLbSpinsDefault;
__device__ int g_hold_site = SG_LOOKBACK_NONE;
__device__ long long g_hold_tile = -1;
// The tile this launch (of `site`) withholds, or -1.
__device__ __forceinline__ int64_t held_tile(int site)
{
    return *(volatile int *)&g_hold_site == site ? (int64_t) * (volatile long long *)&g_hold_tile
                                                 : (int64_t)-1;
}

// Exclusive scans of two values per thread over the block's first 256
// threads (the others pass anything); every thread of the block calls it.
__device__ __forceinline__ uint2 excl_scan2_256(uint32_t a, uint32_t b, uint2 *s_w)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t ia = warp_incl_scan(a), ib = warp_incl_scan(b);
    if (lane == 31 && warp < 8) s_w[warp] = make_uint2(ia, ib);
    __syncthreads();
    uint2 r = make_uint2(ia - a, ib - b);
#pragma unroll
    for (int w = 0; w < 8; ++w) {
        const uint2 t = s_w[w];
        if (w < warp) { r.x += t.x; r.y += t.y; }
    }
    return r;
}

// Four digits' look-back words of a tile (16-byte aligned), past the L1.
__device__ __forceinline__ uint4 load_words(const uint32_t *p)
{
    uint4 w;
    asm volatile("ld.volatile.global.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(w.x), "=r"(w.y), "=r"(w.z), "=r"(w.w)
                 : "l"(p)
                 : "memory");
    return w;
}

__device__ __forceinline__ bool published(const uint4 &w)
{
    constexpr uint32_t f = kLbAgg | kLbPre;
    return (w.x & f) && (w.y & f) && (w.z & f) && (w.w & f);
}

__global__ void __launch_bounds__(kRadixThreads, 2)
k_onesweep(const uint32_t *keys_in, const uint32_t *vals_in,
           uint32_t *__restrict__ keys_out, uint32_t *__restrict__ vals_out,
           const uint32_t *d_n, int shift, uint32_t mask,
           const uint32_t *hist, uint32_t *lookback,
           uint32_t *ticket, uint32_t *err, int site)
{
    after_previous();
    // the warps' digit counts, then the look-back groups' sums
    __shared__ __align__(16) union {
        uint16_t cnt[kRadixWarps][256];
        uint32_t far[kLbGroups][256];
    } S;
    __shared__ __align__(16) uint32_t s_key[kRadixTile], s_val[kRadixTile];
    __shared__ uint32_t s_start[256], s_pre[256];
    __shared__ uint2 s_w[8];
    __shared__ uint32_t s_tile;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    if (t == 0) s_tile = atomicAdd(ticket, 1u);
    const int64_t n = *d_n;
    const uint32_t h = t < 256 ? hist[t] : 0u;
    const int64_t held = held_tile(site);
    const uint32_t max_spins = g_lb_spins;
    for (int i = t; i < kRadixWarps * 128; i += kRadixThreads) ((uint32_t *)&S.cnt[0][0])[i] = 0u;
    for (int i = t; i < kRadixWarps * 64; i += kRadixThreads)
        reinterpret_cast<uint4 *>(s_key)[i] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
    const uint32_t tile = s_tile;
    const int64_t base = (int64_t)tile * kRadixTile;
    if (base >= n) return;     // so is every later tile: nobody waits for this one
    const int cnt = n - base < kRadixTile ? (int)(n - base) : kRadixTile;
    const int w0 = warp * 32 * kRadixItems + lane;      // the thread's first pair in the tile
    uint32_t k[kRadixItems], v[kRadixItems];
#pragma unroll
    for (int r = 0; r < kRadixItems; ++r) k[r] = w0 + 32 * r < cnt ? keys_in[base + w0 + 32 * r] : 0u;
#pragma unroll
    for (int r = 0; r < kRadixItems; ++r) v[r] = w0 + 32 * r < cnt ? vals_in[base + w0 + 32 * r] : 0u;
    // ranks among the warp's earlier pairs of the same digit (the words of
    // lane bits lie where the ordered keys will)
    uint16_t rk[kRadixItems];
#pragma unroll
    for (int r = 0; r < kRadixItems; ++r) {
        const bool in = w0 + 32 * r < cnt;
        const uint32_t d = (k[r] >> shift) & mask;
        uint32_t *m = s_key + warp * 256;
        if (in) atomicOr(&m[d], 1u << lane);
        __syncwarp();
        const uint32_t peers = in ? m[d] : 0u;
        const uint32_t before = in ? S.cnt[warp][d] : 0u;
        rk[r] = (uint16_t)(before + __popc(peers & ((1u << lane) - 1u)));
        __syncwarp();
        if (in && lane == __ffs(peers) - 1) {
            S.cnt[warp][d] = (uint16_t)(before + __popc(peers));
            m[d] = 0u;
        }
        __syncwarp();
    }
    __syncthreads();
    // one digit per thread: the warps' offsets within the digit and the
    // tile's count, published at once
    const bool publish = (int64_t)tile != held;
    uint32_t run = 0u;
    if (t < 256) {
        uint32_t c[kRadixWarps];
#pragma unroll
        for (int w = 0; w < kRadixWarps; ++w) c[w] = S.cnt[w][t];
#pragma unroll
        for (int w = 0; w < kRadixWarps; ++w) {
            S.cnt[w][t] = (uint16_t)run;
            run += c[w];
        }
        if (publish)
            ((volatile uint32_t *)lookback)[(int64_t)tile * 256 + t] =
                (tile == 0 ? kLbPre : kLbAgg) | run;
    }
    // first position of the digit in the tile and in the pass's output
    const uint2 first = excl_scan2_256(run, h, s_w);
    if (t < 256) s_start[t] = first.x;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kRadixItems; ++r) {
        if (w0 + 32 * r < cnt) {
            const uint32_t d = (k[r] >> shift) & mask;
            const uint32_t q = s_start[d] + S.cnt[warp][d] + rk[r];
            s_key[q] = k[r];
            s_val[q] = v[r];
        }
    }
    __syncthreads();
    // look-back: thread (group g, digits 4 q .. 4 q + 3) sums the words of the
    // kLbBatch tiles before hi - g kLbBatch, up to the first inclusive prefix
    uint32_t excl = 0u;
    bool done = tile == 0;
    const int q = t & 63, g = t >> 6;
    const bool used = 4u * q <= mask;
    for (int64_t hi = tile; hi > 0; hi -= kLbGroups * kLbBatch) {
        const int64_t h0 = hi - 1 - g * kLbBatch;
        const uint32_t *words = lookback + h0 * 256 + 4 * q;
        if (used) {
            uint4 w[kLbBatch], sum = make_uint4(0u, 0u, 0u, 0u);
            uint32_t spins = 0, found = 0u;
#pragma unroll
            for (int i = 0; i < kLbBatch; ++i)      // before tile 0: an empty inclusive prefix
                w[i] = h0 - i >= 0 ? load_words(words - 256 * i)
                                   : make_uint4(kLbPre, kLbPre, kLbPre, kLbPre);
#pragma unroll
            for (int i = 0; i < kLbBatch; ++i) {
                if (found == 15u) continue;
                while (!published(w[i])) {       // only these words are read again
                    if (++spins > max_spins) {   // gave up: flag it, leave the order wrong
                        atomicOr(err, kStatusLookback);
                        w[i] = make_uint4(kLbPre, kLbPre, kLbPre, kLbPre);
                        break;
                    }
                    w[i] = load_words(words - 256 * i);
                }
                if (!(found & 1u)) sum.x += w[i].x & kLbCount;
                if (!(found & 2u)) sum.y += w[i].y & kLbCount;
                if (!(found & 4u)) sum.z += w[i].z & kLbCount;
                if (!(found & 8u)) sum.w += w[i].w & kLbCount;
                found |= (w[i].x >> 31) | (w[i].y >> 31) << 1 | (w[i].z >> 31) << 2 |
                         (w[i].w >> 31) << 3;
            }
            sum.x |= (found & 1u) << 31;
            sum.y |= (found & 2u) << 30;
            sum.z |= (found & 4u) << 29;
            sum.w |= (found & 8u) << 28;
            *reinterpret_cast<uint4 *>(&S.far[g][4 * q]) = sum;
        }
        __syncthreads();
        const bool walk = t < 256 && !done;
        if (walk) {
#pragma unroll
            for (int i = 0; i < kLbGroups; ++i) {
                const uint32_t x = t <= (int)mask ? S.far[i][t] : kLbPre;
                if (!done) excl += x & kLbCount;
                done = done || (x & kLbPre) != 0u;
            }
            if (done && publish)
                ((volatile uint32_t *)lookback)[(int64_t)tile * 256 + t] = kLbPre | (excl + run);
        }
        if (!__syncthreads_or(t < 256 && !done)) break;
    }
    if (t < 256) s_pre[t] = first.y + excl - first.x;
    __syncthreads();
    // the digit's pairs of this tile follow one another in the output; after a
    // wait gave up the counts may not match the pairs: nothing past the end
    for (int i = t; i < cnt; i += kRadixThreads) {
        const uint32_t key = s_key[i];
        const uint32_t pos = s_pre[(key >> shift) & mask] + i;
        if (pos < n) {
            if (keys_out) keys_out[pos] = key;
            vals_out[pos] = s_val[i];
        }
    }
}

sg_status tile_scratch(int64_t n_max, int passes, Frame &fr, cudaStream_t st, uint32_t **hist)
{
    const void *had = fr.tscratch.p;
    const size_t bytes = sizeof(uint32_t) * (size_t)radix_scratch_words(n_max, passes);
    sg_status s = ensure(fr.tscratch, bytes);
    if (s != SG_OK) return s;
    if (fr.tscratch.p != had || bytes > fr.tscratch_zeroed)
        SG_CUDA(cudaMemsetAsync(fr.tscratch.p, 0, bytes, st));
    fr.tscratch_zeroed = 0;      // in use from here on
    *hist = (uint32_t *)fr.tscratch.p;
    return SG_OK;
}

sg_status radix_sort_pairs(uint32_t *keys[2], uint32_t *vals[2], int64_t n_max,
                           const uint32_t *d_n, int begin_bit, int end_bit, uint32_t *scratch,
                           uint32_t *d_err, cudaStream_t st, int *result_buf, int site,
                           bool keep_keys)
{
    *result_buf = 0;
    if (n_max <= 0 || end_bit <= begin_bit) return SG_OK;
    if (n_max > (int64_t)kLbCount) {
        set_error("radix sort of %lld pairs exceeds 2^30", (long long)n_max);
        return SG_ERR_OVERFLOW;
    }
    const int passes = (end_bit - begin_bit + 7) / 8;
    const int64_t tiles = (n_max + kRadixTile - 1) / kRadixTile;
    uint32_t *hist = scratch;
    uint32_t *tickets = hist + 2 * 256 * passes;            // [passes], padded to 16
    uint32_t *lookback = tickets + 16;
    int cur = 0;
    for (int p = 0; p < passes; ++p) {
        const int b = radix_bit(begin_bit, end_bit, p);
        const int bits = radix_bit(begin_bit, end_bit, p + 1) - b;
        uint32_t *keys_out = p == passes - 1 && !keep_keys ? nullptr : keys[cur ^ 1];
        launch_after(k_onesweep, (unsigned)tiles, kRadixThreads, 0, st,
            keys[cur], vals[cur], keys_out, vals[cur ^ 1], d_n, b, (1u << bits) - 1u,
            hist + 256 * p, lookback + (int64_t)p * tiles * 256, tickets + p, d_err, site);
        SG_LAUNCHED();
        cur ^= 1;
    }
    *result_buf = cur;
    return SG_OK;
}

// ------------------------------------------------------------------ depth stage
// The depth stage as two chained scans around the radix passes.  A block
// takes the next tile of kChainTile entries (an atomic ticket, so tiles are
// taken in order), publishes its total, and walks back over earlier tiles'
// published totals until an inclusive prefix (64-bit words: two flag bits,
// a 62-bit count), as the radix passes do:
//   k_compact_depth: the Gaussians with a non-zero tile count, in id order,
//     as (depth bits, id) pairs, the number of them, and the digit
//     histograms of the four radix passes over their keys;
//   k_pair_offsets: in depth order, the exclusive scan of the tile counts
//     count[ids[i]] (gathered as it goes) into pair offsets, and the total.
// Both are bound by latency (a few MB, in L2).  The compaction publishes its
// tile's total before it counts digits, with plain shared-memory atomics
// (ballots over 64 digits a thread held the publication back): 26 -> 11 us at
// 1M Gaussians, 41 -> 17 us at 2M, tiles of 2048 so that 1M give every SM
// three blocks.  The offsets gather a 4-byte count per Gaussian (one L1 request
// each, about 5 us at 1.5M) and take tiles of 8192 above 256k Gaussians, whose
// shorter look-back chain is worth more than the fuller chip (at 1M 12 us; 4096
// 16, 2048 19), and of 2048 below, where the chain is short (150k: the stage 52
// us, 56 with 8192); counting the tiles done, in exact mode, adds 1 to 1.5 us.
// One warp walks back, 32 words a round: 128 words a round or all warps reading
// took 11 -> 12 and 14 -> 17 us.
constexpr int kChainThreads = 256;
constexpr int kChainWarps = kChainThreads / 32;
constexpr int kChainChunks = kChainTile / kChainThreads;   // 32-entry chunks per warp
// Chunks of a tile of k_pair_offsets, and the scene size up to which its tiles
// are small.
constexpr int kOffSmall = 8, kOffLarge = 32;
constexpr int64_t kOffSmallN = 262144;
static_assert(kOffSmall >= kChainChunks, "look-back words sized by kChainTile");
constexpr unsigned long long kChAgg = 1ull << 62, kChPre = 2ull << 62,
                             kChCount = (1ull << 62) - 1ull;

constexpr int kChainBatch = 1;     // earlier tiles' words a lane of the walking warp loads a round

struct ChainShared {
    unsigned long long excl;
    uint32_t warp[kChainWarps];
    uint32_t tile;
};

// Publish the tile's total (thread 0).
__device__ __forceinline__ void chain_publish(unsigned long long *lb, int64_t tile,
                                              unsigned long long total, bool publish)
{
    if (threadIdx.x == 0 && publish)
        ((volatile unsigned long long *)lb)[tile] = (tile == 0 ? kChPre : kChAgg) | total;
}

// Exclusive prefix of tile `tile` (whose total is published) from the earlier
// tiles' words; every thread of the block calls it and gets it, warp 0 walks
// (more threads reading words not yet published slow their writers down).  A
// wait that runs out sets *err (the prefix is then wrong, never unbounded).
__device__ __forceinline__ unsigned long long chain_lookback(unsigned long long *lb, int64_t tile,
                                                             unsigned long long total,
                                                             bool publish, uint32_t *err,
                                                             ChainShared &S)
{
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x;
        volatile unsigned long long *v = lb;
        const uint32_t max_spins = g_lb_spins;
        unsigned long long excl = 0;
        uint32_t spins = 0;
        bool found = false;
        for (int64_t hi = tile; hi > 0 && !found; hi -= 32 * kChainBatch) {
            unsigned long long w[kChainBatch];
#pragma unroll
            for (int i = 0; i < kChainBatch; ++i) {
                const int64_t tt = hi - 1 - 32 * i - lane;
                // before tile 0: an empty inclusive prefix
                w[i] = tt >= 0 ? v[tt] : (unsigned long long)kChPre;
            }
#pragma unroll
            for (int i = 0; i < kChainBatch; ++i) {
                if (found) continue;
                const int64_t tt = hi - 1 - 32 * i - lane;
                while ((w[i] & (kChAgg | kChPre)) == 0ull) {
                    if (++spins > max_spins) {   // gave up: flag it
                        atomicOr(err, kStatusLookback);
                        w[i] = kChPre;
                        break;
                    }
                    w[i] = v[tt];
                }
                const uint32_t pre = __ballot_sync(0xffffffffu, (w[i] & kChPre) != 0ull);
                const int last = pre ? __ffs(pre) - 1 : 31;     // lanes [0, last] are summed
                unsigned long long c = lane <= last ? (w[i] & kChCount) : 0ull;
#pragma unroll
                for (int o = 16; o; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
                excl += c;
                found = pre != 0u;
            }
        }
        if (lane == 0) {
            if (tile > 0 && publish) v[tile] = kChPre | (excl + total);
            S.excl = excl;
        }
    }
    __syncthreads();
    return S.excl;
}

__global__ void __launch_bounds__(kChainThreads)
k_compact_depth(const uint32_t *count, const float *depth, int64_t n,
                int64_t ntiles, uint32_t *__restrict__ keys, uint32_t *__restrict__ vals,
                uint32_t *__restrict__ d_nvalid, uint32_t *hist,
                unsigned long long *lb, uint32_t *ticket,
                uint32_t *err, uint4 *__restrict__ zero, int64_t nzero)
{
    after_previous();
    __shared__ uint32_t s_h[4][256];
    __shared__ ChainShared S;
    // the tile sort's scratch, zeroed here rather than by a launch of its own
    for (int64_t i = (int64_t)blockIdx.x * kChainThreads + threadIdx.x; i < nzero;
         i += (int64_t)gridDim.x * kChainThreads)
        zero[i] = make_uint4(0u, 0u, 0u, 0u);
    for (int i = threadIdx.x; i < 4 * 256; i += kChainThreads) (&s_h[0][0])[i] = 0;
    if (threadIdx.x == 0) S.tile = atomicAdd(ticket, 1u);
    __syncthreads();
    const int64_t tile = S.tile;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // warp w owns kChainChunks x 32 consecutive entries of the tile
    const int64_t wbase = tile * kChainTile + (int64_t)warp * 32 * kChainChunks;
    uint32_t bal[kChainChunks], key[kChainChunks], cnt[kChainChunks];
#pragma unroll
    for (int r = 0; r < kChainChunks; ++r) {
        const int64_t i = wbase + r * 32 + lane;
        cnt[r] = i < n ? count[i] : 0u;
        key[r] = i < n ? __float_as_uint(depth[i]) : 0u;   // depth > 0: bits are monotone
    }
    uint32_t wtot = 0;
#pragma unroll
    for (int r = 0; r < kChainChunks; ++r) {
        bal[r] = __ballot_sync(0xffffffffu, cnt[r] > 0u);
        wtot += __popc(bal[r]);
    }
    if (lane == 0) S.warp[warp] = wtot;
    __syncthreads();
    uint32_t before = 0, total = 0;
#pragma unroll
    for (int w = 0; w < kChainWarps; ++w) {
        const uint32_t c = S.warp[w];
        before += w < warp ? c : 0u;
        total += c;
    }
    const bool publish = tile != held_tile(SG_LOOKBACK_COMPACT);
    chain_publish(lb, tile, total, publish);
    // the digit counts, while earlier tiles publish
#pragma unroll
    for (int r = 0; r < kChainChunks; ++r)
        if (cnt[r] > 0u)
#pragma unroll
            for (int p = 0; p < 4; ++p) atomicAdd(&s_h[p][(key[r] >> (8 * p)) & 255u], 1u);
    const uint32_t excl = (uint32_t)chain_lookback(lb, tile, total, publish, err, S);
    if (threadIdx.x == 0 && tile == ntiles - 1) *d_nvalid = excl + total;
    uint32_t pos = excl + before;
#pragma unroll
    for (int r = 0; r < kChainChunks; ++r) {
        if ((bal[r] >> lane) & 1u) {
            const uint32_t q = pos + __popc(bal[r] & ((1u << lane) - 1u));
            keys[q] = key[r];
            vals[q] = (uint32_t)(wbase + r * 32 + lane);
        }
        pos += __popc(bal[r]);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 4 * 256; i += kChainThreads) {
        const uint32_t c = (&s_h[0][0])[i];
        if (c) atomicAdd(&hist[i], c);
    }
}

// The counts and the status word to the frame's pinned words (host; NULL:
// nobody waits for them), the sequence number last.
__device__ __forceinline__ void tell_host(volatile uint32_t *host, uint32_t nvalid, uint32_t pairs,
                                          uint32_t status, uint32_t seq)
{
    if (!host) return;
    host[0] = nvalid;
    host[1] = pairs;
    host[kScalStatus] = status;
    __threadfence_system();
    host[kHostCountSeq] = seq;
}

// Entry i's pairs [off, off + n): its offset, and the binning blocks whose first
// pair is one of them.  Offsets of 2^32 and more, which only a render that drops
// pairs can reach (its capacity is below 2^31), are stored as 2^32 - 1: wrapped
// ones would decrease, and binning takes them to be sorted.
__device__ __forceinline__ void put_offset(int64_t i, unsigned long long off, uint32_t n,
                                           uint32_t *__restrict__ offsets,
                                           uint32_t *__restrict__ owner, int64_t owner_cap)
{
    offsets[i] = off < 0xffffffffull ? (uint32_t)off : 0xffffffffu;
    for (unsigned long long b = (off + kBinChunk - 1) / kBinChunk;
         b * kBinChunk < off + n && (int64_t)b < owner_cap; ++b)
        owner[b] = (uint32_t)i;
}

template <int kOffChunks>
__global__ void __launch_bounds__(kChainThreads)
k_pair_offsets(const uint32_t *ids, const uint32_t *count, int64_t n,
               const uint32_t *d_nvalid, uint32_t *__restrict__ offsets,
               uint32_t *d_total, unsigned long long *lb,
               uint32_t *ticket, uint32_t *done, uint32_t *err,
               uint32_t *__restrict__ owner, int64_t owner_cap, volatile uint32_t *host, uint32_t seq)
{
    after_previous();
    constexpr int kOffTile = kOffChunks * kChainThreads;
    __shared__ ChainShared S;
    if (threadIdx.x == 0) S.tile = atomicAdd(ticket, 1u);
    const int64_t nv = *d_nvalid;
    __syncthreads();
    const int64_t tile = S.tile;
    const int64_t ntiles = (nv + kOffTile - 1) / kOffTile;
    if (nv == 0) {
        if (tile == 0 && threadIdx.x == 0) {
            *d_total = 0u;
            tell_host(host, 0u, 0u, *(volatile uint32_t *)err, seq);
        }
        return;
    }
    if (tile >= ntiles) return;   // so is every later tile: nobody waits for this one
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t wbase = tile * kOffTile + (int64_t)warp * 32 * kOffChunks;
    uint32_t c[kOffChunks];
#pragma unroll
    for (int r = 0; r < kOffChunks; ++r) {
        const int64_t i = wbase + r * 32 + lane;
        c[r] = i < nv ? ids[i] : 0xffffffffu;
    }
    // an id is outside 0..n-1 only after a look-back wait of the depth sort
    // gave up (err set, the sort's output partly unwritten): count it as 0
#pragma unroll
    for (int r = 0; r < kOffChunks; ++r) c[r] = (int64_t)c[r] < n ? count[c[r]] : 0u;
    uint32_t run = 0;   // the warp's entries before chunk r
#pragma unroll
    for (int r = 0; r < kOffChunks; ++r) {
        const uint32_t inc = warp_incl_scan(c[r]);
        const uint32_t v = c[r];
        c[r] = run + inc - v;
        run += __shfl_sync(0xffffffffu, inc, 31);
    }
    if (lane == 0) S.warp[warp] = run;
    __syncthreads();
    unsigned long long before = 0, total = 0;
#pragma unroll
    for (int w = 0; w < kChainWarps; ++w) {
        const uint32_t x = S.warp[w];
        before += w < warp ? x : 0u;
        total += x;
    }
    const bool publish = tile != held_tile(SG_LOOKBACK_OFFSETS);
    chain_publish(lb, tile, total, publish);
    const unsigned long long excl = chain_lookback(lb, tile, total, publish, err, S);
    if (threadIdx.x == 0) {
        if (tile == ntiles - 1) {
            // saturated, so that a total of 2^32 pairs or more reads as an overflow
            const unsigned long long tot = excl + total;
            *d_total = tot > 0xffffffffull ? 0xffffffffu : (uint32_t)tot;
        }
        // The tile whose wait ends last tells the host: a wait that gave up set
        // the status word before its tile counted itself here, so the host learns
        // of every one with the count.  (The last tile telling it at once was 1 to
        // 1.4 us sooner and could miss a status: 251x243 181.8 us a call, now 182.8.)
        if (host) {
            __threadfence();
            if (atomicAdd(done, 1u) == (uint32_t)ntiles - 1u) {
                __threadfence();
                tell_host(host, (uint32_t)nv, *(volatile uint32_t *)d_total,
                          *(volatile uint32_t *)err, seq);
            }
        }
    }
    const unsigned long long pre = excl + before;
#pragma unroll
    for (int r = 0; r < kOffChunks; ++r) {
        const int64_t i = wbase + r * 32 + lane;
        // the next entry's offset: the entry's pairs are [off, next)
        uint32_t next = __shfl_down_sync(0xffffffffu, c[r], 1);
        const uint32_t chunk_end =
            r + 1 < kOffChunks ? __shfl_sync(0xffffffffu, c[r + 1 < kOffChunks ? r + 1 : r], 0) : run;
        if (lane == 31) next = chunk_end;
        if (i < nv) put_offset(i, pre + c[r], next - c[r], offsets, owner, owner_cap);
    }
}

// The whole depth stage of a scene of at most kSmallN Gaussians, in one block:
// compaction in id order, four stable 8-bit passes over the depth bits in shared
// memory, and the offsets, as the kernels above make them.  Bound by the latency
// of its steps (a pass: digits of a warp's 128 keys matched 32 at a time, counts
// of 32 warps scanned, one scatter).  One launch for six: 27 -> 16 us with their
// gaps at 4096 Gaussians (64x64 view 82 -> 71 us).  A thread holds four entries,
// which fills a block at 4096; the look-back passes spread what is more over the
// SMs.
constexpr int kSmallThreads = 1024, kSmallPer = 4, kSmallN = kSmallThreads * kSmallPer;
constexpr size_t kSmallZero = 64 * 1024;

__global__ void __launch_bounds__(kSmallThreads)
k_depth_small(const uint32_t *count, const float *depth, int n,
              uint32_t *__restrict__ vals, uint32_t *__restrict__ d_nvalid,
              uint32_t *__restrict__ offsets, uint32_t *__restrict__ d_total,
              const uint32_t *err, uint32_t *__restrict__ owner, int64_t owner_cap,
              volatile uint32_t *host, uint32_t seq, uint4 *__restrict__ zero, int64_t nzero)
{
    after_previous();
    constexpr uint32_t full = 0xffffffffu;
    __shared__ uint32_t s_key[kSmallN];
    __shared__ uint16_t s_val[kSmallN];
    // a warp's keys of a digit; rows 2 longer: the four threads of a digit read rows 8
    // apart, from banks of their own
    __shared__ __align__(4) uint16_t s_cnt[32][258];
    __shared__ uint32_t s_base[256], s_w[32];
    for (int64_t i = threadIdx.x; i < nzero; i += kSmallThreads) zero[i] = make_uint4(0u, 0u, 0u, 0u);
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5, first = warp * 32 * kSmallPer + lane;
    const uint32_t below = (1u << lane) - 1u;
    {
        uint32_t bal[kSmallPer], key[kSmallPer], wtot = 0u;
#pragma unroll
        for (int r = 0; r < kSmallPer; ++r) {
            const int i = first + 32 * r;
            bal[r] = __ballot_sync(full, i < n && count[i] > 0u);
            key[r] = i < n ? __float_as_uint(depth[i]) : 0u;
            wtot += __popc(bal[r]);
        }
        if (lane == 0) s_w[warp] = wtot;
        __syncthreads();
        uint32_t pos = __reduce_add_sync(full, lane < warp ? s_w[lane] : 0u);
#pragma unroll
        for (int r = 0; r < kSmallPer; ++r) {
            if ((bal[r] >> lane) & 1u) {
                const uint32_t q = pos + __popc(bal[r] & below);
                s_key[q] = key[r];
                s_val[q] = (uint16_t)(first + 32 * r);
            }
            pos += __popc(bal[r]);
        }
    }
    const int nv = (int)__reduce_add_sync(full, s_w[lane]);
    __syncthreads();
    for (int p = 0; p < 4; ++p) {
        uint32_t key[kSmallPer], val[kSmallPer], rank[kSmallPer];
        for (int i = lane; i < 128; i += 32) reinterpret_cast<uint32_t *>(s_cnt[warp])[i] = 0u;
        __syncwarp();
#pragma unroll
        for (int r = 0; r < kSmallPer; ++r) {
            const int i = first + 32 * r;
            const bool live = i < nv;
            key[r] = live ? s_key[i] : 0u;
            val[r] = live ? s_val[i] : 0u;
            const uint32_t d = (key[r] >> (8 * p)) & 255u;
            const uint32_t peers = __match_any_sync(full, live ? d : 256u);
            const uint32_t had = s_cnt[warp][d];
            __syncwarp();
            if (live && lane == __ffs(peers) - 1) s_cnt[warp][d] = (uint16_t)(had + __popc(peers));
            __syncwarp();
            rank[r] = had + __popc(peers & below);
        }
        __syncthreads();
        // per digit, the keys of earlier warps: four threads a digit, eight warps each
        const int digit = t >> 2, part = t & 3;
        uint32_t sum = 0u;
#pragma unroll
        for (int q = 0; q < 8; ++q) sum += s_cnt[8 * part + q][digit];
        uint32_t inc = sum;
#pragma unroll
        for (int o = 1; o < 4; o <<= 1) {
            const uint32_t x = __shfl_up_sync(full, inc, o, 4);
            if (part >= o) inc += x;
        }
        uint32_t run = inc - sum;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const uint32_t c = s_cnt[8 * part + q][digit];
            s_cnt[8 * part + q][digit] = (uint16_t)run;
            run += c;
        }
        // the digits' first positions: the last of the four threads has the total
        const uint32_t tot = part == 3 ? inc : 0u;
        const uint32_t di = warp_incl_scan(tot);
        if (lane == 31) s_w[warp] = di;
        __syncthreads();
        const uint32_t pre = __reduce_add_sync(full, lane < warp ? s_w[lane] : 0u);
        if (part == 3) s_base[digit] = pre + di - tot;
        __syncthreads();
#pragma unroll
        for (int r = 0; r < kSmallPer; ++r) {
            if (first + 32 * r >= nv) continue;
            const uint32_t d = (key[r] >> (8 * p)) & 255u;
            const uint32_t q = s_base[d] + s_cnt[warp][d] + rank[r];
            s_key[q] = key[r];
            s_val[q] = (uint16_t)val[r];
        }
        __syncthreads();
    }
    // the offsets, as k_pair_offsets
    uint32_t c[kSmallPer], run = 0u;
#pragma unroll
    for (int r = 0; r < kSmallPer; ++r) {
        const int i = first + 32 * r;
        const uint32_t id = i < nv ? s_val[i] : 0u;
        const uint32_t v = i < nv ? count[id] : 0u;
        if (i < nv) vals[i] = id;
        const uint32_t inc = warp_incl_scan(v);
        c[r] = run + inc - v;
        run += __shfl_sync(full, inc, 31);
    }
    if (lane == 0) s_w[warp] = run;
    __syncthreads();
    unsigned long long total = 0, pre = 0;
    for (int w = 0; w < 32; ++w) {
        pre += w < warp ? s_w[w] : 0u;
        total += s_w[w];
    }
#pragma unroll
    for (int r = 0; r < kSmallPer; ++r) {
        const int i = first + 32 * r;
        uint32_t next = __shfl_down_sync(full, c[r], 1);
        const uint32_t chunk_end =
            r + 1 < kSmallPer ? __shfl_sync(full, c[r + 1 < kSmallPer ? r + 1 : r], 0) : run;
        if (lane == 31) next = chunk_end;
        if (i < nv) put_offset(i, pre + c[r], next - c[r], offsets, owner, owner_cap);
    }
    if (t == 0) {
        const uint32_t sat = total > 0xffffffffull ? 0xffffffffu : (uint32_t)total;
        *d_nvalid = (uint32_t)nv;
        *d_total = sat;
        tell_host(host, (uint32_t)nv, sat, *(const volatile uint32_t *)err, seq);
    }
}

sg_status depth_stage(const uint32_t *d_count, const float *d_depth, int64_t n, uint32_t *keys[2],
                      uint32_t *vals[2], uint32_t *d_scal, uint32_t *d_offsets, Frame &fr,
                      cudaStream_t st, int *result_buf, uint32_t host_seq)
{
    *result_buf = 0;
    fr.tscratch_zeroed = 0;
    if (n <= 0) {   // no projection kernel ran: clear the status word too
        SG_CUDA(cudaMemsetAsync(d_scal, 0, 4 * (kScalStatus + 1), st));
        return SG_OK;
    }
    if (n > (int64_t)kLbCount) {
        set_error("depth sort of %lld Gaussians exceeds 2^30", (long long)n);
        return SG_ERR_OVERFLOW;
    }
    // after the radix scratch, zeroed with it: two tickets and the number of
    // offset tiles done (four words), then one 64-bit word per tile for each of
    // the two chained scans
    const int64_t ntiles = (n + kChainTile - 1) / kChainTile;
    if (fr.hist.bytes < sizeof(uint32_t) * (size_t)depth_stage_words(n)) {
        set_error("internal: depth stage scratch missing");
        return SG_ERR_INVALID;
    }
    uint32_t *hist = (uint32_t *)fr.hist.p;
    sg_status s;
    static_assert(radix_scratch_words(1, 4) % 2 == 0, "64-bit chain words stay aligned");
    unsigned long long *chain = (unsigned long long *)(hist + radix_scratch_words(n, 4));
    uint32_t *tickets = (uint32_t *)chain;      // [0] compaction, [1] offsets, [2] offsets done
    uint32_t *err = (uint32_t *)fr.scalars.p + kScalStatus;
    if (n <= kSmallN) {
        // one block zeroes what a scene of this size needs of the tile sort's
        // scratch, not all that a larger render has left
        const size_t zero = fr.tscratch.bytes < kSmallZero ? fr.tscratch.bytes : kSmallZero;
        launch_after(k_depth_small, 1, kSmallThreads, 0, st, d_count, d_depth, (int)n, vals[0], d_scal,
                     d_offsets, d_scal + 1, err, (uint32_t *)fr.owner.p, (int64_t)(fr.owner.bytes / 4),
                     host_seq ? (volatile uint32_t *)fr.h_scalars : nullptr, host_seq,
                     (uint4 *)fr.tscratch.p, (int64_t)(zero / 16));
        SG_LAUNCHED();
        fr.tscratch_zeroed = zero / 16 * 16;
        return SG_OK;
    }
    launch_after(k_compact_depth, (unsigned)ntiles, kChainThreads, 0, st,
        d_count, d_depth, n, ntiles, keys[0], vals[0], d_scal, hist, chain + 2, tickets, err,
        (uint4 *)fr.tscratch.p, (int64_t)(fr.tscratch.bytes / 16));
    SG_LAUNCHED();
    fr.tscratch_zeroed = fr.tscratch.bytes / 16 * 16;
    // (only the ids of the sorted order are read again)
    if ((s = radix_sort_pairs(keys, vals, n, d_scal, 0, 32, hist, err, st, result_buf,
                              SG_LOOKBACK_DEPTH_SORT, false)) != SG_OK)
        return s;
    const bool small = n <= kOffSmallN;
    const int64_t off_tile = (int64_t)kChainThreads * (small ? kOffSmall : kOffLarge);
    auto k_off = small ? k_pair_offsets<kOffSmall> : k_pair_offsets<kOffLarge>;
    launch_after(k_off, (unsigned)((n + off_tile - 1) / off_tile), kChainThreads, 0, st,
        vals[*result_buf], d_count, n, d_scal, d_offsets, d_scal + 1, chain + 2 + ntiles,
        tickets + 1, tickets + 2, err, (uint32_t *)fr.owner.p, (int64_t)(fr.owner.bytes / 4),
        host_seq ? (volatile uint32_t *)fr.h_scalars : nullptr, host_seq);
    SG_LAUNCHED();
    return SG_OK;
}

// ------------------------------------------------------------------ binning

// Expand each valid Gaussian (depth order) into its (tile, Gaussian) pairs:
// pair o of Gaussian g goes to position offsets[g] + o, tile rows outer and
// columns inner.  Pairs at positions >= cap are not written (capacity mode:
// the caller learns of them from the dropped-pairs count).
// Balanced by pairs: block b writes pairs [b C, (b + 1) C) of the
// depth-ordered expansion (C = kBinChunk; pair p belongs to the valid
// Gaussian k with offsets[k] <= p < offsets[k + 1]).  The owner of its first
// pair is in the table that k_pair_offsets wrote (beyond the table, a
// cooperative search over the offsets, 512 samples per round).  The block
// loads the at most C + 1 Gaussians its pairs can belong to, marks each one's
// first pair, and a running maximum over the pairs gives every pair its
// owner; a thread takes four consecutive pairs and writes them as 16 bytes.
// A Gaussian that covers thousands of tiles is spread over many blocks.
// Bound by instructions and the latency of its loads (8 bytes a pair to L2):
// a search in shared memory, two integer divisions and 16 digit ballots a
// pair took 26 us for 1.5M pairs and 60 us for 3.9M; now 17 and 34 us (blocks
// of 1024 pairs and 256 threads: 19 and 35).
constexpr int kBinThreads = 512;
constexpr int kBinPasses = 3;         // tile ids up to 24 bits when k_bin counts the digits
static_assert(kBinChunk == 4 * kBinThreads, "four pairs a thread");

__device__ __forceinline__ int pmod_i(int a, int n)
{
    const int m = a % n;
    return m < 0 ? m + n : m;
}

__global__ void __launch_bounds__(kBinThreads)
k_bin(const uint32_t *ids, const uint32_t *offsets,
      const uint32_t *d_scal, const int4 *tiles, int ntx, int wrap_x,
      uint32_t cap, uint32_t *__restrict__ keys, uint32_t *__restrict__ vals,
      uint32_t *hist, int end_bit, const uint32_t *err,
      const uint32_t *owner, int64_t owner_cap, uint2 *__restrict__ ranges,
      int64_t ntiles)
{
    after_previous();
    for (int64_t i = (int64_t)blockIdx.x * kBinThreads + threadIdx.x; i < ntiles;
         i += (int64_t)gridDim.x * kBinThreads)
        ranges[i] = make_uint2(0u, 0u);     // every tile's list empty, for the tile ranges
    // per Gaussian of the block: first pair, id, tile columns (first, count),
    // tile rows (first, last); per pair: its owner, where it is the first
    __shared__ uint32_t s_off[kBinChunk + 1], s_id[kBinChunk + 1];
    __shared__ uint2 s_rg[kBinChunk + 1];
    __shared__ __align__(8) uint16_t s_own[kBinChunk];
    __shared__ uint32_t s_max[kBinThreads / 32];
    __shared__ uint32_t s_h[kBinPasses][256];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int passes = (end_bit + 7) / 8;
    for (int i = t; i < kBinPasses * 256; i += kBinThreads) (&s_h[0][0])[i] = 0u;
    for (int i = t; i < kBinChunk / 2; i += kBinThreads) reinterpret_cast<uint32_t *>(s_own)[i] = 0u;
    const int64_t nvalid = d_scal[0];
    const int64_t K = min((int64_t)d_scal[1], (int64_t)cap);
    const int64_t p0 = (int64_t)blockIdx.x * kBinChunk;
    // after a look-back wait of the depth stage gave up, the ids and offsets
    // are not trustworthy (offsets may decrease): write nothing
    if (p0 >= K || nvalid == 0 || *err) return;
    const int64_t p1 = min(K, p0 + kBinChunk);
    // the owner of p0: the largest k with offsets[k] <= p0 (offsets[0] = 0,
    // strictly increasing below 2^32 - 1: every valid Gaussian has a pair)
    int64_t k0 = 0;
    if ((int64_t)blockIdx.x < owner_cap) {
        k0 = owner[blockIdx.x];
    } else {
        int64_t hi = nvalid;
        while (hi - k0 > 1) {
            const int64_t step = (hi - k0 + kBinThreads - 1) / kBinThreads;
            const int64_t idx = k0 + t * step;
            const bool le = idx < hi && (int64_t)offsets[idx] <= p0;
            const int c = __syncthreads_count(le);
            k0 = k0 + (int64_t)(c - 1) * step;
            hi = min(hi, k0 + step);
        }
    }
    const int nk = (int)min((int64_t)kBinChunk + 1, nvalid - k0);
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kBinChunk / kBinThreads + 1; ++r) {
        const int i = r * kBinThreads + t;
        if (i >= nk) continue;
        const uint32_t off = offsets[k0 + i], g = ids[k0 + i];
        if ((int64_t)off >= p1) continue;
        const int4 q = tiles[g];
        s_off[i] = off;
        s_id[i] = g;
        const int x = wrap_x ? pmod_i(q.x, ntx) : q.x;
        s_rg[i] = make_uint2((uint32_t)x | (uint32_t)(q.y - q.x + 1) << 16,
                             (uint32_t)q.z | (uint32_t)q.w << 16);
        if ((int64_t)off >= p0) s_own[off - p0] = (uint16_t)i;
    }
    __syncthreads();
    // the owners, as local indices, of pairs p0 + 4 t ..
    const ushort4 o = *reinterpret_cast<const ushort4 *>(s_own + 4 * t);
    uint32_t m[4] = {o.x, max((uint32_t)o.x, (uint32_t)o.y), o.z, o.w};
    m[2] = max(m[2], m[1]);
    m[3] = max(m[3], m[2]);
    uint32_t inc = m[3];
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t x = __shfl_up_sync(0xffffffffu, inc, d);
        if (lane >= d) inc = max(inc, x);
    }
    uint32_t before = __shfl_up_sync(0xffffffffu, inc, 1);
    if (lane == 0) before = 0u;
    if (lane == 31) s_max[warp] = inc;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < kBinThreads / 32; ++w)
        if (w < warp) before = max(before, s_max[w]);
    uint32_t key[4], val[4];
    const int64_t pos0 = p0 + 4 * t;
    const int nin = p1 - pos0 >= 4 ? 4 : (int)max((int64_t)0, p1 - pos0);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const uint32_t j = max(before, m[e]);
        const uint2 rg = s_rg[j];
        const int w = (int)(rg.x >> 16), local = (int)((uint32_t)(pos0 + e) - s_off[j]);
        // local / w (both below 2^24): the float quotient is off by one at most
        int row = (int)__fdividef((float)local, (float)w), col = local - row * w;
        if (col < 0) { --row; col += w; }
        else if (col >= w) { ++row; col -= w; }
        const int ty = min((int)(rg.y >> 16), (int)(rg.y & 0xffffu) + row);
        int x = (int)(rg.x & 0xffffu) + col;
        if (wrap_x && x >= ntx) x -= ntx;
        key[e] = (uint32_t)(ty * ntx + x);
        val[e] = s_id[j];
    }
    if (nin == 4) {
        *reinterpret_cast<uint4 *>(keys + pos0) = make_uint4(key[0], key[1], key[2], key[3]);
        *reinterpret_cast<uint4 *>(vals + pos0) = make_uint4(val[0], val[1], val[2], val[3]);
    } else {
        for (int e = 0; e < nin; ++e) {
            keys[pos0 + e] = e == 0 ? key[0] : e == 1 ? key[1] : key[2];
            vals[pos0 + e] = e == 0 ? val[0] : e == 1 ? val[1] : val[2];
        }
    }
    if (hist) {
        // the digit counts of every tile-sort pass
        for (int p = 0; p < passes; ++p) {
            const int b = radix_bit(0, end_bit, p);
            const uint32_t mask = (1u << (radix_bit(0, end_bit, p + 1) - b)) - 1u;
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if (e < nin) atomicAdd(&s_h[p][(key[e] >> b) & mask], 1u);
        }
        __syncthreads();
        for (int i = t; i < passes * 256; i += kBinThreads) {
            const uint32_t c = (&s_h[0][0])[i];
            if (c) atomicAdd(&hist[i], c);
        }
    }
}

sg_status bin_pairs(const uint32_t *d_ids, const uint32_t *d_offsets, const uint32_t *d_nvalid,
                    const int4 *d_tiles, int ntx, int wrap_x, int64_t cap, uint32_t *d_keys,
                    uint32_t *d_vals, cudaStream_t st, const uint32_t *d_err, const Buf &owner,
                    uint2 *d_ranges, int64_t ntiles, uint32_t *d_hist, int end_bit)
{
    if (cap <= 0) {
        SG_CUDA(cudaMemsetAsync(d_ranges, 0, sizeof(uint2) * ntiles, st));
        return SG_OK;
    }
    if (d_hist && (end_bit < 1 || end_bit > 8 * kBinPasses)) {
        set_error("internal: %d-bit tile ids", end_bit);
        return SG_ERR_INVALID;
    }
    launch_after(k_bin, (unsigned)((cap + kBinChunk - 1) / kBinChunk), kBinThreads, 0, st,
        d_ids, d_offsets, d_nvalid, d_tiles, ntx, wrap_x, (uint32_t)cap, d_keys, d_vals, d_hist,
        end_bit, d_err, (const uint32_t *)owner.p, (int64_t)(owner.bytes / 4), d_ranges, ntiles);
    SG_LAUNCHED();
    return SG_OK;
}

// Per-tile [start, end) of the sorted pairs, and for camera lists (kMask)
// a per-pair 32-bit word of the tile's pixel columns (bits 0-15) and rows
// (bits 16-31) whose centres lie inside the Gaussian's extent box, by the
// same float comparisons as the per-ray test.  A compositing warp gets from
// it, in a few integer operations, whether the entry reaches its 8x4
// sub-block and which of its lanes the box holds, so it never stages an
// entry that no live ray of its sub-block can see and loads no box.  After a
// look-back wait gave up (*err) the pairs may hold stale tile ids: every
// range stays empty (zeroed by the binning).
// Each thread takes kRangePer consecutive pairs (16-byte loads of keys and
// ids; the lists' buffers are 256-byte aligned), the boxes' loads issued
// together.  The columns whose centre c + 1/2 is in [lo, hi] are the run from
// ceil(lo - 1/2) to floor(hi - 1/2): the subtraction is exact in float for
// 1/2 <= lo < 2^23, rounds to a value with the same ceiling below 1/2 (every
// lo <= 1/2 starts at column 0), and an image has no columns beyond 2^14.
// Measured: 16 comparisons a side took 20 us for 1.5M pairs and 45 us for
// 3.9M; now 11 and 22.
constexpr int kRangePer = 4;

// Bits of the kTile centres first + 1/2 .. first + kTile - 1/2 in [lo, hi].
__device__ __forceinline__ uint32_t centre_bits(float lo, float hi, int first)
{
    const float f = (float)first;
    const int a = (int)fmaxf(0.f, fminf((float)kTile, ceilf(lo - 0.5f) - f));
    const int b = (int)fmaxf(-1.f, fminf((float)(kTile - 1), floorf(hi - 0.5f) - f));
    return (0xffffu << a) & (0xffffu >> (kTile - 1 - b));
}

// Quotient and remainder of t < 2^24 by n, inv = 1 / n rounded: the float
// quotient is off by one at most.
__device__ __forceinline__ void div_small(uint32_t t, int n, float inv, int &q, int &r)
{
    q = (int)((float)t * inv);
    r = (int)t - q * n;
    if (r < 0) { --q; r += n; }
    else if (r >= n) { ++q; r -= n; }
}

__device__ __forceinline__ void load4(const uint32_t *__restrict__ p, int64_t i, int64_t n,
                                      uint32_t v[kRangePer])
{
    if (i + kRangePer <= n) {
        const uint4 x = *reinterpret_cast<const uint4 *>(p + i);
        v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
    } else {
#pragma unroll
        for (int j = 0; j < kRangePer; ++j) v[j] = i + j < n ? p[i + j] : 0u;
    }
}

// The ends of the tiles' runs among a thread's pairs [i0, i0 + kRangePer).
__device__ __forceinline__ void write_ranges(const uint32_t *__restrict__ keys, int64_t i0, int64_t K,
                                             const uint32_t t[kRangePer], uint2 *__restrict__ ranges)
{
    const uint32_t before = i0 > 0 ? keys[i0 - 1] : 0u;
    const uint32_t after = i0 + kRangePer < K ? keys[i0 + kRangePer] : 0u;
#pragma unroll
    for (int j = 0; j < kRangePer; ++j) {
        const int64_t i = i0 + j;
        if (i >= K) break;
        const uint32_t left = j > 0 ? t[j - 1] : before;
        const uint32_t right = j + 1 < kRangePer ? t[j + 1] : after;
        if (i == 0 || left != t[j]) ranges[t[j]].x = (uint32_t)i;
        if (i == K - 1 || right != t[j]) ranges[t[j]].y = (uint32_t)(i + 1);
    }
}

template <bool kMask>
__global__ void __launch_bounds__(256)
k_ranges(const uint32_t *keys, const uint32_t *d_K,
         uint2 *__restrict__ ranges, const uint32_t *ids,
         const float4 *rects, int ntx, float inv_ntx, uint32_t *__restrict__ mask,
         const uint32_t *err)
{
    after_previous();
    const int64_t i0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * kRangePer;
    const int64_t K = *d_K;
    if (i0 >= K || *err) return;
    uint32_t t[kRangePer], id[kRangePer];
    load4(keys, i0, K, t);
    float4 rc[kRangePer];
    if (kMask) {
        load4(ids, i0, K, id);
#pragma unroll
        for (int j = 0; j < kRangePer; ++j)      // the extent box, 16 B per Gaussian
            rc[j] = i0 + j < K ? rects[id[j]] : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    write_ranges(keys, i0, K, t, ranges);
    if (kMask) {
        uint32_t m[kRangePer];
#pragma unroll
        for (int j = 0; j < kRangePer; ++j) {
            int tx, ty;
            div_small(t[j], ntx, inv_ntx, ty, tx);
            m[j] = centre_bits(rc[j].x, rc[j].y, tx * kTile) |
                   centre_bits(rc[j].z, rc[j].w, ty * kTile) << 16;
        }
        if (i0 + kRangePer <= K) {
            *reinterpret_cast<uint4 *>(mask + i0) = make_uint4(m[0], m[1], m[2], m[3]);
        } else {
#pragma unroll
            for (int j = 0; j < kRangePer; ++j)
                if (i0 + j < K) mask[i0 + j] = m[j];
        }
    }
}

sg_status tile_ranges(const uint32_t *d_keys, const uint32_t *d_K, int64_t K_max, uint2 *d_ranges,
                      cudaStream_t st, const uint32_t *d_err,
                      const uint32_t *d_ids, const float4 *d_rects, int ntx, uint32_t *d_words)
{
    if (K_max == 0) return SG_OK;
    const unsigned grid = (unsigned)((K_max + 256 * kRangePer - 1) / (256 * kRangePer));
    if (d_words)
        launch_after(k_ranges<true>, grid, 256, 0, st, d_keys, d_K, d_ranges, d_ids, d_rects, ntx,
                                             1.f / (float)ntx, d_words, d_err);
    else
        launch_after(k_ranges<false>, grid, 256, 0, st, d_keys, d_K, d_ranges, nullptr, nullptr, 0, 0.f,
                                              nullptr, d_err);
    SG_LAUNCHED();
    return SG_OK;
}

// LiDAR lists: per-tile ranges, and per pair the ray masks of the work
// items of its tile (k-th item of the tile: lmask[k * stride + i]), so that
// the compositing walks skip entries that reach none of their rays without
// loading their records.  A ray is in the box iff its column's azimuth (the
// alias nearest the box centre) and its beam's elevation are, so the mask
// takes one test per column and one per beam of the item.  Both the forward
// and the backward walks read these masks, so they take the same decisions.
// Four consecutive pairs a thread, loaded together; lists are sorted by tile,
// so that the four mostly share one and each table entry is loaded once for
// them.  Measured (2M Gaussians, 3.7M pairs): one pair a thread 43 us, now 36
// (38 with the table read word by word).
__global__ void __launch_bounds__(256)
k_ranges_lidar(const uint32_t *keys, const uint32_t *d_K, int64_t stride,
               uint2 *__restrict__ ranges, const uint32_t *ids,
               const float4 *rects, const uint2 *__restrict__ tile_items,
               const LidarItemRays *__restrict__ tab, uint32_t *__restrict__ lmask,
               const uint32_t *err)
{
    after_previous();
    const int64_t i0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * kRangePer;
    const int64_t K = *d_K;
    if (i0 >= K || *err) return;
    const int np = K - i0 < kRangePer ? (int)(K - i0) : kRangePer;
    uint32_t t[kRangePer], id[kRangePer];
    load4(keys, i0, K, t);
    load4(ids, i0, K, id);
    float4 rc[kRangePer];
    float cx[kRangePer];
#pragma unroll
    for (int j = 0; j < kRangePer; ++j)
        rc[j] = j < np ? rects[id[j]] : make_float4(0.f, 0.f, 0.f, 0.f);
    write_ranges(keys, i0, K, t, ranges);
#pragma unroll
    for (int j = 0; j < kRangePer; ++j) cx[j] = 0.5f * (rc[j].x + rc[j].y);
    // runs [j0, j1) of the pairs that share a tile (all four, mostly)
    for (int j0 = 0; j0 < np;) {
        const uint32_t tile = j0 == 0 ? t[0] : j0 == 1 ? t[1] : j0 == 2 ? t[2] : t[3];
        int j1 = j0 + 1;
#pragma unroll
        for (int j = 1; j < kRangePer; ++j)
            if (j == j1 && j < np && t[j] == tile) j1 = j + 1;
        const uint2 ti = tile_items[tile];
        for (uint32_t k = 0; k < ti.y; ++k) {
            const LidarItemRays &R = tab[ti.x + k];
            uint32_t mc[kRangePer] = {0u, 0u, 0u, 0u}, me[kRangePer] = {0u, 0u, 0u, 0u};
            const float4 az4 = *reinterpret_cast<const float4 *>(R.col_az);
            const uint4 cb4 = *reinterpret_cast<const uint4 *>(R.col_bits);
            const float az[4] = {az4.x, az4.y, az4.z, az4.w};
            const uint32_t cb[4] = {cb4.x, cb4.y, cb4.z, cb4.w};     // 0: no such column
            const int nbeams = R.nbeams;
#pragma unroll
            for (int s = 0; s < kLidarColsMax; ++s) {
#pragma unroll
                for (int j = 0; j < kRangePer; ++j) {
                    const float ra = az[s] + 360.f * rintf((cx[j] - az[s]) * (1.f / 360.f));
                    mc[j] |= (ra >= rc[j].x && ra <= rc[j].y) ? cb[s] : 0u;
                }
            }
            for (int b0 = 0; b0 < nbeams; b0 += 4) {
                const float4 el4 = *reinterpret_cast<const float4 *>(R.beam_el + b0);
                const uint4 bb4 = *reinterpret_cast<const uint4 *>(R.beam_bits + b0);
                const float el[4] = {el4.x, el4.y, el4.z, el4.w};
                const uint32_t bb[4] = {bb4.x, bb4.y, bb4.z, bb4.w};  // 0: no such beam
#pragma unroll
                for (int b = 0; b < 4; ++b)
#pragma unroll
                    for (int j = 0; j < kRangePer; ++j)
                        me[j] |= (el[b] >= rc[j].z && el[b] <= rc[j].w) ? bb[b] : 0u;
            }
            uint32_t *out = lmask + (int64_t)k * stride + i0;
            if (j0 == 0 && j1 == kRangePer) {
                *reinterpret_cast<uint4 *>(out) =
                    make_uint4(mc[0] & me[0], mc[1] & me[1], mc[2] & me[2], mc[3] & me[3]);
            } else {
#pragma unroll
                for (int j = 0; j < kRangePer; ++j)
                    if (j >= j0 && j < j1) out[j] = mc[j] & me[j];
            }
        }
        j0 = j1;
    }
}

sg_status lidar_tile_ranges(const uint32_t *d_keys, const uint32_t *d_K, int64_t K_max,
                            uint2 *d_ranges, cudaStream_t st, const uint32_t *d_err,
                            const uint32_t *d_ids, const float4 *d_rects, const Lidar &L,
                            uint32_t *d_lmask,
                            int64_t lmask_stride)
{
    if (K_max == 0) return SG_OK;
    const unsigned grid = (unsigned)((K_max + 256 * kRangePer - 1) / (256 * kRangePer));
    launch_after(k_ranges_lidar, grid, 256, 0, st,
        d_keys, d_K, lmask_stride, d_ranges, d_ids, d_rects, L.d_tile_items, L.d_item_ray_tab,
        d_lmask, d_err);
    SG_LAUNCHED();
    return SG_OK;
}

// Capacity mode: keep at most `cap` pairs; d_K is clamped to it and the
// number of pairs beyond it is stored in d_dropped (0 when all fit).
__global__ void k_clamp_pairs(uint32_t *d_K, uint32_t cap,
                              uint32_t *__restrict__ d_dropped)
{
    after_previous();
    const uint32_t K = *d_K;
    *d_dropped = K > cap ? K - cap : 0u;
    if (K > cap) *d_K = cap;
}

sg_status clamp_pairs(uint32_t *d_K, int64_t cap, uint32_t *d_dropped, cudaStream_t st)
{
    launch_after(k_clamp_pairs, 1, 1, 0, st, d_K, (uint32_t)cap, d_dropped);
    SG_LAUNCHED();
    return SG_OK;
}

}  // namespace sg

extern "C" sg_status sg_debug_lookback(uint32_t max_spins, int hold_site, int64_t hold_tile)
{
    if (hold_site < 0 || hold_site > SG_LOOKBACK_TILE_SORT || hold_tile < -1) {
        sg::set_error("sg_debug_lookback: site %d / tile %lld out of range", hold_site,
                      (long long)hold_tile);
        return SG_ERR_INVALID;
    }
    const uint32_t spins = max_spins ? max_spins : sg::kLbSpinsDefault;
    const long long tile = hold_site ? (long long)hold_tile : -1;
    SG_CUDA(cudaDeviceSynchronize());   // no kernel reads them meanwhile
    SG_CUDA(cudaMemcpyToSymbol(sg::g_lb_spins, &spins, sizeof(spins)));
    SG_CUDA(cudaMemcpyToSymbol(sg::g_hold_site, &hold_site, sizeof(hold_site)));
    SG_CUDA(cudaMemcpyToSymbol(sg::g_hold_tile, &tile, sizeof(tile)));
    return SG_OK;
}
