// DENSE multi-hop sampling (Algorithm 1) for many independent mini-batches per pass.
//
// Layout kept on the device (hop-major, sampling order):
//   nodes[]     hop 0 = the targets of all batches, hop h+1 = the deltas found from hop h,
//               inside a hop batch after batch, inside a batch in the order found (targets: caller order)
//   ent_off[]   for each sampled node its first entry in ent_nbrs / ent_repr (same order as nodes)
//   ent_repr[]  the neighbour's LOCAL row: its position in the batch's node list taken in
//               sampling order (targets first).  In that order the rows layer l needs are the
//               prefix [0, N_l) of the batch, which is what Algorithm 2 achieves by cutting the
//               front of node_ids in the paper's (reversed) order.
// The paper's arrays, with ascending ids inside a delta, are produced from this by mg_dense_view and
// mg_dense_export_many.
//
// Every kernel sizes itself from counters in device memory (DenseHeader), so a k-hop sample is
// issued without a host round trip per hop; the host reads the header once at the end.

#include <stdarg.h>

#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <utility>

#include "mg_device.cuh"
#include "mg_internal.cuh"

namespace {

constexpr int kThreads = 256;
constexpr int64_t kStageTargets = 16384;   // targets in host memory that are read without a copy of their own

// -------------------------------------------------------------------------------------
// generic exclusive scan over a device-sized range (three kernels, no inter-block waits)
// -------------------------------------------------------------------------------------
constexpr int kScanTile = 2048;  // 256 threads x 8

struct ScanRange {       // all device pointers
    const int32_t* lo;   // range is data[*lo .. *hi)
    const int32_t* hi;
    const int32_t* base; // value added to every output (nullable)
};

__device__ __forceinline__ uint32_t block_excl_scan_256(uint32_t v, uint32_t* smem /*>= 9*/, uint32_t* total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t inc = warp_incl_scan(v);
    if (lane == 31) smem[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        uint32_t w = lane < 8 ? smem[lane] : 0u;
        const uint32_t wi = warp_incl_scan(w);
        if (lane < 8) smem[lane] = wi - w;
        if (lane == 7) smem[8] = wi;
    }
    __syncthreads();
    const uint32_t res = inc - v + smem[warp];
    *total = smem[8];
    __syncthreads();
    return res;
}

__global__ void __launch_bounds__(kThreads) k_scan_reduce(const uint32_t* data, ScanRange r, uint32_t* tile_sums) {
    __shared__ uint32_t sm[9];
    const int32_t lo = *r.lo, n = *r.hi - lo;
    const int ntiles = (n + kScanTile - 1) / kScanTile;
    for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
        uint32_t s = 0;
        const int start = t * kScanTile + threadIdx.x * 8;
#pragma unroll
        for (int j = 0; j < 8; ++j)
            if (start + j < n) s += data[lo + start + j];
        uint32_t total;
        block_excl_scan_256(s, sm, &total);
        if (threadIdx.x == 0) tile_sums[t] = total;
    }
}

// single block: exclusive scan of the tile sums in place; total (plus base) to *total_out
__global__ void __launch_bounds__(1024) k_scan_tiles(uint32_t* tile_sums, ScanRange r, uint32_t* total_out) {
    __shared__ uint32_t warp_tot[33];
    const int n = *r.hi - *r.lo;
    const int ntiles = (n + kScanTile - 1) / kScanTile;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t carry = 0;
    for (int start = 0; start < ntiles; start += 1024) {
        const int i = start + threadIdx.x;
        const uint32_t v = i < ntiles ? tile_sums[i] : 0u;
        const uint32_t inc = warp_incl_scan(v);
        if (lane == 31) warp_tot[warp] = inc;
        __syncthreads();
        if (warp == 0) {
            const uint32_t w = warp_tot[lane];
            const uint32_t wi = warp_incl_scan(w);
            warp_tot[lane] = wi - w;
            if (lane == 31) warp_tot[32] = wi;
        }
        __syncthreads();
        if (i < ntiles) tile_sums[i] = carry + warp_tot[warp] + inc - v;
        carry += warp_tot[32];
        __syncthreads();
    }
    if (threadIdx.x == 0 && total_out) *total_out = carry + (r.base ? (uint32_t)*r.base : 0u);
}

__global__ void __launch_bounds__(kThreads) k_scan_down(uint32_t* data, ScanRange r, const uint32_t* tile_sums) {
    __shared__ uint32_t sm[9];
    const int32_t lo = *r.lo, n = *r.hi - lo;
    const uint32_t base = r.base ? (uint32_t)*r.base : 0u;
    const int ntiles = (n + kScanTile - 1) / kScanTile;
    for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
        uint32_t v[8], s = 0;
        const int start = t * kScanTile + threadIdx.x * 8;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            v[j] = (start + j < n) ? data[lo + start + j] : 0u;
            s += v[j];
        }
        uint32_t total;
        uint32_t run = block_excl_scan_256(s, sm, &total) + tile_sums[t] + base;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            if (start + j < n) data[lo + start + j] = run;
            run += v[j];
        }
    }
}

// -------------------------------------------------------------------------------------
// begin of a sample
// -------------------------------------------------------------------------------------
struct TableGeom {
    int32_t size;   // slots per batch (a multiple of 8)
};

// The host-known part of a sample (header, target offsets, per-batch row tables, seeds) is read straight from mapped
// pinned memory by a kernel instead of being copied by a copy engine: a copy engine may be busy for a long time with
// a partition that is being swapped in, and the sample would wait behind it.  The same kernel clears the id tables and the
// counters: a memset node in the captured graph held the kernels behind it up by 10 to 14 us.
struct BeginArgs {
    const int32_t* stage;
    int32_t n_hdr, n_off, n_cum, n_seed_words, seed_at, n_cnt;
    int64_t n_table4;   // 16-byte pieces of the id tables
    int32_t *hdr, *node_off, *cum, *seeds, *batch_cnt;
    int4* hkeys;
};
__global__ void __launch_bounds__(kThreads) k_begin(BeginArgs a) {
    const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, step = (int64_t)gridDim.x * blockDim.x;
    const int32_t total = a.n_hdr + a.n_off + a.n_cum + a.n_seed_words;
    for (int64_t i = tid; i < total; i += step) {
        int32_t j = (int32_t)i;
        if (j < a.n_hdr) a.hdr[j] = a.stage[j];
        else if ((j -= a.n_hdr) < a.n_off) a.node_off[j] = a.stage[a.n_hdr + j];
        else if ((j -= a.n_off) < a.n_cum) a.cum[j] = a.stage[a.n_hdr + a.n_off + j];
        else a.seeds[j - a.n_cum] = a.stage[a.seed_at + (j - a.n_cum)];
    }
    for (int64_t i = tid; i < a.n_cnt; i += step) a.batch_cnt[i] = 0;
    for (int64_t i = tid; i < a.n_table4; i += step) a.hkeys[i] = make_int4(-1, -1, -1, -1);
}

// -------------------------------------------------------------------------------------
// per hop: count, scan and pick in one kernel
// -------------------------------------------------------------------------------------
// Bound by the latency of random look-ups (a node's row bounds, then one DRAM burst per picked id) and, for small hops, by
// launches: one thread per node reads the row bounds, the tile's entry counts are scanned in the block, the tiles' running
// totals are chained through one 64-bit word per tile (decoupled look-back), and the block's warps then pick for the tile's
// nodes from shared memory.  Before, these were five kernels with the row bounds, degrees and counts going through memory
// between them (one mini-batch of three hops on 1M nodes: 48 -> 32 us; 128 mini-batches, last hop of 2.7M nodes: 315 -> 288
// us).  A tile has as few nodes as leave one for every block that the SMs hold (hop_tile): the picks of a warp's nodes are one chain after
// the other, and a hop of 1,000 nodes took 21 us with 256 of them per block, 10 us with 32.  Tiles are handed out by a
// counter, as chain_tiles wants it.
// Hop 0 also enters the targets: residency and range checks, the id table (Algorithm 1 wants unique targets).  The other hops start from the
// counts of new nodes per mini-batch: every block sums them up for itself (block 0 writes the sums down), and the tiles' nodes are
// read from the mini-batches' runs of new ids and put one behind the other on the way (a kernel of its own for
// that took 3.4 to 5 us per hop of one mini-batch, 26 us for the two inner hops of 128).  Small calls gain a launch per hop; on large ones the
// hops take up what the placing leaves: with k_place 170 -> 164 us for 32 mini-batches of 114,000 nodes, 467 -> 465 for 128.
struct HopArgs {
    DenseHeader* hdr;
    int hop;
    int32_t fanout;
    int32_t* nodes;
    int32_t* node_batch;
    const int64_t* row_off[2];    // [1] null: one direction; else the outgoing list, whose picks follow the first list's
    const int32_t* row_nbrs[2];
    int32_t* ent_off;
    int32_t* ent_nbrs;
    int32_t* ent_repr;            // receives the batch id of the entry (k_insert turns it into the id-table slot)
    int32_t batch_of_entry;       // (0: nobody reads it, and a thread per node leaves it out)
    const uint64_t* seeds;
    int64_t cap_entries;
    uint64_t* tile_state;
    int32_t tile_cap;             // nodes of a tile that the launch has shared memory for
    int32_t n_sms, per_sm;        // (blocks of this instance that an SM holds)
    int32_t B, k;
    // hops > 0: the nodes are what k_insert found new in the hop before
    const int32_t* new_ids;       // by rank, mini-batch b's from the place of its first entry on
    const uint32_t* batch_cnt;    // [B] how many
    int64_t cap_nodes;
    int32_t node_limit;           // nodes that a mini-batch may have with them
    int32_t* cum;
    int32_t* node_off;
    // hop 0
    const int32_t* tgt_off;
    int32_t* hkeys;
    int32_t* hvals;
    TableGeom tg;
    int64_t n_nodes;
    FeatGeom feat;
};

// Blocks of k_hop that an SM holds by their registers.  Groups of lanes: five (declared for four they take 48 registers; declared for five they
// lose loads in flight).  A thread per node: four of 64 registers, five for the fanouts that leave few look-ups in flight anyway (0.5M nodes of 2 in
// blocks of 48 registers 57 us, of 64 registers 65).
constexpr int kHopBlocks = 5;
__host__ __device__ constexpr int hop_blocks(bool thread, int f) { return thread && f > 2 ? 4 : kHopBlocks; }

// Nodes of a tile.  Below 256 as few as leave a tile for every block that the SMs hold (groups of lanes: with four per SM the hop of one
// mini-batch takes 34.9 us instead of 28.7; a thread per node, where a fifth waits for a second wave: 94,000 nodes of 5 in tiles for four
// 15 us, for five 21); above 256 where twelve tiles per SM are left all the same: the chain through the tiles costs about 13 ns each (2.7M nodes:
// 620 us with tiles of 64, 475 with 128, 342 with 256, 288 with 1,024).  A thread per node has tiles of up to 512 for the first reason too: it takes
// two nodes at little more than the time of one, and tiles of 256 came to a second wave (200,000 nodes of 1 23.0 -> 18.3 us, 18.7 by groups of lanes; of 5
// 25.3 -> 17.8, both lists of 10 43.3 -> 37.9).
constexpr int kTilesPerSmLarge = 12, kTileMax = 1024, kTileSets = kTileMax / kThreads;
constexpr int kTileParts = kTileSets * kThreads / 32;
static_assert(kTileParts <= 32, "one warp scans the tile's warp totals");
__host__ __device__ __forceinline__ int hop_tile(int64_t n, int n_sms, int per_sm, bool thread = false) {
    for (int t = 32; t < (thread ? kTileMax : kThreads); t <<= 1)
        if (n <= (int64_t)t * per_sm * n_sms) return t;
    for (int t = kTileMax; t > kThreads; t >>= 1)
        if (n > (int64_t)t * kTilesPerSmLarge * n_sms) return t;
    return kThreads;
}
// shared memory per node of a tile: id, mini-batch, first entry; first edge and length of its row, once per direction
__host__ __device__ __forceinline__ int hop_node_bytes(bool inout) { return 12 + (inout ? 24 : 12); }

// Fanouts of up to kThreadPicks are picked by a thread per node where the hop may have tiles of kThreads nodes, else by a group of lanes per node.  Lanes: one look-up in flight per lane and as many Philox calls as draws; threads:
// a quarter of the calls and all of a node's look-ups in flight.  us, lanes / threads: 71,000 nodes of 20 in one mini-batch 47 / 23, 2.7M nodes of 5 302 / 297
// (DRAM bursts of the picks), 0.5M 67 / 54, 128,000 of 15 36 / 27, 0.3M of 10 55 / 38, of 7 49 / 33, both lists 90 / 55 and 81 / 52; on 16M nodes,
// whose look-ups are DRAM bursts, 0.32M of 10 88 / 91.  Hops without caps may
// have far less than their bound: 2,320 nodes of 10 8.3 / 8.3, 22,000 of 5 13.3 / 9.4, of 20 23.3 / 16.2, both lists 22,400 of 5 15.5 / 12.0, of 12 23.9 / 24.3, of 20
// 36.7 / 28.7, 69,600 of 10 44.8 / 32.0.  (There the small tiles had been left to groups of lanes, four blocks or fewer to an SM instead of five: 36.5 -> 45.)
constexpr int kThreadPicks = 20;
static bool hop_by_thread(int f, int64_t bound, int n_sms) { return hop_tile(bound, n_sms, kHopBlocks) >= kThreads && f <= kThreadPicks; }
// shared memory for the picks of a block's threads
static size_t hop_pick_bytes(int f, bool inout) { return (size_t)kThreads * f * (inout ? 2 : 1) * sizeof(uint32_t); }

// Shared memory of the blocks on one SM, and what of it leaves look-ups a useful L1: the driver takes the smallest split that holds the blocks, and beyond
// 196 KiB that is the one of 228, with 28 KiB left (2M nodes of 6 in both lists, four blocks of 48 KiB: 818 us, groups of lanes 552).  A thread per node stays below it:
// in the largest tiles of which all blocks do, or, where the picks alone are too many, with fewer blocks.
constexpr size_t kSmemPerSm = 228 * 1024, kSmemWithL1 = 196 * 1024, kSmemOfBlock = 1024 + 256;   // (the system's part of a block and its static variables)

// How a hop of at most `bound` nodes is launched; `tables`: bytes of the mini-batches' tables.  (us, always 1,024 nodes a tile / smaller ones: both lists,
// 2M nodes of 6 818 / 424, 1M of 15 833 / 408; fewer blocks: 0.5M of 20 551 / 318, 94,000 of 20 147 / 70.)
struct HopLaunch {
    bool thread;        // a thread per node
    int32_t per_sm;     // blocks that an SM holds
    int32_t tile_cap;   // nodes of a tile at most
    size_t smem;
};
static HopLaunch hop_launch(int f, int64_t bound, int n_sms, bool inout, size_t tables) {
    HopLaunch l;
    l.thread = hop_by_thread(f, bound, n_sms);
    l.per_sm = hop_blocks(l.thread, f);
    l.tile_cap = hop_tile(bound, n_sms, l.per_sm, l.thread);
    if (l.thread && bound > (int64_t)kThreads * l.per_sm * n_sms) l.tile_cap = std::max(l.tile_cap, kTileMax / 2);   // (fewer nodes than the bound may want larger tiles)
    auto room = [&](int tile) { return tables + (size_t)tile * hop_node_bytes(inout) + (l.thread ? hop_pick_bytes(f, inout) : 0); };
    if (l.thread) {
        int tile = l.tile_cap;
        while (tile > kThreads && l.per_sm * (room(tile) + kSmemOfBlock) > kSmemWithL1) tile /= 2;
        if (l.per_sm * (room(tile) + kSmemOfBlock) <= kSmemWithL1) l.tile_cap = tile;
        else while (l.per_sm > 2 && l.per_sm * (room(l.tile_cap) + kSmemOfBlock) > kSmemWithL1) --l.per_sm;
    }
    l.smem = room(l.tile_cap);
    if (l.thread && l.per_sm < hop_blocks(true, f)) l.smem = std::max(l.smem, kSmemPerSm / (l.per_sm + 1));   // (no room for one more)
    if (f > 32) l.smem += (size_t)(kThreads / 32) * 2 * f * sizeof(uint32_t);   // (64 KiB at the largest fanout)
    return l;
}

// the mini-batch of target i: a 32-way search of the warp for its first target, then a walk
__device__ __forceinline__ int target_batch(const int32_t* __restrict__ off, int B, int32_t first, int32_t i) {
    const int lane = threadIdx.x & 31;
    int lo = 0, len = B;   // off[lo] <= first, the answer lies in [lo, lo + len)
    while (len > 1) {
        const int step = (len + 31) / 32;
        const uint32_t below = __ballot_sync(0xFFFFFFFFu, lane * step < len && off[lo + min(lane * step, len - 1)] <= first);   // lane 0 always
        const int last = 31 - __clz(below);
        lo += last * step;
        len = min(step, len - last * step);
    }
    while (off[lo + 1] <= i) ++lo;
    return lo;
}

// Floyd's subset algorithm, G lanes per node: slot t draws x in [0, d-f+t]; it keeps x unless an earlier slot already holds
// x, in which case it keeps d-f+t.  Draws are independent of each other, so all lanes draw at once and only the "already
// held" test runs slot by slot.  It is left out when no two draws of a node are alike: slot 0 keeps its draw, and so does
// every later slot, as the earlier ones hold nothing but their own.  Returns the lane's position in the row, *rank its rank
// among the f picks.
template <int G>
__device__ __forceinline__ uint32_t floyd_pick(bool on, uint32_t d, int32_t f, int gl, int gshift, uint64_t seed, uint32_t v, uint32_t hop,
                                               uint32_t slot_base, int* rank) {
    const uint32_t gmask = (G == 32) ? 0xFFFFFFFFu : (((1u << (G & 31)) - 1u) << gshift);
    uint32_t x = 0xFFFFFFFFu, jt = 0, pick = 0xFFFFFFFFu;
    if (on && gl < f) {
        jt = d - (uint32_t)f + (uint32_t)gl;
        x = __umulhi(draw_word(seed, v, hop, slot_base + (uint32_t)gl), jt + 1u);
    }
    const uint32_t same = __match_any_sync(0xFFFFFFFFu, x) & gmask;
    if (!__any_sync(0xFFFFFFFFu, on && gl < f && same != 1u << (threadIdx.x & 31))) pick = x;
    else
        for (int t = 0; t < f; ++t) {
            const uint32_t xt = __shfl_sync(0xFFFFFFFFu, x, gshift + t);
            const uint32_t hit = __ballot_sync(0xFFFFFFFFu, gl < t && pick == xt) & gmask;
            if (gl == t) pick = hit ? jt : xt;
        }
    // (the f picks are distinct; every lane of the warp takes part in the shuffles, whatever its node needs)
    int r = 0;
    for (int t = 0; t < f; ++t) {
        const uint32_t pt = __shfl_sync(0xFFFFFFFFu, pick, gshift + t);
        r += (pt < pick) ? 1 : 0;
    }
    *rank = r;
    return pick;
}

// Batcher's odd-even merge sort of N values as a list of exchanges, so that a thread can sort what it holds in registers.
template <int N> struct SortNet {
    int n;
    int a[N <= 1 ? 1 : N * N], b[N <= 1 ? 1 : N * N];
    constexpr SortNet() : n(0), a(), b() {
        for (int p = 1; p < N; p *= 2)
            for (int k = p; k >= 1; k /= 2)
                for (int j = k % p; j + k < N; j += 2 * k)
                    for (int i = 0; i < k && i + j + k < N; ++i)
                        if ((i + j) / (2 * p) == (i + j + k) / (2 * p)) { a[n] = i + j; b[n] = i + j + k; ++n; }
    }
};
template <int I, int J>
__device__ __forceinline__ void exchange(uint32_t* x) {
    const uint32_t lo = min(x[I], x[J]), hi = max(x[I], x[J]);
    x[I] = lo; x[J] = hi;
}
template <int N, int... C>
__device__ __forceinline__ void sort_values(uint32_t* x, std::integer_sequence<int, C...>) {
    constexpr SortNet<N> net;
    (exchange<net.a[C], net.b[C]>(x), ...);
}

// Floyd's subset algorithm, a thread per node: the same draws as floyd_pick's, a Philox call for every four of them.  pick[0 .. f) are
// the picks in ascending order.
template <int G>
__device__ __forceinline__ void floyd_thread(uint32_t d, int32_t f, uint64_t seed, uint32_t v, uint32_t hop, uint32_t slot_base, uint32_t (&pick)[G]) {
#pragma unroll
    for (int c = 0; c < G; c += 4) {
        uint32_t w[4];
        philox4x32_10(v, 0u, hop, (slot_base + (uint32_t)c) >> 2, (uint32_t)seed, (uint32_t)(seed >> 32), w);
#pragma unroll
        for (int u = 0; u < 4 && c + u < G; ++u) pick[c + u] = w[u];
    }
#pragma unroll
    for (int t = 0; t < G; ++t) {
        const uint32_t jt = d - (uint32_t)f + (uint32_t)t;
        const uint32_t x = __umulhi(pick[t], jt + 1u);
        bool hit = false;
#pragma unroll
        for (int q = 0; q < t; ++q) hit |= pick[q] == x;
        pick[t] = t < f ? (hit ? jt : x) : 0xFFFFFFFFu;
    }
    constexpr SortNet<G> net;
    sort_values<G>(pick, std::make_integer_sequence<int, net.n>{});
}

// A hop's nodes per mini-batch, summed up over the mini-batches: the new nodes of hop - 1 are hop's.  Every block takes the sums for itself
// (a kernel of one block for it cost 2 us and a gap per hop); block 0 writes them down.  Returns one past the hop's last node.
struct NewNodes {
    DenseHeader* hdr;
    int32_t hop, B, k;
    const uint32_t* batch_cnt;   // [B] new nodes of hop - 1
    int64_t cap_nodes;
    int32_t node_limit;          // nodes that a mini-batch may have with them
    const int32_t* ent_off;
    int32_t* cum;
    int32_t* node_off;
};
__device__ __forceinline__ int64_t sum_new_nodes(const NewNodes& a, int32_t* next_off, int32_t* list_at, uint32_t* part /* [kThreads / 32] */) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t carry = (uint32_t)a.hdr->hop_base[a.hop];
    for (int s0 = 0; s0 < a.B; s0 += kThreads) {
        const int b = s0 + (int)threadIdx.x;
        const uint32_t v = b < a.B ? a.batch_cnt[b] : 0u;
        const int32_t run = b < a.B ? a.ent_off[a.node_off[(a.hop - 1) * (a.B + 1) + b]] : 0;
        const uint32_t inc = warp_incl_scan(v);
        if (lane == 31) part[warp] = inc;
        __syncthreads();
        uint32_t before = carry, total = 0;
        for (int w = 0; w < kThreads / 32; ++w) { if (w < warp) before += part[w]; total += part[w]; }
        if (b < a.B) {
            next_off[b] = (int32_t)(before + inc - v);
            list_at[b] = run;
            if (blockIdx.x == 0) {
                a.node_off[a.hop * (a.B + 1) + b] = next_off[b];
                const int32_t rows = a.cum[b * (a.k + 2) + a.hop] + (int32_t)v;
                a.cum[b * (a.k + 2) + a.hop + 1] = rows;
                if (rows > a.node_limit) atomicOr(&a.hdr->status, ST_CAP_TABLE);
            }
        }
        carry += total;
        __syncthreads();
    }
    const int64_t end = carry;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        if (end > a.cap_nodes) atomicOr(&a.hdr->status, ST_CAP_NODES);
        else {
            a.hdr->hop_base[a.hop + 1] = (int32_t)end;
            a.node_off[a.hop * (a.B + 1) + a.B] = (int32_t)end;
        }
    }
    return end;
}

// G lanes per node, fanout <= G <= 32; a warp holds 32 / G nodes (G need not divide 32: the lanes left over idle, and
// G = 5 or 10 keeps 30 lanes busy where the next power of two keeps 20).  G = 0: any fanout up to MG_MAX_FANOUT, a node per
// warp at a time, picks staged in shared memory.
// THREAD (G <= kThreadPicks): a thread per node, for hops of many nodes.
template <int G, bool THREAD>
__global__ void __launch_bounds__(kThreads, THREAD ? hop_blocks(true, G) : 4) k_hop(HopArgs a) {
    extern __shared__ __align__(16) uint8_t hop_sm[];   // the tile's nodes, then (G = 0) per warp x[f], pick[f]
    __shared__ uint32_t part[kTileParts];
    __shared__ int32_t sh_tile;
    __shared__ uint32_t sh_before, sh_end;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int32_t f = a.fanout;
    const bool inout = a.row_off[1] != nullptr;
    int32_t* next_off = reinterpret_cast<int32_t*>(hop_sm);   // [B] (hops > 0) first node of the mini-batch in the hop ...
    int32_t* list_at = next_off + a.B;                        // ... and its run of new_ids
    const int32_t lo = a.hdr->hop_base[a.hop];
    int32_t n;
    if (a.hop == 0) n = a.hdr->hop_base[1] - lo;
    else {
        if (__syncthreads_or(a.hdr->status != 0)) return;   // (the whole block: another one may be setting it)
        const int64_t end = sum_new_nodes({a.hdr, a.hop, a.B, a.k, a.batch_cnt, a.cap_nodes, a.node_limit, a.ent_off, a.cum, a.node_off}, next_off, list_at, part);
        if (end > a.cap_nodes) return;   // (nothing is written outside the arenas; the kernels that follow see the status)
        n = (int32_t)(end - lo);
    }
    // (an empty hop has one empty tile: it closes the entry range)
    const int32_t tile_nodes = min(hop_tile(n, a.n_sms, a.per_sm, THREAD), a.tile_cap), n_tiles = max(1, (n + tile_nodes - 1) / tile_nodes);
    const int sets = (tile_nodes + kThreads - 1) / kThreads;   // nodes per thread
    int64_t* node_r0 = reinterpret_cast<int64_t*>(hop_sm + (a.hop > 0 ? 8 * (size_t)a.B : 0));   // [dirs][tile_cap]
    uint32_t* node_deg = reinterpret_cast<uint32_t*>(node_r0 + (inout ? 2 : 1) * a.tile_cap);   // [dirs][tile_cap]
    int32_t* node_id = reinterpret_cast<int32_t*>(node_deg + (inout ? 2 : 1) * a.tile_cap);
    int32_t* node_b = node_id + a.tile_cap;
    uint32_t* node_out = reinterpret_cast<uint32_t*>(node_b + a.tile_cap);
    const uint64_t tag = (((uint64_t)a.hdr->epoch << 3) | (uint64_t)a.hop) * kChainTag;
    const int32_t* __restrict__ targets = reinterpret_cast<const int32_t*>(a.hdr->targets);
    for (;;) {
        __syncthreads();
        // (after an error no block takes another tile; one that was taken is always closed)
        if (threadIdx.x == 0) sh_tile = *reinterpret_cast<volatile uint32_t*>(&a.hdr->status) ? INT32_MAX : (int32_t)atomicAdd(&a.hdr->ticket[a.hop], 1u);
        __syncthreads();
        const int32_t tile = sh_tile;
        if (tile >= n_tiles) break;
        const int32_t n_here = min(tile_nodes, n - tile * tile_nodes);
        // node t = q * 256 + thread of the tile: its id and row bounds
        uint32_t inc[kTileSets];
        if constexpr (THREAD) {
            // the look-ups of all sets are in flight before the first is used
            int32_t vs[kTileSets], bs[kTileSets];
            uint32_t cnt[kTileSets];
#pragma unroll
            for (int q = 0; q < kTileSets; ++q) {
                const int32_t t = q * kThreads + (int32_t)threadIdx.x, local = tile * tile_nodes + t;
                vs[q] = 0; bs[q] = 0; cnt[q] = 0;
                if (q >= sets) continue;
                if (a.hop == 0) {
                    if (t < n_here) vs[q] = targets[local];
                    if (t - lane < n_here) bs[q] = target_batch(a.tgt_off, a.B, local - lane, min(local, n - 1));
                } else if (t < n_here) {
                    bs[q] = upper_segment(next_off, a.B, lo + local);
                    vs[q] = __ldg(a.new_ids + list_at[bs[q]] + (lo + local - next_off[bs[q]]));
                }
            }
#pragma unroll
            for (int dir = 0; dir < 2; ++dir) {   // incoming + outgoing sampling: up to `fanout` of each list
                if (dir == 1 && !inout) break;
                const int64_t* __restrict__ off = a.row_off[dir];
                int64_t r0[kTileSets], r1[kTileSets];
#pragma unroll
                for (int q = 0; q < kTileSets; ++q) {
                    const int32_t t = q * kThreads + (int32_t)threadIdx.x;
                    r0[q] = 0; r1[q] = 0;
                    if (q < sets && t < n_here && (a.hop > 0 || (vs[q] >= 0 && (int64_t)vs[q] < a.n_nodes))) { r0[q] = __ldg(off + vs[q]); r1[q] = __ldg(off + vs[q] + 1); }
                }
#pragma unroll
                for (int q = 0; q < kTileSets; ++q) {
                    const int32_t t = q * kThreads + (int32_t)threadIdx.x;
                    if (q >= sets || t >= n_here) continue;
                    const uint32_t d = (uint32_t)(r1[q] - r0[q]);
                    cnt[q] += min(d, (uint32_t)f);
                    node_r0[dir * a.tile_cap + t] = r0[q];
                    node_deg[dir * a.tile_cap + t] = d;
                }
            }
#pragma unroll
            for (int q = 0; q < kTileSets; ++q) {
                if (q >= sets) break;
                const int32_t t = q * kThreads + (int32_t)threadIdx.x, local = tile * tile_nodes + t;
                if (t < n_here) {
                    node_id[t] = vs[q]; node_b[t] = bs[q]; node_out[t] = cnt[q];
                    if (a.hop > 0) {
                        a.nodes[lo + local] = vs[q];
                        a.node_batch[lo + local] = bs[q];
                    }
                }
                inc[q] = warp_incl_scan(cnt[q]);
                if (lane == 31) part[q * (kThreads / 32) + warp] = inc[q];
            }
        } else {
#pragma unroll
            for (int q = 0; q < kTileSets; ++q) {
                if (q >= sets) break;
                const int32_t t = q * kThreads + (int32_t)threadIdx.x, local = tile * tile_nodes + t;
                const bool node_ok = t < n_here;
                int32_t v = 0, b = 0;
                bool in_range = node_ok;
                if (node_ok) {
                    if (a.hop == 0) v = targets[local];
                    else {
                        b = upper_segment(next_off, a.B, lo + local);
                        v = a.new_ids[list_at[b] + (lo + local - next_off[b])];
                        a.nodes[lo + local] = v;
                        a.node_batch[lo + local] = b;
                    }
                }
                if (a.hop == 0) {
                    if (t - lane < n_here) b = target_batch(a.tgt_off, a.B, local - lane, min(local, n - 1));
                    in_range = node_ok && v >= 0 && (int64_t)v < a.n_nodes;
                }
                uint32_t cnt = 0;
                if (in_range) {
                    const int64_t r0 = a.row_off[0][v];
                    const uint32_t d = (uint32_t)(a.row_off[0][v + 1] - r0);
                    cnt = min(d, (uint32_t)f);
                    node_r0[t] = r0;
                    node_deg[t] = d;
                    if (inout) {   // incoming + outgoing sampling: up to `fanout` of each list
                        const int64_t q0 = a.row_off[1][v];
                        const uint32_t dq = (uint32_t)(a.row_off[1][v + 1] - q0);
                        cnt += min(dq, (uint32_t)f);
                        node_r0[a.tile_cap + t] = q0;
                        node_deg[a.tile_cap + t] = dq;
                    }
                } else if (node_ok) {
                    node_r0[t] = 0; node_deg[t] = 0;
                    if (inout) { node_r0[a.tile_cap + t] = 0; node_deg[a.tile_cap + t] = 0; }
                }
                if (node_ok) { node_id[t] = v; node_b[t] = b; node_out[t] = cnt; }
                inc[q] = warp_incl_scan(cnt);
                if (lane == 31) part[q * (kThreads / 32) + warp] = inc[q];
            }
        }
        __syncthreads();
        // entries before each warp's nodes inside the tile, the tile's count; the tiles before this one
        if (warp == 0) {
            const uint32_t w = lane < sets * (kThreads / 32) ? part[lane] : 0u;
            const uint32_t wi = warp_incl_scan(w);
            const uint32_t total = __shfl_sync(0xFFFFFFFFu, wi, 31);
            if (lane < kTileParts) part[lane] = wi - w;
            bool gave_up = false;
            const uint32_t before = chain_tiles(a.tile_state, tile, tag, (uint32_t)a.hdr->ent_base[a.hop], total, kChainPolls, &gave_up);
            if (gave_up) atomicOr(&a.hdr->status, ST_INTERNAL);
            if (lane == 0) {
                const uint32_t end = before + total;
                sh_before = before;
                sh_end = end;
                if ((int64_t)end > a.cap_entries) atomicOr(&a.hdr->status, ST_CAP_ENTRIES);
                else if (tile == n_tiles - 1) {
                    a.hdr->ent_base[a.hop + 1] = (int32_t)end;
                    a.ent_off[lo + n] = (int32_t)end;   // (past the hop's own nodes: the sentinel)
                }
            }
        }
        __syncthreads();
        const bool fits = (int64_t)sh_end <= a.cap_entries;
#pragma unroll
        for (int q = 0; q < kTileSets; ++q) {
            const int32_t t = q * kThreads + (int32_t)threadIdx.x, local = tile * tile_nodes + t;
            if (q >= sets || t >= n_here) break;
            const uint32_t out0 = sh_before + part[q * (kThreads / 32) + warp] + inc[q] - node_out[t];
            node_out[t] = out0;
            a.ent_off[lo + local] = (int32_t)out0;
            if (a.hop == 0) {
                const int32_t v = node_id[t], b = node_b[t];
                a.nodes[local] = v;
                a.node_batch[local] = b;
                if (v < 0 || (int64_t)v >= a.n_nodes) atomicOr(&a.hdr->status, ST_RANGE);
                else if (!feat_resident(a.feat, v)) atomicOr(&a.hdr->status, ST_NONRESIDENT);
                else {
                    bool is_new;
                    const int32_t slot = table_insert(a.hkeys + (int64_t)b * a.tg.size, a.tg.size, v, &is_new);
                    if (slot < 0) atomicOr(&a.hdr->status, ST_CAP_TABLE);
                    else if (!is_new) atomicOr(&a.hdr->status, ST_DUPLICATE);
                    else a.hvals[(int64_t)b * a.tg.size + slot] = local - a.tgt_off[b];
                }
            }
        }
        if (!fits) break;   // (uniform over the block)
        __syncthreads();
        if constexpr (THREAD) {
            // a thread per node: a Philox call gives four draws, and all picks of a node are looked up together.  The warp's entries are
            // put one behind the other in shared memory and written from there.
            uint32_t* out = reinterpret_cast<uint32_t*>(node_out + a.tile_cap) + (size_t)warp * 32 * f * (inout ? 2 : 1);
#pragma unroll 1
            for (int t0 = warp * 32; t0 < n_here; t0 += kThreads) {
                const int t = min(t0 + lane, n_here - 1);
                const bool on = t0 + lane < n_here;
                const uint32_t g0 = node_out[t], base = __shfl_sync(0xFFFFFFFFu, g0, 0);
                const int32_t gb = node_b[t];
                uint32_t at = g0 - base;
#pragma unroll 1
                for (int dir = 0; dir < (inout ? 2 : 1); ++dir) {   // (the second direction's picks follow the first's)
                    const uint32_t d = on ? node_deg[dir * a.tile_cap + t] : 0u, cnt = min(d, (uint32_t)f);
                    const int32_t* __restrict__ row = a.row_nbrs[dir] + node_r0[dir * a.tile_cap + t];
                    uint32_t pick[G];
                    if (d > (uint32_t)f) floyd_thread<G>(d, f, a.seeds[gb], (uint32_t)node_id[t], (uint32_t)a.hop, dir ? (uint32_t)MG_OUT_SLOT_BASE : 0u, pick);
                    else {   // all neighbours, in row order
#pragma unroll
                        for (int j = 0; j < G; ++j) pick[j] = (uint32_t)j;
                    }
#pragma unroll
                    for (int j = 0; j < G; ++j) if ((uint32_t)j < cnt) pick[j] = (uint32_t)__ldg(row + pick[j]);
#pragma unroll
                    for (int j = 0; j < G; ++j) if ((uint32_t)j < cnt) out[at + j] = pick[j];
                    at += cnt;
                }
                const uint32_t total = __reduce_max_sync(0xFFFFFFFFu, on ? at : 0u);
                __syncwarp();
                for (uint32_t i = lane; i < total; i += 32) a.ent_nbrs[base + i] = (int32_t)out[i];
                if (a.batch_of_entry) {
                    const int32_t b0 = __shfl_sync(0xFFFFFFFFu, gb, 0);
                    if (__all_sync(0xFFFFFFFFu, gb == b0)) {
                        for (uint32_t i = lane; i < total; i += 32) a.ent_repr[base + i] = b0;
                    } else {
                        __syncwarp();
                        if (on) for (uint32_t i = g0 - base; i < at; ++i) out[i] = (uint32_t)gb;
                        __syncwarp();
                        for (uint32_t i = lane; i < total; i += 32) a.ent_repr[base + i] = (int32_t)out[i];
                    }
                }
                __syncwarp();
            }
        } else
        // the picks: warp after warp takes nodes of the tile
        for (int dir = 0; dir < (inout ? 2 : 1); ++dir) {
            const int32_t* __restrict__ row_nbrs = a.row_nbrs[dir];
            const uint32_t slot_base = dir ? (uint32_t)MG_OUT_SLOT_BASE : 0u;
            const int64_t* dir_r0 = node_r0 + dir * a.tile_cap;
            const uint32_t* dir_deg = node_deg + dir * a.tile_cap;
            if (G > 0) {
                constexpr int GG = G > 0 ? G : 1, kPerWarp = 32 / GG;
                const int grp = lane / GG;                // group inside the warp (== kPerWarp: a left-over lane)
                const int gl = lane - grp * GG;           // lane inside the group
                for (int s = warp * kPerWarp; s < n_here; s += (kThreads / 32) * kPerWarp) {
                    const bool on = grp < kPerWarp && s + grp < n_here;
                    const int at = min(s + grp, n_here - 1);
                    const int32_t gb = node_b[at];
                    const int64_t gr0 = dir_r0[at];
                    const uint32_t gd = on ? dir_deg[at] : 0u;
                    // (the second direction's picks follow the first's)
                    const uint32_t g0 = node_out[at] + (dir ? min(node_deg[at], (uint32_t)f) : 0u);
                    const bool floyd = gd > (uint32_t)f;
                    uint32_t p = (uint32_t)gl;            // all neighbours, in row order
                    int rank = gl;
                    if (__any_sync(0xFFFFFFFFu, floyd)) {
                        int r;
                        const uint32_t fp = floyd_pick<GG>(floyd, gd, f, gl, grp * GG, floyd ? a.seeds[gb] : 0ull, (uint32_t)node_id[at],
                                                           (uint32_t)a.hop, slot_base, &r);
                        if (floyd) { p = fp; rank = r; }
                    }
                    if (floyd ? gl < f : (uint32_t)gl < gd) {
                        a.ent_nbrs[g0 + rank] = row_nbrs[gr0 + (int64_t)p];
                        a.ent_repr[g0 + rank] = gb;
                    }
                }
            } else {
                uint32_t* xs = reinterpret_cast<uint32_t*>(node_out + a.tile_cap) + (size_t)warp * 2 * f;
                uint32_t* picks = xs + f;
                for (int s = warp; s < n_here; s += kThreads / 32) {
                    const uint32_t gv = (uint32_t)node_id[s];
                    const int32_t gb = node_b[s];
                    const int64_t gr0 = dir_r0[s];
                    const uint32_t gd = dir_deg[s];
                    const uint32_t g0 = node_out[s] + (dir ? min(node_deg[s], (uint32_t)f) : 0u);
                    const bool floyd = gd > (uint32_t)f;   // (uniform over the warp)
                    if (floyd) {
                        for (int t = lane; t < f; t += 32) {
                            const uint32_t jt = gd - (uint32_t)f + (uint32_t)t;
                            xs[t] = __umulhi(draw_word(a.seeds[gb], gv, (uint32_t)a.hop, slot_base + (uint32_t)t), jt + 1u);
                        }
                        __syncwarp();
                        for (int t = 0; t < f; ++t) {
                            const uint32_t xt = xs[t];
                            bool hit = false;
                            for (int q = lane; q < t; q += 32) hit |= (picks[q] == xt);
                            const bool any = __any_sync(0xFFFFFFFFu, hit);
                            if (lane == 0) picks[t] = any ? (gd - (uint32_t)f + (uint32_t)t) : xt;
                            __syncwarp();
                        }
                    }
                    const int32_t take = (int32_t)min(gd, (uint32_t)f);
                    for (int t = lane; t < take; t += 32) {
                        uint32_t p = (uint32_t)t;
                        int rank = t;
                        if (floyd) {
                            p = picks[t];
                            rank = 0;
                            for (int q = 0; q < f; ++q) rank += (picks[q] < p) ? 1 : 0;
                        }
                        a.ent_nbrs[g0 + rank] = row_nbrs[gr0 + (int64_t)p];
                        a.ent_repr[g0 + rank] = gb;
                    }
                    __syncwarp();
                }
            }
        }
        if (n_tiles <= (int32_t)gridDim.x) break;   // a tile for every block: nothing is left to take
    }
}

// Deduplication: every entry's neighbour id goes into its batch's id table.  One thread owns PER entries; their
// compare-and-swaps go out back to back and the probes of those that met another id go on in rounds, all open entries of the
// thread at a time.  Bound by the rounds a block needs for its longest probe, one L2 round trip each (reads of four or eight
// slots in place of the next compare-and-swap made it slower: 134 -> 160 us for the inner hops of 128 mini-batches, 292 -> 339 us
// for 12.6M entries of 16 large ones), so small tables are kept sparse (mg_sample_many), and by the counter of the mini-batch
// that all blocks in flight add to.
struct InsertArgs {
    DenseHeader* hdr;
    int hop;
    const int32_t* ent_nbrs;
    int32_t* ent_repr;   // in: batch id; out: the node's row (new node) or -1 - (batch * table_size + slot)
    int32_t* hkeys;
    TableGeom tg;
    int32_t* new_ids;            // [cap_entries] a mini-batch's new ids, from its first entry's place on
    int32_t B, k;
    const int32_t* node_off;     // [hop + 1][B + 1] valid
    const int32_t* ent_off;
    const int32_t* cum;          // [B][k+2]
    int32_t* hvals;
    uint32_t* batch_cnt;         // [B] new nodes of the hop per mini-batch, zero before the launch
    int32_t max_nodes_per_batch;
};

constexpr int kInsertThreads = 128, kInsertBlocks = 12;   // per SM
constexpr int kInsertPerThread = 4;
constexpr int kInsertSpan = 16;   // mini-batches a block's chunk of entries may touch on the fast path

// New nodes are not sorted on the device: nothing the path computes depends on the order of ids inside a delta (the
// paper's arrays, with ascending ids, are an export: mg_dense_batch_perm).  A new node takes the next free row of its
// mini-batch right here -- one global atomic per (block, mini-batch) --, its table value is written at once, and its id goes to
// its rank in the mini-batch's run of new_ids (a mini-batch has no more new nodes than entries, so the run starts where its
// entries do and no second counter is needed: with one list of (mini-batch, id, rank) for all, which wants a counter for its
// length, 16 mini-batches of 790,000 entries took 284 us instead of 254, and 128 of 29,000 119 instead of 95).
template <int PER>
__global__ void __launch_bounds__(kInsertThreads, kInsertBlocks) k_insert(InsertArgs a) {
    constexpr int kWarps = kInsertThreads / 32, kChunk = kInsertThreads * PER;
    __shared__ uint32_t warp_tot[kWarps];
    __shared__ uint32_t span_cnt[kInsertSpan], span_base[kInsertSpan];
    __shared__ int32_t span_row[kInsertSpan];   // first row of the hop's new nodes in the mini-batch
    __shared__ int32_t span_list[kInsertSpan];  // its run of new_ids
    __shared__ int32_t first_batch, last_batch;
    const int32_t lo = a.hdr->ent_base[a.hop], hi = a.hdr->ent_base[a.hop + 1];
    if (__syncthreads_or(a.hdr->status != 0)) return;   // (the whole block: another one may be setting it)
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    auto row_of = [&](int32_t batch) { return a.cum[batch * (a.k + 2) + a.hop + 1]; };
    auto list_of = [&](int32_t batch) { return a.ent_off[a.node_off[a.hop * (a.B + 1) + batch]]; };
    for (int32_t base = lo + blockIdx.x * kChunk; base < hi; base += gridDim.x * kChunk) {
        int32_t u[PER], b[PER], old[PER];
        uint32_t slot[PER], rank[PER];
        uint32_t open = 0, new_bits = 0;
#pragma unroll
        for (int j = 0; j < PER; ++j) {
            const int32_t e = base + j * kInsertThreads + threadIdx.x;
            u[j] = -1; b[j] = 0; old[j] = -1; slot[j] = 0;
            if (e < hi) { u[j] = a.ent_nbrs[e]; b[j] = a.ent_repr[e]; }
        }
        if (threadIdx.x == 0) first_batch = b[0];   // thread 0's first item is the chunk's first entry
        if (threadIdx.x == 32) last_batch = a.ent_repr[min(hi - base, kChunk) - 1 + base];
        if (threadIdx.x < kInsertSpan) span_cnt[threadIdx.x] = 0;
        __syncthreads();
        const int32_t b0 = first_batch;   // entries are ordered by mini-batch, so a chunk touches a short run of them
        const bool one_batch = b0 == last_batch;
        const int span = (int)threadIdx.x - 32;   // threads 32..47: a mini-batch of the run each
        int32_t my_row = 0, my_list = 0;
        if (span >= 0 && span < (one_batch ? 1 : kInsertSpan) && b0 + span < a.B) { my_row = row_of(b0 + span); my_list = list_of(b0 + span); }
#pragma unroll
        for (int j = 0; j < PER; ++j)
            if (u[j] >= 0) {
                slot[j] = table_hash(u[j], a.tg.size);
                old[j] = atomicCAS(&a.hkeys[(int64_t)b[j] * a.tg.size + slot[j]], -1, u[j]);
            }
#pragma unroll
        for (int j = 0; j < PER; ++j) {
            if (u[j] < 0) continue;
            if (old[j] == -1) new_bits |= 1u << j;
            else if (old[j] != u[j]) open |= 1u << j;
        }
        for (int32_t probe = 1; open; ++probe) {   // linear probing
            if (probe >= a.tg.size) { atomicOr(&a.hdr->status, ST_CAP_TABLE); break; }
#pragma unroll
            for (int j = 0; j < PER; ++j)
                if (open >> j & 1) {
                    slot[j] = slot[j] + 1u == (uint32_t)a.tg.size ? 0u : slot[j] + 1u;
                    old[j] = atomicCAS(&a.hkeys[(int64_t)b[j] * a.tg.size + slot[j]], -1, u[j]);
                }
#pragma unroll
            for (int j = 0; j < PER; ++j)
                if (open >> j & 1) {
                    if (old[j] == -1) new_bits |= 1u << j;
                    if (old[j] == -1 || old[j] == u[j]) open &= ~(1u << j);
                }
        }
        __syncwarp();
        uint32_t in_warp = 0;
#pragma unroll
        for (int j = 0; j < PER; ++j) {
            const bool fresh = new_bits >> j & 1;
            // an entry that found its node already in the table gets the node's row later (k_place): it leaves
            // -1 - (table index) behind; the entry of a new node gets its row below
            if (!fresh && u[j] >= 0) a.ent_repr[base + j * kInsertThreads + threadIdx.x] = -1 - (b[j] * a.tg.size + (int32_t)slot[j]);
            rank[j] = 0;
            if (one_batch) {
                const uint32_t ballot = __ballot_sync(0xFFFFFFFFu, fresh);
                rank[j] = in_warp + __popc(ballot & ((1u << lane) - 1u));
                in_warp += __popc(ballot);
            } else if (fresh) {
                const int32_t bb = b[j] - b0;
                rank[j] = bb < kInsertSpan ? atomicAdd(&span_cnt[bb], 1u) : atomicAdd(&a.batch_cnt[b[j]], 1u);
            }
        }
        if (lane == 0) warp_tot[warp] = in_warp;
        if (span >= 0 && span < kInsertSpan) { span_row[span] = my_row; span_list[span] = my_list; }
        __syncthreads();
        if (threadIdx.x < kInsertSpan) {   // the block's run of its mini-batches' rows: one round trip
            uint32_t c = span_cnt[threadIdx.x];
            if (one_batch) {
                c = 0;
                if (threadIdx.x == 0)
                    for (int w = 0; w < kWarps; ++w) c += warp_tot[w];
            }
            if (c) span_base[threadIdx.x] = atomicAdd(&a.batch_cnt[b0 + (int)threadIdx.x], c);
        }
        __syncthreads();
        uint32_t before = 0;
        if (one_batch)
            for (int w = 0; w < warp; ++w) before += warp_tot[w];
#pragma unroll
        for (int j = 0; j < PER; ++j)
            if (new_bits >> j & 1) {
                const int32_t bb = b[j] - b0;
                const bool near = bb < kInsertSpan;
                rank[j] += near ? before + span_base[bb] : 0u;
                const int64_t row = (int64_t)(near ? span_row[bb] : row_of(b[j])) + rank[j];
                if (row < a.max_nodes_per_batch) a.hvals[(int64_t)b[j] * a.tg.size + slot[j]] = (int32_t)row;
                else atomicOr(&a.hdr->status, ST_CAP_TABLE);
                a.ent_repr[base + j * kInsertThreads + threadIdx.x] = (int32_t)row;   // final: no table read for this entry
                a.new_ids[(int64_t)(near ? span_list[bb] : list_of(b[j])) + rank[j]] = u[j];
            }
        __syncthreads();
    }
}

// -------------------------------------------------------------------------------------
// Last hop: deduplication in shared memory
// -------------------------------------------------------------------------------------
// The last hop has most of the entries (12.9M of 16.6M on the bench) and its new nodes are never looked up again, so
// it does not go through the id tables in global memory.  The ids of a mini-batch are split by hash into nb buckets.
// k_bucket_entries: block (mini-batch, r) takes the r-th share of the mini-batch's entries and the r-th share of the
// nodes it already has (hops 0..hop) and writes both grouped by bucket (a counting sort inside the block): (id, entry)
// pairs and (id, row) pairs, with the groups' bounds.
// k_dedupe_last: block (mini-batch, bucket) holds the bucket's id table (keys and rows, S slots) in shared memory.  It
// enters its bucket's earlier nodes, then its bucket's entries from every share (dense), ranks its new nodes (a scan over
// the table, no atomics), takes a run of the mini-batch's rows and of the list of new nodes with ONE global atomic
// each, and gives every entry its node's row.
// Both are bound by instruction issue and shared-memory round trips, so the number of buckets follows from how evenly the
// blocks fill the SMs (dedup_buckets): 4 blocks for one mini-batch of 53,000 nodes left 144 SMs idle (25 + 52 us against 6 + 17
// with 64), 37 mini-batches of 63,000 nodes go from 84 + 29 to 68 + 22 us, 128 of 95,000 from 285 to 273 us.
constexpr int kDedupMaxSlots = 26624;    // 208 KiB of keys + rows per block
constexpr int kDedupMaxBuckets = 64;
constexpr int kDedupMaxTables = 16;      // largest tables that a mini-batch may need
constexpr int64_t kDedupMinNodes = 1 << 20;   // room for nodes of all mini-batches up to which the global tables are the faster way
constexpr int kBucketThreads = 512;
constexpr int kDedupSlots512 = 6656, kDedupSlots256 = 3328;   // tables up to this size: blocks of 512 / 256 threads

struct DedupArgs {
    DenseHeader* hdr;
    int hop;
    int32_t B, k, nb, S;
    const int32_t* nodes;
    const int32_t* node_off;    // [hop + 1][B + 1] valid
    const int32_t* ent_off;
    const int32_t* ent_nbrs;
    int32_t* ent_repr;
    int2* pairs;                // [entries of the hop] (id, entry), grouped by (mini-batch, share, bucket); from
                                // node_pairs0 on: (id, row) of the earlier nodes, grouped the same way
    int32_t* share_off;         // [2][B][nb][nb + 1] group bounds (positions in pairs): entries, then earlier nodes
    const int32_t* cum;         // [B][k + 2]
    uint32_t* batch_cnt;        // [B] new nodes of the hop per mini-batch, zero before the launch
    int32_t* new_ids;           // [cap_entries] a mini-batch's new ids, from its first entry's place on
    int32_t max_nodes_per_batch;
    int64_t node_pairs0;
};

// Buckets per mini-batch: work of the SM with the most blocks, in mini-batches, plus 0.004 of one for every block's fixed cost
// (at least min_nb, so that a bucket's table fits a block; at most 64, and no buckets of fewer than 256 nodes).
int dedup_buckets(int64_t B, int64_t cap_batch, int64_t min_nb, int n_sms) {
    const int64_t max_nb = std::max<int64_t>(min_nb, std::min<int64_t>(kDedupMaxBuckets, cap_batch / 256));
    int64_t best = min_nb;
    double best_cost = 1e30;
    for (int64_t nb = min_nb; nb <= max_nb; ++nb) {
        const double per_sm = (double)((B * nb + n_sms - 1) / n_sms);
        const double cost = per_sm / (double)nb + 0.004 * per_sm;
        if (cost < best_cost - 1e-9) { best_cost = cost; best = nb; }
    }
    return (int)best;
}

// slots of a bucket's table: its share of the nodes plus a twelfth plus eight standard deviations of how a hash fills buckets
int64_t dedup_slots_for(int64_t nodes) {
    return ((nodes * 13 + 11) / 12 + 8 * (int64_t)std::sqrt((double)nodes) + 64 + 127) / 128 * 128;
}

// Bucket and first slot of an id: one hash, the bucket from its top, the slot from what is left.  (A multiplication alone puts
// the multiples of some strides next to each other -- a table for one bucket of 64 would overflow where one of seven did not
// --, so its upper half is folded into the lower and multiplied again.)
__device__ __forceinline__ uint32_t dedup_hash(int32_t id) {
    uint32_t h = (uint32_t)id * 0x9E3779B1u;
    h ^= h >> 16;
    return h * 0x85EBCA6Bu;
}
__device__ __forceinline__ uint32_t dedup_bucket(int32_t id, uint32_t nb) { return __umulhi(dedup_hash(id), nb); }
__device__ __forceinline__ uint32_t dedup_slot(int32_t id, uint32_t nb, uint32_t S) { return __umulhi(dedup_hash(id) * nb, S); }

__global__ void __launch_bounds__(kBucketThreads) k_bucket_entries(DedupArgs a) {
    constexpr int kWarps = kBucketThreads / 32;
    __shared__ uint32_t cnt[kWarps][kDedupMaxBuckets];
    __shared__ uint32_t base[kDedupMaxBuckets + 1];
    __shared__ int32_t hop_lo[MG_MAX_HOPS + 1], hop_row0[MG_MAX_HOPS + 2];
    if (__syncthreads_or(a.hdr->status != 0)) return;   // (the whole block: another one may be setting it)
    const uint32_t nb = (uint32_t)a.nb;
    const int32_t b = (int32_t)(blockIdx.x / nb);
    const uint32_t r = blockIdx.x % nb;
    const int warp = threadIdx.x >> 5;
    if (threadIdx.x <= (unsigned)a.hop) hop_lo[threadIdx.x] = a.node_off[threadIdx.x * (a.B + 1) + b];
    if (threadIdx.x <= (unsigned)a.hop + 1) hop_row0[threadIdx.x] = a.cum[b * (a.k + 2) + threadIdx.x];
    __syncthreads();
    // pass 0: the entries of the hop; pass 1: the nodes the mini-batch already has, item t = the node of row t
    for (int pass = 0; pass < 2; ++pass) {
        int64_t first, last, out0;
        if (pass == 0) {
            first = a.ent_off[a.node_off[a.hop * (a.B + 1) + b]];
            last = a.ent_off[a.node_off[a.hop * (a.B + 1) + b + 1]];
            out0 = first;
        } else {
            first = 0;
            last = hop_row0[a.hop + 1];
            out0 = a.node_pairs0;   // this mini-batch's node pairs follow those of the mini-batches before it
            for (int j = 0; j <= a.hop; ++j) out0 += hop_lo[j] - a.node_off[j * (a.B + 1)];
        }
        const int32_t len = (int32_t)((last - first + nb - 1) / nb);
        const int32_t s_lo = (int32_t)min(last, first + (int64_t)r * len);
        const int32_t s_hi = (int32_t)min(last, (int64_t)s_lo + len);
        auto id_at = [&](int32_t i) -> int32_t {
            if (pass == 0) return a.ent_nbrs[i];
            int j = 0;
            while (j < a.hop && hop_row0[j + 1] <= i) ++j;
            return a.nodes[hop_lo[j] + (i - hop_row0[j])];
        };
        for (int i = threadIdx.x; i < kWarps * kDedupMaxBuckets; i += kBucketThreads) (&cnt[0][0])[i] = 0;
        __syncthreads();
        // (four loads in flight per thread: the walk is latency-bound otherwise)
        for (int32_t e0 = s_lo + (int32_t)threadIdx.x; e0 < s_hi; e0 += 4 * kBucketThreads) {
            int32_t id[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) id[u] = e0 + u * kBucketThreads < s_hi ? id_at(e0 + u * kBucketThreads) : -1;
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (e0 + u * kBucketThreads < s_hi) atomicAdd(&cnt[warp][dedup_bucket(id[u], nb)], 1u);
        }
        __syncthreads();
        if (threadIdx.x < nb) {   // this bucket's pairs of the share: warp after warp
            uint32_t run = 0;
            for (int w = 0; w < kWarps; ++w) { const uint32_t c = cnt[w][threadIdx.x]; cnt[w][threadIdx.x] = run; run += c; }
            base[threadIdx.x] = run;
        }
        __syncthreads();
        if (warp == 0) {   // (two buckets per lane)
            const uint32_t q0 = 2u * (threadIdx.x & 31), q1 = q0 + 1;
            const uint32_t c0 = q0 < nb ? base[q0] : 0u, c1 = q1 < nb ? base[q1] : 0u;
            const uint32_t before = warp_incl_scan(c0 + c1) - c0 - c1;
            __syncwarp();
            if (q0 <= nb) base[q0] = before;
            if (q1 <= nb) base[q1] = before + c0;
            if (q1 + 1 == nb) base[nb] = before + c0 + c1;
        }
        __syncthreads();
        const int64_t dst0 = out0 + (s_lo - first);
        if (threadIdx.x <= nb)
            a.share_off[(((int64_t)pass * a.B + b) * nb + r) * (nb + 1) + threadIdx.x] = (int32_t)(dst0 + base[threadIdx.x]);
        for (int32_t e0 = s_lo + (int32_t)threadIdx.x; e0 < s_hi; e0 += 4 * kBucketThreads) {
            int32_t id[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) id[u] = e0 + u * kBucketThreads < s_hi ? id_at(e0 + u * kBucketThreads) : -1;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int32_t e = e0 + u * kBucketThreads;
                if (e >= s_hi) continue;
                const uint32_t q = dedup_bucket(id[u], nb);
                a.pairs[dst0 + base[q] + atomicAdd(&cnt[warp][q], 1u)] = make_int2(id[u], e);
            }
        }
        __syncthreads();
    }
}

// (1,024 threads: 32 registers, a few of them spilled, for two blocks per SM where tables leave room for them: 64 mini-batches of 47,000 nodes in half as much room
// again 76.3 -> 63.1 us; where they don't, 128 of 96,000 254 -> 258)
template <int kDedupThreads>
__global__ void __launch_bounds__(kDedupThreads, kDedupThreads == 1024 ? 2 : 1536 / kDedupThreads) k_dedupe_last(DedupArgs a) {
    extern __shared__ int32_t dedup_sm[];
    __shared__ uint32_t row_base, warp_tot[kDedupThreads / 32];
    __shared__ int32_t run_lo[2][kDedupMaxBuckets], run_start[2][kDedupMaxBuckets + 1];
    if (__syncthreads_or(a.hdr->status != 0)) return;   // (the whole block: another one may be setting it)
    const uint32_t nb = (uint32_t)a.nb;
    const int32_t b = (int32_t)(blockIdx.x / nb);
    const uint32_t bucket = blockIdx.x % nb;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x < 2 * nb) {   // this bucket's runs of pairs, one per share: entries [0], earlier nodes [1] ...
        const uint32_t which = threadIdx.x / nb, r = threadIdx.x % nb;
        const int32_t* so = a.share_off + (((int64_t)which * a.B + b) * nb + r) * (nb + 1) + bucket;
        run_lo[which][r] = so[0];
        run_start[which][r + 1] = so[1] - so[0];
    }
    __syncthreads();
    if (warp < 2) {   // ... and their lengths' prefix (two shares per lane)
        int32_t* rs = run_start[warp];
        const uint32_t r0 = 2u * lane, r1 = r0 + 1;
        const uint32_t c0 = r0 < nb ? (uint32_t)rs[r0 + 1] : 0u, c1 = r1 < nb ? (uint32_t)rs[r1 + 1] : 0u;
        const uint32_t end = warp_incl_scan(c0 + c1);
        __syncwarp();
        if (r0 < nb) rs[r0 + 1] = (int32_t)(end - c1);
        if (r1 < nb) rs[r1 + 1] = (int32_t)end;
        if (lane == 0) rs[0] = 0;
    }
    __syncthreads();
    // the table: half as many slots again as there can be ids, no more than there is room for.  (As many as there is room for are cleared and looked through
    // for nothing where callers leave much of it: 37 mini-batches in four times the room they take 85.6 -> 78.9 us, 32 larger ones 104 -> 94.5, 128 303 -> 289; in half as
    // much again as they take, as before.)
    const uint32_t ids = (uint32_t)run_start[0][nb] + (uint32_t)run_start[1][nb];
    const uint32_t S = min((uint32_t)a.S, ids + ids / 2 + 32u);
    int32_t* keys = dedup_sm;
    int32_t* vals = dedup_sm + S;
    for (uint32_t i = threadIdx.x; i < S; i += kDedupThreads) keys[i] = -1;
    __syncthreads();
    auto pair_at = [&](int which, int32_t i) -> int2* {   // i-th pair of the bucket: which share's run it falls in (run_start ascends)
        uint32_t lo = 0, hi = nb;                           // run_start[lo] <= i < run_start[hi]
        while (hi - lo > 1) {
            const uint32_t mid = (lo + hi) >> 1;
            if (run_start[which][mid] <= i) lo = mid; else hi = mid;
        }
        return a.pairs + run_lo[which][lo] + (i - run_start[which][lo]);
    };
    // the nodes the mini-batch already has (this bucket's): rows = positions
    {
        const int32_t n_old = run_start[1][nb];
        for (int32_t i0 = threadIdx.x; i0 < n_old; i0 += 4 * kDedupThreads) {
            int2 it[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) it[u] = *pair_at(1, min(i0 + u * kDedupThreads, n_old - 1));
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (i0 + u * kDedupThreads >= n_old) continue;
                const int32_t id = it[u].x;
                uint32_t s = dedup_slot(id, nb, S), probe = 0;
                for (; probe < S; ++probe) {
                    const int32_t old = atomicCAS(&keys[s], -1, id);
                    if (old == -1) { vals[s] = it[u].y; break; }
                    if (old == id) { atomicOr(&a.hdr->status, ST_DUPLICATE); break; }   // only targets can repeat
                    s = s + 1u == S ? 0u : s + 1u;
                }
                if (probe >= S) atomicOr(&a.hdr->status, ST_CAP_TABLE);
            }
        }
    }
    __syncthreads();
    // this bucket's entries: enter the id, leave its slot in place of the id
    const int32_t n_pairs = run_start[0][nb];
    for (int32_t i0 = threadIdx.x; i0 < n_pairs; i0 += 4 * kDedupThreads) {
        int2* pp[4];
        int32_t id[4], old[4];
        uint32_t s[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {   // four loads, then four first-probe compare-and-swaps, in flight per thread
            const int32_t i = i0 + u * kDedupThreads;
            pp[u] = pair_at(0, min(i, n_pairs - 1));
            id[u] = i < n_pairs ? pp[u]->x : -1;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            s[u] = dedup_slot(id[u], nb, S);
            old[u] = id[u] >= 0 ? atomicCAS(&keys[s[u]], -1, id[u]) : id[u];
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (id[u] < 0) continue;
            bool fresh = old[u] == -1;
            if (!fresh && old[u] != id[u]) {   // first slot taken by another id: linear probing
                uint32_t probe = 1;
                for (; probe < S; ++probe) {
                    s[u] = s[u] + 1u == S ? 0u : s[u] + 1u;
                    const int32_t o = atomicCAS(&keys[s[u]], -1, id[u]);
                    if (o == -1) { fresh = true; break; }
                    if (o == id[u]) break;
                }
                if (probe >= S) { atomicOr(&a.hdr->status, ST_CAP_TABLE); s[u] = 0; fresh = false; }
            }
            if (fresh) vals[s[u]] = -1;   // new: ranked below
            pp[u]->x = (int32_t)s[u];
        }
    }
    __syncthreads();
    // rank the new nodes of this block's table, take a run of the mini-batch's rows
    uint32_t mine = 0;
    for (uint32_t i = threadIdx.x; i < S; i += kDedupThreads) mine += (keys[i] != -1 && vals[i] < 0) ? 1u : 0u;
    const uint32_t inc = warp_incl_scan(mine);
    if (lane == 31) warp_tot[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        const uint32_t w = lane < kDedupThreads / 32 ? warp_tot[lane] : 0u;
        const uint32_t wi = warp_incl_scan(w);
        if (lane < kDedupThreads / 32) warp_tot[lane] = wi - w;
        if (lane == 31) row_base = wi ? atomicAdd(&a.batch_cnt[b], wi) : 0u;
    }
    __syncthreads();
    const int32_t first_row = a.cum[b * (a.k + 2) + a.hop + 1];
    int32_t* list = a.new_ids + a.ent_off[a.node_off[a.hop * (a.B + 1) + b]];
    uint32_t rk = warp_tot[warp] + inc - mine;
    for (uint32_t i = threadIdx.x; i < S; i += kDedupThreads) {
        if (keys[i] == -1 || vals[i] >= 0) continue;
        const uint32_t rank = row_base + rk;
        const int64_t row = (int64_t)first_row + rank;
        if (row >= a.max_nodes_per_batch) atomicOr(&a.hdr->status, ST_CAP_TABLE);
        vals[i] = (int32_t)row;
        list[rank] = keys[i];
        ++rk;
    }
    __syncthreads();
    // every entry of the bucket gets its node's row
    for (int32_t i0 = threadIdx.x; i0 < n_pairs; i0 += 4 * kDedupThreads) {
        int2 p[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) p[u] = *pair_at(0, min(i0 + u * kDedupThreads, n_pairs - 1));
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (i0 + u * kDedupThreads < n_pairs) a.ent_repr[p[u].y] = vals[p[u].x];
    }
}

// -------------------------------------------------------------------------------------
// radix sort of 64-bit keys on bits [lo_bit, lo_bit + bits), for the export of one mini-batch
// -------------------------------------------------------------------------------------
constexpr int kSortKeysPerThread = 16;
constexpr int kSortTile = kThreads * kSortKeysPerThread;  // 4096
constexpr int kRadixBits = 9;
constexpr int kBins = 1 << kRadixBits;
constexpr int kBinsPerThread = kBins / kThreads;

__global__ void __launch_bounds__(kThreads)
k_radix_hist(const uint64_t* __restrict__ keys, const SortParams* sp, int shift, uint32_t* hist) {
    __shared__ uint32_t sh[kBins];
    const int32_t n = sp->n, ntiles = sp->ntiles;
    for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
#pragma unroll
        for (int q = 0; q < kBinsPerThread; ++q) sh[threadIdx.x + q * kThreads] = 0;
        __syncthreads();
        const int32_t tb = t * kSortTile, tn = min(kSortTile, n - tb);
#pragma unroll 4
        for (int j = 0; j < kSortKeysPerThread; ++j) {
            const int32_t l = j * kThreads + threadIdx.x;
            if (l < tn) atomicAdd(&sh[(uint32_t)(keys[tb + l] >> shift) & (kBins - 1)], 1u);
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < kBinsPerThread; ++q) {
            const int bin = threadIdx.x + q * kThreads;
            hist[(size_t)t + (size_t)bin * ntiles] = sh[bin];
        }
        __syncthreads();
    }
}

// One stable counting pass.  A tile's keys are ranked per digit (warp by warp, 32 keys at a time with
// match_any), laid out digit by digit in shared memory, and written from there, so that every run of
// equal digits leaves the SM as consecutive addresses.
__global__ void __launch_bounds__(kThreads)
k_radix_scatter(const uint64_t* __restrict__ keys, uint64_t* __restrict__ out, const SortParams* sp, int shift,
                const uint32_t* __restrict__ hist_scanned) {
    extern __shared__ __align__(16) uint8_t sort_smem[];
    uint64_t* stage = reinterpret_cast<uint64_t*>(sort_smem);                          // [kSortTile]
    uint32_t (*cnt)[kBins] = reinterpret_cast<uint32_t (*)[kBins]>(stage + kSortTile);   // [warps][kBins]
    uint32_t* tile_base = reinterpret_cast<uint32_t*>(cnt + kThreads / 32);             // [kBins] first slot of a digit in the tile
    uint32_t* glob_base = tile_base + kBins;                                            // [kBins] first output position
    __shared__ uint32_t warp_tot[kThreads / 32];
    const int32_t n = sp->n, ntiles = sp->ntiles;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int kWarps = kThreads / 32;
    constexpr int kPerWarp = kSortTile / kWarps;  // 512 consecutive keys per warp
    for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
        for (int w = 0; w < kWarps; ++w)
#pragma unroll
            for (int q = 0; q < kBinsPerThread; ++q) cnt[w][threadIdx.x + q * kThreads] = 0;
        __syncthreads();
        uint64_t key[kSortKeysPerThread];
        uint32_t rank[kSortKeysPerThread];
        const int32_t tb = t * kSortTile, tile_n = min(kSortTile, n - tb);
        const int32_t wl = warp * kPerWarp;   // the warp's first key inside the tile
#pragma unroll
        for (int r = 0; r < kSortKeysPerThread; ++r) {
            const bool ok = wl + r * 32 + lane < tile_n;
            key[r] = ok ? keys[tb + wl + r * 32 + lane] : 0ull;
            const uint32_t dg = ok ? ((uint32_t)(key[r] >> shift) & (kBins - 1)) : 0xFFFFFFFFu;
            const uint32_t peers = __match_any_sync(0xFFFFFFFFu, dg);
            const int leader = __ffs(peers) - 1;
            uint32_t old = 0;
            if (ok && lane == leader) {
                old = cnt[warp][dg];
                cnt[warp][dg] = old + __popc(peers);
            }
            old = __shfl_sync(0xFFFFFFFFu, old, leader);
            rank[r] = old + __popc(peers & ((1u << lane) - 1u));
            __syncwarp();
        }
        __syncthreads();
        // per digit: prefix over the warps, total in the tile; then an exclusive scan over the digits
        uint32_t mine[kBinsPerThread], sum = 0;
#pragma unroll
        for (int q = 0; q < kBinsPerThread; ++q) {
            const int bin = threadIdx.x * kBinsPerThread + q;   // consecutive bins per thread: scan order = bin order
            uint32_t run = 0;
            for (int w = 0; w < kWarps; ++w) { const uint32_t c = cnt[w][bin]; cnt[w][bin] = run; run += c; }
            mine[q] = run;
            sum += run;
        }
        const uint32_t inc = warp_incl_scan(sum);
        if (lane == 31) warp_tot[warp] = inc;
        __syncthreads();
        uint32_t before = inc - sum;
        for (int w = 0; w < warp; ++w) before += warp_tot[w];
#pragma unroll
        for (int q = 0; q < kBinsPerThread; ++q) {
            const int bin = threadIdx.x * kBinsPerThread + q;
            tile_base[bin] = before;
            glob_base[bin] = hist_scanned[(size_t)t + (size_t)bin * ntiles];
            before += mine[q];
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < kSortKeysPerThread; ++r) {
            if (wl + r * 32 + lane < tile_n) {
                const uint32_t dg = (uint32_t)(key[r] >> shift) & (kBins - 1);
                stage[tile_base[dg] + cnt[warp][dg] + rank[r]] = key[r];
            }
        }
        __syncthreads();
        for (int32_t i = threadIdx.x; i < tile_n; i += kThreads) {
            const uint64_t kx = stage[i];
            const uint32_t dg = (uint32_t)(kx >> shift) & (kBins - 1);
            out[glob_base[dg] + ((uint32_t)i - tile_base[dg])] = kx;
        }
        __syncthreads();
    }
}

constexpr size_t kScatterSmem = (size_t)kSortTile * 8 + (size_t)(kThreads / 32) * kBins * 4 + 2 * (size_t)kBins * 4;

// -------------------------------------------------------------------------------------
// place the last hop's new nodes, give the entries their rows
// -------------------------------------------------------------------------------------
// The new nodes per mini-batch are summed up as in k_hop, and their runs of new ids put one behind the other (a warp takes 128 nodes at a
// time, four loads in flight per thread); an entry, of whatever hop, that met a known node -> that node's row (entries of new nodes got
// theirs at insert time; the shared-memory path of the last hop leaves none).  Block 0 writes the packed row bases of every layer and the
// per-batch entry bounds of every hop, and the sample's summary (header, per-batch tables) for the host, stored straight into mapped pinned
// memory.  A copy engine is not used on purpose: a large output copy of a forward pass may be queued on it, and the host would wait for
// that copy before it learned the sample's sizes.  (After an error the summary still goes out: it carries the status word.)
struct PlaceArgs {
    DenseHeader* hdr;
    const int32_t* new_ids;      // the last hop's new ids by rank, mini-batch b's from the place of its first entry on
    const uint32_t* batch_cnt;   // [B] new nodes of the last hop
    int64_t cap_nodes;
    int32_t* nodes;
    int32_t* node_batch;
    const int32_t* hvals;
    int32_t hops_in_table;       // hops whose entries went through the global tables: k, or k - 1
    int32_t node_limit;          // nodes that a mini-batch may have in all
    int32_t* ent_repr;
    int32_t B, k;
    int32_t* cum;
    int32_t* node_off;
    int32_t n_hdr;
    const int32_t* ent_off;
    int32_t* rowbase;
    int32_t* ent_hop;
    int32_t* out;                // n_hdr header words, cum, node_off, rowbase, ent_hop
};

__device__ __forceinline__ void finish_sample(const PlaceArgs& a, bool bad) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int32_t B = a.B, k = a.k;
    const int32_t n_cum = B * (k + 2), n_off = (k + 1) * (B + 1), n_ent = k * (B + 1);
    int32_t* o_cum = a.out + a.n_hdr;
    int32_t* o_off = o_cum + n_cum;
    int32_t* o_row = o_off + n_off;
    int32_t* o_ent = o_row + n_off;
    const volatile int32_t* h32 = reinterpret_cast<const volatile int32_t*>(a.hdr);
    for (int32_t i = threadIdx.x; i < a.n_hdr; i += blockDim.x) a.out[i] = h32[i];
    if (bad) return;
    for (int l = warp; l <= k; l += kThreads / 32) {   // a warp per layer: rows of the mini-batches, summed up
        uint32_t carry = 0;
        for (int s0 = 0; s0 < B; s0 += 32) {
            const int b = s0 + lane;
            const uint32_t v = b < B ? (uint32_t)a.cum[b * (k + 2) + (k - l + 1)] : 0u;
            const uint32_t inc = warp_incl_scan(v);
            if (b < B) {
                const int32_t r = (int32_t)(carry + inc - v);
                a.rowbase[l * (B + 1) + b] = r;
                o_row[l * (B + 1) + b] = r;
            }
            carry += __shfl_sync(0xFFFFFFFFu, inc, 31);
        }
        if (lane == 0) { a.rowbase[l * (B + 1) + B] = (int32_t)carry; o_row[l * (B + 1) + B] = (int32_t)carry; }
    }
    for (int32_t i = threadIdx.x; i < n_ent; i += blockDim.x) {   // (hop h = i / (B + 1), as in node_off)
        const int32_t e = a.ent_off[a.node_off[i]];
        a.ent_hop[i] = e;
        o_ent[i] = e;
    }
    for (int32_t i = threadIdx.x; i < n_cum; i += blockDim.x) o_cum[i] = a.cum[i];
    for (int32_t i = threadIdx.x; i < n_off; i += blockDim.x) o_off[i] = a.node_off[i];
}

constexpr int kPlacePerThread = 4;

__global__ void __launch_bounds__(kThreads, 8) k_place(PlaceArgs a) {
    extern __shared__ int32_t next_off[];   // [B] first node of the mini-batch among the new ones ...
    int32_t* list_at = next_off + a.B;      // ... and its run of new_ids
    __shared__ uint32_t part[kThreads / 32];
    const int lane = threadIdx.x & 31;
    const int32_t start = a.hdr->hop_base[a.k], hi = a.hdr->ent_base[a.hops_in_table];
    // (the whole block alike: block 0 may be adding to the status)
    bool bad = __syncthreads_or(a.hdr->status != 0);
    int64_t end = start;
    if (!bad) {
        end = sum_new_nodes({a.hdr, a.k, a.B, a.k, a.batch_cnt, a.cap_nodes, a.node_limit, a.ent_off, a.cum, a.node_off}, next_off, list_at, part);
        bad = end > a.cap_nodes;   // (nothing is written outside the arenas)
    }
    if (blockIdx.x == 0) { __syncthreads(); finish_sample(a, bad); return; }
    if (bad) return;
    const int32_t step = (int32_t)(gridDim.x - 1) * kThreads, tid = (int32_t)(blockIdx.x - 1) * kThreads + (int32_t)threadIdx.x;
    for (int64_t at0 = start + (int64_t)(tid >> 5) * (32 * kPlacePerThread); at0 < end; at0 += (int64_t)step * kPlacePerThread) {
        int32_t b = 0;   // the mini-batch of the warp's first node
        for (int32_t above = a.B; above - b > 1;) {
            const int32_t mid = (b + above) >> 1;
            if (next_off[mid] <= at0) b = mid; else above = mid;
        }
        int32_t id[kPlacePerThread], batch[kPlacePerThread];
#pragma unroll
        for (int j = 0; j < kPlacePerThread; ++j) {
            const int64_t at = at0 + j * 32 + lane;
            if (at < end) {
                while (b + 1 < a.B && next_off[b + 1] <= at) ++b;
                id[j] = a.new_ids[list_at[b] + (int32_t)(at - next_off[b])];
                batch[j] = b;
            }
        }
#pragma unroll
        for (int j = 0; j < kPlacePerThread; ++j) {
            const int64_t at = at0 + j * 32 + lane;
            if (at < end) { a.nodes[at] = id[j]; a.node_batch[at] = batch[j]; }
        }
    }
    for (int64_t e0 = tid; e0 < hi; e0 += (int64_t)step * kPlacePerThread) {
        int32_t v[kPlacePerThread];
#pragma unroll
        for (int j = 0; j < kPlacePerThread; ++j) { const int64_t e = e0 + (int64_t)j * step; v[j] = e < hi ? a.ent_repr[e] : 0; }
#pragma unroll
        for (int j = 0; j < kPlacePerThread; ++j) if (v[j] < 0) a.ent_repr[e0 + (int64_t)j * step] = a.hvals[-1 - v[j]];
    }
}

// -------------------------------------------------------------------------------------
// export to the paper's layout (mg_dense_view)
// -------------------------------------------------------------------------------------
// The device keeps every delta in discovery order.  The paper's arrays list the ids of a delta in ascending order
// (targets in the caller's order), so an export goes through a permutation of the mini-batch's local rows:
// perm[c] = local row of canonical row c, inv[l] = canonical row of local row l.
struct BatchGeom {
    int32_t k, V, n_targets;
    int32_t cum[MG_MAX_HOPS + 2];      // local row base per hop
    int32_t node_off[MG_MAX_HOPS + 1]; // first node of the mini-batch's run in each hop
};

__device__ __forceinline__ int hop_of_row(const BatchGeom& g, int32_t l) {
    int h = 0;
    while (h < g.k && l >= g.cum[h + 1]) ++h;
    return h;
}

// keys (canonical delta, id, local row) of the rows of hops >= 1
__global__ void __launch_bounds__(kThreads)
k_perm_keys(BatchGeom g, const int32_t* __restrict__ nodes, int id_bits, uint64_t* keys) {
    const int32_t n = g.V - g.n_targets;
    for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int32_t l = g.n_targets + i;
        const int h = hop_of_row(g, l);
        const int32_t id = nodes[g.node_off[h] + (l - g.cum[h])];
        keys[i] = ((uint64_t)(g.k - h) << (MG_SLOT_BITS + id_bits)) | ((uint64_t)(uint32_t)id << MG_SLOT_BITS) | (uint64_t)l;
    }
}

__global__ void __launch_bounds__(kThreads)
k_perm_fill(BatchGeom g, const uint64_t* __restrict__ sorted, int32_t* perm, int32_t* inv) {
    const int32_t n = g.V - g.n_targets;
    for (int32_t c = blockIdx.x * blockDim.x + threadIdx.x; c < g.V; c += gridDim.x * blockDim.x) {
        // deltas k-1 .. 0 (hops >= 1) come first in the sorted keys; the targets keep the caller's order at the end
        const int32_t l = c < n ? (int32_t)(sorted[c] & ((1u << MG_SLOT_BITS) - 1u)) : c - n;
        perm[c] = l;
        inv[l] = c;
    }
}

struct ExportArgs {
    BatchGeom g;
    int32_t n0;                       // |Delta_0|: canonical rows below n0 have no sampled neighbours
    int32_t nio[MG_MAX_HOPS + 2];     // canonical node_id_offsets
    const int32_t *nodes, *ent_off, *ent_nbrs, *ent_repr, *perm, *inv;
    int32_t *o_node_ids, *o_nio, *o_nbrs, *o_nbr_off, *o_repr;
};

// node ids in canonical order; the sampled nodes' entry counts go to o_nbr_off (scanned next)
__global__ void __launch_bounds__(kThreads) k_export_nodes(ExportArgs a) {
    const int32_t tid = blockIdx.x * blockDim.x + threadIdx.x;
    if (tid <= a.g.k + 1) a.o_nio[tid] = a.nio[tid];
    for (int32_t c = tid; c < a.g.V; c += gridDim.x * blockDim.x) {
        const int32_t l = a.perm[c];
        const int h = hop_of_row(a.g, l);
        const int32_t idx = a.g.node_off[h] + (l - a.g.cum[h]);
        a.o_node_ids[c] = a.nodes[idx];
        if (c >= a.n0) a.o_nbr_off[c - a.n0] = a.ent_off[idx + 1] - a.ent_off[idx];
    }
}

// in-place exclusive scan of data[0, n), total to data[n] (one block)
__global__ void __launch_bounds__(1024) k_export_scan(int32_t* data, int32_t n) {
    __shared__ uint32_t warp_tot[33];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t carry = 0;
    for (int s0 = 0; s0 < n; s0 += 1024) {
        const int i = s0 + threadIdx.x;
        const uint32_t v = i < n ? (uint32_t)data[i] : 0u;
        const uint32_t inc = warp_incl_scan(v);
        if (lane == 31) warp_tot[warp] = inc;
        __syncthreads();
        if (warp == 0) {
            const uint32_t w = warp_tot[lane];
            const uint32_t wi = warp_incl_scan(w);
            warp_tot[lane] = wi - w;
            if (lane == 31) warp_tot[32] = wi;
        }
        __syncthreads();
        if (i < n) data[i] = (int32_t)(carry + warp_tot[warp] + inc - v);
        carry += warp_tot[32];
        __syncthreads();
    }
    if (threadIdx.x == 0) data[n] = (int32_t)carry;
}

// nbrs and repr_map: the entries of canonical node c start at o_nbr_off[c - n0]
__global__ void __launch_bounds__(kThreads) k_export_entries(ExportArgs a) {
    for (int32_t c = a.n0 + blockIdx.x * blockDim.x + threadIdx.x; c < a.g.V; c += gridDim.x * blockDim.x) {
        const int32_t l = a.perm[c];
        const int h = hop_of_row(a.g, l);
        const int32_t idx = a.g.node_off[h] + (l - a.g.cum[h]);
        const int32_t e0 = a.ent_off[idx], e1 = a.ent_off[idx + 1];
        const int32_t o0 = a.o_nbr_off[c - a.n0];
        for (int32_t e = e0; e < e1; ++e) {
            a.o_nbrs[o0 + (e - e0)] = a.ent_nbrs[e];
            a.o_repr[o0 + (e - e0)] = a.inv[a.ent_repr[e]];
        }
    }
}

// -------------------------------------------------------------------------------------
// export of every mini-batch at once (mg_dense_export_many): the canonical DENSE ordering for the whole sample
// -------------------------------------------------------------------------------------
// A segment is a (mini-batch, delta) pair; in output order mini-batch follows mini-batch, inside it the farthest delta comes
// first.  Its ids are distinct, so a node's place in it is the number of smaller ids.  The ids are split by their top bits
// into bins -- counted per tile (k_export_count), written bin after bin in any order (k_export_split) --, and then ordered bin by bin
// (k_export_order): a warp compares the ids of a bin of up to 128 all with all, a block takes a larger one through bitmaps in
// shared memory, whose set bits below an id are its rank.  The same bins carry the sampled nodes' entry counts,
// so that a node's place in the packed entries falls out of its place in the bin.  Targets keep the caller's order and take no part.
// Bound by the latency of a few dependent passes over what stays in L2.  Before, a radix sort of three passes with a scan each, a kernel
// for the order and a scan of all counts, 24 kernels: 310 us for 32 mini-batches of 114,000 nodes on a graph of 8M, now 150 us (begin 6,
// count 18, split 28, order 50, entries 35, and their gaps).  (Two bins per warp and not eight: ordering 4 mini-batches of
// 300 targets takes 12 us instead of 34, one of 1,000 14 instead of 25.)
// A segment has as many bins as give it 32 to 64 nodes each, up to 4,096.  With 512 at most the bins of a delta of 100,000 nodes went to blocks
// instead of warps, and ids next to each other into a handful of bins: the export of 128 mini-batches on a graph of 111M nodes 1.26 ms (now 0.69;
// the radix sort 1.29), there the order alone of 32 deltas of 100,000 spread ids 246 us (now 54) and of 100,000 consecutive ones 278 (now 139).
struct ExportSeg {
    int32_t in0, len;        // its nodes in the arena
    int32_t out0;            // its first row in the packed canonical node list
    int32_t row0, lrow0;     // first packed row of the mini-batch; local row of the segment's first node in sampling order
    int32_t hop, n_tiles;
    int32_t bin0, bins, shift;   // bin of an id: bin0 + (id >> shift)
    int32_t off_shift;       // canonical row c has its offset at o_nbr_off[c + off_shift]
    int32_t ent_rel, ent0;   // its first entry in the mini-batch's packed entries, and where those start
    uint32_t ticket;         // tiles that have been counted
};
struct ExportCounts { int32_t n_tiles, n_bins, n_dense; };
struct ExportManyArgs {
    int32_t B, k, id_bits, n_bins_max;
    int32_t nodes_per_warp;  // of k_export_many_entries: 1 to 32
    int32_t hop_base[MG_MAX_HOPS + 2];
    const int32_t *nodes, *node_batch, *node_off, *cum, *rowbase0, *ent_hop, *ent_off, *ent_nbrs, *ent_repr;
    int32_t *o_node_ids, *o_nio, *o_nbrs, *o_repr, *o_nbr_off;
    int32_t* inv;            // per packed row in sampling order: the canonical row in the mini-batch
    int32_t* ent_to;         // per sampled node (arena): its first entry in the packed entry list
    ExportSeg* segs;         // [B (k + 1)]
    int2* tiles;             // (segment, tile inside it)
    ExportCounts* counts;
    uint32_t* bin_end;       // per bin: nodes, then where the next one goes, at last where the bin ends
    uint32_t* bin_ents;      // per bin: entries, then the bin's first in the mini-batch's packed entries
    int32_t* bin_seg;
    int2* keys;              // (id, local row in sampling order) in place of the packed rows, ordered by bin
    int32_t* dense_bins;     // the bins of more than kExportWarpKeys nodes
};

constexpr int kExportBinsLog = 12;     // bins of a segment at most
constexpr int kExportWarpKeys = 128;   // keys that a warp compares all with all
constexpr int kExportPairKeys = 1024;  // ... and a block, where the bin's range takes more than one bitmap
constexpr int kExportMapLog = 17;      // ids of a bitmap
constexpr int kExportBinsPerThread = (1 << kExportBinsLog) / kThreads;

// bins of a segment: a power of two that gives them 32 to 64 nodes on average (more in segments of over 262,144); none where nothing
// is to be ordered
__device__ __forceinline__ int export_bins_log(int32_t len, int id_bits) {
    const int want = len <= 64 ? 0 : 32 - __clz((len - 1) >> 6);
    return min(want, min(kExportBinsLog, id_bits));
}

// Block 0: the segments in output order and their tiles.  The others: bins to zero, and what is known of every mini-batch.
__global__ void __launch_bounds__(1024) k_export_begin(ExportManyArgs a) {
    const int32_t k = a.k, B = a.B;
    auto entries = [&](int32_t b, int32_t h) { return a.ent_hop[h * (B + 1) + b + 1] - a.ent_hop[h * (B + 1) + b]; };
    if (blockIdx.x > 0) {
        const int32_t step = (int32_t)(gridDim.x - 1) * 1024, t0 = (int32_t)(blockIdx.x - 1) * 1024 + (int32_t)threadIdx.x;
        for (int32_t i = t0; i < 2 * a.n_bins_max; i += step) a.bin_end[i] = 0u;   // (bin_ents follows)
        for (int32_t b = t0; b < B; b += step) {
            const int32_t* cum = a.cum + (int64_t)b * (k + 2);
            int32_t run = 0, ents = 0;
            a.o_nio[(int64_t)b * (k + 2)] = 0;
            for (int j = 0; j <= k; ++j) { run += cum[k - j + 1] - cum[k - j]; a.o_nio[(int64_t)b * (k + 2) + j + 1] = run; }
            for (int h = 0; h < k; ++h) ents += entries(b, h);
            a.o_nbr_off[a.rowbase0[b] + b + cum[k]] = ents;   // the terminal entry, behind the sampled nodes'
        }
        return;
    }
    __shared__ int32_t warp_sum[3][32];
    __shared__ int32_t carry[3];   // tiles, nodes, bins
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x < 3) carry[threadIdx.x] = 0;
    __syncthreads();
    const int32_t n_seg = B * (k + 1);
    for (int32_t s0 = 0; s0 < n_seg; s0 += 1024) {
        const int32_t s = s0 + (int32_t)threadIdx.x, b = s / (k + 1), h = k - s % (k + 1);
        ExportSeg g;
        g.in0 = 0; g.len = 0; g.bins = 0; g.shift = 0;
        if (s < n_seg) {
            g.in0 = a.node_off[h * (B + 1) + b];
            g.len = a.node_off[h * (B + 1) + b + 1] - g.in0;
            if (h > 0 && g.len > 0) {
                const int lg = export_bins_log(g.len, a.id_bits);
                g.bins = 1 << lg;
                g.shift = a.id_bits - lg;
            }
        }
        g.n_tiles = (g.len + kSortTile - 1) / kSortTile;
        const int32_t mine[3] = {g.n_tiles, g.len, g.bins};
        int32_t at[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const int32_t inc = (int32_t)warp_incl_scan((uint32_t)mine[q]);
            if (lane == 31) warp_sum[q][warp] = inc;
            at[q] = inc - mine[q];
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            at[q] += carry[q];
            for (int w = 0; w < warp; ++w) at[q] += warp_sum[q][w];
        }
        __syncthreads();
        if (threadIdx.x == 1023)
#pragma unroll
            for (int q = 0; q < 3; ++q) carry[q] = at[q] + mine[q];
        if (s < n_seg) {
            const int32_t* cum = a.cum + (int64_t)b * (k + 2);
            g.out0 = at[1];
            g.row0 = a.rowbase0[b];
            g.lrow0 = cum[h];
            g.hop = h;
            g.bin0 = at[2];
            g.off_shift = b - (cum[k + 1] - cum[k]);
            g.ent_rel = 0;
            g.ent0 = 0;
            for (int j = 0; j < k; ++j) {   // entries are packed mini-batch after mini-batch, inside one in the order of its nodes
                g.ent0 += a.ent_hop[j * (B + 1) + b] - a.ent_hop[j * (B + 1)];
                if (j > h) g.ent_rel += entries(b, j);
            }
            g.ticket = 0u;
            a.segs[s] = g;
            for (int32_t t = 0; t < g.n_tiles; ++t) a.tiles[at[0] + t] = make_int2(s, t);
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) { a.counts->n_tiles = carry[0]; a.counts->n_bins = carry[2]; a.counts->n_dense = 0; }
}

// Nodes and entries per bin; the block that counts a segment's last tile sums them up over its bins.
__global__ void __launch_bounds__(kThreads) k_export_count(ExportManyArgs a) {
    constexpr int kMaxBins = 1 << kExportBinsLog, kPer = kSortTile / kThreads;
    __shared__ uint32_t cnt[kMaxBins], ents[kMaxBins], part[2][kThreads / 32];
    __shared__ bool last;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int32_t n_tiles = a.counts->n_tiles;
    for (int32_t t = blockIdx.x; t < n_tiles; t += gridDim.x) {
        const int2 tile = a.tiles[t];
        const ExportSeg g = a.segs[tile.x];
        if (g.bins == 0) continue;   // (the whole block)
        const bool sampled = g.hop < a.k;
        __syncthreads();
        for (int i = threadIdx.x; i < g.bins; i += kThreads) { cnt[i] = 0u; ents[i] = 0u; }
        __syncthreads();
        const int32_t i0 = g.in0 + tile.y * kSortTile, n = min(kSortTile, g.len - tile.y * kSortTile);
        int32_t id[kPer];
#pragma unroll
        for (int j = 0; j < kPer; ++j) { const int32_t i = j * kThreads + (int32_t)threadIdx.x; id[j] = i < n ? a.nodes[i0 + i] : -1; }
#pragma unroll
        for (int j = 0; j < kPer; ++j) if (id[j] >= 0) atomicAdd(&cnt[id[j] >> g.shift], 1u);
        if (sampled) {
            uint32_t e[kPer];
#pragma unroll
            for (int j = 0; j < kPer; ++j) {
                const int32_t i = i0 + j * kThreads + (int32_t)threadIdx.x;
                e[j] = id[j] >= 0 ? (uint32_t)(a.ent_off[i + 1] - a.ent_off[i]) : 0u;
            }
#pragma unroll
            for (int j = 0; j < kPer; ++j) if (e[j]) atomicAdd(&ents[id[j] >> g.shift], e[j]);
        }
        __syncthreads();
        for (int i = threadIdx.x; i < g.bins; i += kThreads)
            if (cnt[i]) {
                atomicAdd(&a.bin_end[g.bin0 + i], cnt[i]);
                if (ents[i]) atomicAdd(&a.bin_ents[g.bin0 + i], ents[i]);
            }
        __threadfence();
        __syncthreads();
        if (threadIdx.x == 0) last = atomicAdd(&a.segs[tile.x].ticket, 1u) == (uint32_t)g.n_tiles - 1u;
        __syncthreads();
        if (!last) continue;
        __threadfence();
        const int per = max(1, g.bins / kThreads), q0 = per * (int)threadIdx.x;   // (bins are a power of two)
        uint32_t c[kExportBinsPerThread], e[kExportBinsPerThread], c_sum = 0, e_sum = 0;
#pragma unroll
        for (int q = 0; q < kExportBinsPerThread; ++q) {
            const bool on = q < per && q0 + q < g.bins;
            c[q] = on ? __ldcg(&a.bin_end[g.bin0 + q0 + q]) : 0u;
            e[q] = on ? __ldcg(&a.bin_ents[g.bin0 + q0 + q]) : 0u;
        }
#pragma unroll
        for (int q = 0; q < kExportBinsPerThread; ++q) { c_sum += c[q]; e_sum += e[q]; }
        const uint32_t ci = warp_incl_scan(c_sum), ei = warp_incl_scan(e_sum);
        if (lane == 31) { part[0][warp] = ci; part[1][warp] = ei; }
        __syncthreads();
        uint32_t c_at = (uint32_t)g.out0 + ci - c_sum, e_at = (uint32_t)g.ent_rel + ei - e_sum;
        for (int w = 0; w < warp; ++w) { c_at += part[0][w]; e_at += part[1][w]; }
#pragma unroll
        for (int q = 0; q < kExportBinsPerThread; ++q) {
            if (q >= per || q0 + q >= g.bins) break;
            const int32_t bin = g.bin0 + q0 + q;
            a.bin_end[bin] = c_at;
            a.bin_ents[bin] = e_at;
            a.bin_seg[bin] = tile.x;
            if (c[q] > (uint32_t)kExportWarpKeys) a.dense_bins[atomicAdd(&a.counts->n_dense, 1)] = bin;
            c_at += c[q];
            e_at += e[q];
        }
    }
}

// a node at its place: canonical row c of the packed list
__device__ __forceinline__ void export_node(const ExportManyArgs& a, const ExportSeg& g, int32_t c, int32_t id, int32_t local) {
    a.o_node_ids[c] = id;
    a.inv[g.row0 + local] = c - g.row0;
}
// ... and its entries: the first one stands at `rel` of the mini-batch's
__device__ __forceinline__ void export_offset(const ExportManyArgs& a, const ExportSeg& g, int32_t c, int32_t local, int32_t rel) {
    a.o_nbr_off[c + g.off_shift] = rel;
    a.ent_to[g.in0 + local - g.lrow0] = g.ent0 + rel;
}

// Every node to its bin (one global atomic per tile and bin); targets stay where they are.
__global__ void __launch_bounds__(kThreads) k_export_split(ExportManyArgs a) {
    constexpr int kMaxBins = 1 << kExportBinsLog, kPer = kSortTile / kThreads;
    __shared__ uint32_t cnt[kMaxBins], base[kMaxBins];
    const int32_t n_tiles = a.counts->n_tiles;
    for (int32_t t = blockIdx.x; t < n_tiles; t += gridDim.x) {
        const int2 tile = a.tiles[t];
        const ExportSeg g = a.segs[tile.x];
        const int32_t first = tile.y * kSortTile, n = min(kSortTile, g.len - first);
        if (g.bins == 0) {
            for (int32_t i = threadIdx.x; i < n; i += kThreads) {
                const int32_t at = g.in0 + first + i, local = g.lrow0 + first + i, c = g.out0 + first + i;
                export_node(a, g, c, a.nodes[at], local);
                if (g.hop < a.k) export_offset(a, g, c, local, g.ent_rel + a.ent_off[at] - a.ent_off[g.in0]);
            }
            continue;
        }
        __syncthreads();
        for (int i = threadIdx.x; i < g.bins; i += kThreads) cnt[i] = 0u;
        __syncthreads();
        int32_t id[kPer];
        uint32_t rank[kPer];
#pragma unroll
        for (int j = 0; j < kPer; ++j) { const int32_t i = j * kThreads + (int32_t)threadIdx.x; id[j] = i < n ? a.nodes[g.in0 + first + i] : -1; }
#pragma unroll
        for (int j = 0; j < kPer; ++j) rank[j] = id[j] >= 0 ? atomicAdd(&cnt[id[j] >> g.shift], 1u) : 0u;
        __syncthreads();
        for (int i = threadIdx.x; i < g.bins; i += kThreads) if (cnt[i]) base[i] = atomicAdd(&a.bin_end[g.bin0 + i], cnt[i]);
        __syncthreads();
#pragma unroll
        for (int j = 0; j < kPer; ++j)
            if (id[j] >= 0) a.keys[base[id[j] >> g.shift] + rank[j]] = make_int2(id[j], g.lrow0 + first + j * kThreads + (int32_t)threadIdx.x);
    }
}

__global__ void __launch_bounds__(kThreads, 5) k_export_order(ExportManyArgs a) {
    constexpr int kWarps = kThreads / 32, kMapWords = (1 << kExportMapLog) / 32, kBinsPerWarp = 2;
    __shared__ __align__(16) uint32_t map[kMapWords];   // a bitmap, or the ids of bins that are compared all with all
    __shared__ uint16_t below[kMapWords];               // set bits before a word among those of its warp
    __shared__ uint32_t warp_tot[kWarps], warp_lo[kWarps], warp_hi[kWarps], warp_next[kWarps];
    static_assert(kWarps * kExportWarpKeys <= kMapWords && kExportPairKeys <= kMapWords, "ids fit the bitmap's place");
    static_assert(kMapWords / kWarps * 32 <= 65536 && kMapWords % (32 * kWarps) == 0, "a warp's words");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int32_t n_bins = a.counts->n_bins, n_dense = a.counts->n_dense;
    auto bin_start = [&](const ExportSeg& g, int32_t bin) { return bin == g.bin0 ? g.out0 : (int32_t)a.bin_end[bin - 1]; };
    // large bins: a block each
    for (int32_t w = blockIdx.x; w < n_dense; w += gridDim.x) {
        const int32_t bin = a.dense_bins[w];
        const ExportSeg g = a.segs[a.bin_seg[bin]];
        const int32_t start = bin_start(g, bin), n = (int32_t)a.bin_end[bin] - start;
        const int2* __restrict__ keys = a.keys + start;
        const bool sampled = g.hop < a.k;
        const uint32_t id0 = (uint32_t)(bin - g.bin0) << g.shift;
        auto for_keys = [&](auto&& f) {   // (id inside the bin's range, local row), four loads in flight per thread
            for (int32_t i0 = threadIdx.x; i0 < n; i0 += 4 * kThreads) {
                int2 key[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) key[u] = i0 + u * kThreads < n ? keys[i0 + u * kThreads] : make_int2(-1, 0);
#pragma unroll
                for (int u = 0; u < 4; ++u) if (key[u].x >= 0) f((uint32_t)key[u].x - id0, key[u].y);
            }
        };
        // The range that the bin's ids really have: bitmaps start at the smallest id and skip what has none, so that their number
        // follows the ids and not the width of a bin (of a graph of 111M nodes: 27,000 ids in a segment of more than 131,072 nodes, up to
        // all of them in one of 64).
        uint32_t lo = 0, hi = (1u << g.shift) - 1u;
        if (g.shift > kExportMapLog) {
            uint32_t first = hi, last = 0;
            for_keys([&](uint32_t at, int32_t) { first = min(first, at); last = max(last, at); });
            first = __reduce_min_sync(0xFFFFFFFFu, first);
            last = __reduce_max_sync(0xFFFFFFFFu, last);
            if (lane == 0) { warp_lo[warp] = first; warp_hi[warp] = last; }
            __syncthreads();
            lo = warp_lo[0]; hi = warp_hi[0];
            for (int q = 1; q < kWarps; ++q) { lo = min(lo, warp_lo[q]); hi = max(hi, warp_hi[q]); }
        }
        // All with all: instructions by the square of the bin; bitmaps: by their words, where the ids' range takes several (in
        // units of what a warp issues for 512 words)
        const int64_t bitmaps = ((hi - lo) >> kExportMapLog) + 1;
        if (n <= kExportPairKeys && bitmaps > 1 && (int64_t)((n + kThreads - 1) / kThreads) * n * 2 <= bitmaps * 512) {
            constexpr int kPer = kExportPairKeys / kThreads;
            __syncthreads();
            int2 key[kPer];
            int32_t rank[kPer];
#pragma unroll
            for (int r = 0; r < kPer; ++r) {
                const int i = r * kThreads + (int)threadIdx.x;
                key[r] = i < n ? keys[i] : make_int2(INT32_MAX, 0);
                rank[r] = 0;
                map[i] = (uint32_t)key[r].x;
            }
            __syncthreads();
            for (int i = 0; i < n; i += 4) {
                const int4 v = *reinterpret_cast<const int4*>(&map[i]);
#pragma unroll
                for (int r = 0; r < kPer; ++r)
                    if (r == 0 || n > r * kThreads) rank[r] += (v.x < key[r].x) + (v.y < key[r].x) + (v.z < key[r].x) + (v.w < key[r].x);
            }
#pragma unroll
            for (int r = 0; r < kPer; ++r)
                if (r * kThreads + (int)threadIdx.x < n) {
                    export_node(a, g, start + rank[r], key[r].x, key[r].y);
                    if (sampled) a.o_nbr_off[start + rank[r] + g.off_shift] = key[r].y;   // (until the counts are summed up below)
                }
        } else {
            uint32_t before = 0;   // ids in the bitmaps so far
            for (;;) {
                const int words = (int)min((hi - lo) / 32 + 1, (uint32_t)kMapWords);
                const int warp_words = (words + 32 * kWarps - 1) / (32 * kWarps) * 32;
                uint32_t next = UINT32_MAX;   // the smallest id behind this bitmap
                __syncthreads();
                for (int i = threadIdx.x; i < words; i += kThreads) map[i] = 0u;
                __syncthreads();
                for_keys([&](uint32_t at, int32_t) {
                    if (at < lo) return;
                    if (at - lo < 32u * kMapWords) atomicOr(&map[(at - lo) >> 5], 1u << ((at - lo) & 31));
                    else next = min(next, at);
                });
                __syncthreads();
                uint32_t run = 0;
                for (int i = warp * warp_words + lane; i < min(words, (warp + 1) * warp_words) + lane; i += 32) {
                    const uint32_t c = i < words ? (uint32_t)__popc(map[i]) : 0u;
                    const uint32_t inc = warp_incl_scan(c);
                    if (i < words) below[i] = (uint16_t)(run + inc - c);
                    run += __shfl_sync(0xFFFFFFFFu, inc, 31);
                }
                next = __reduce_min_sync(0xFFFFFFFFu, next);
                if (lane == 0) { warp_tot[warp] = run; warp_next[warp] = next; }
                __syncthreads();
                for_keys([&](uint32_t at, int32_t local) {
                    if (at < lo || at - lo >= 32u * kMapWords) return;
                    const int wd = (int)((at - lo) >> 5);
                    uint32_t rank = before + below[wd] + (uint32_t)__popc(map[wd] & ((1u << ((at - lo) & 31)) - 1u));
                    for (int q = 0; q < wd / warp_words; ++q) rank += warp_tot[q];
                    export_node(a, g, start + (int32_t)rank, (int32_t)(id0 + at), local);
                    if (sampled) a.o_nbr_off[start + (int32_t)rank + g.off_shift] = local;
                });
                for (int q = 0; q < kWarps; ++q) { before += warp_tot[q]; next = min(next, warp_next[q]); }
                if (next == UINT32_MAX) break;
                lo = next;
            }
        }
        if (!sampled) continue;
        // in order now: the nodes' entry counts, summed up from the bin's first entry on, four consecutive nodes per thread
        uint32_t run = a.bin_ents[bin];
        for (int32_t i0 = 0; i0 < n; i0 += 4 * kThreads) {
            __syncthreads();
            const int32_t i = i0 + 4 * (int32_t)threadIdx.x, c = start + i;
            int32_t local[4];
            uint32_t ents[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) local[u] = i + u < n ? a.o_nbr_off[c + u + g.off_shift] : -1;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int32_t at = g.in0 + local[u] - g.lrow0;
                ents[u] = local[u] >= 0 ? (uint32_t)(a.ent_off[at + 1] - a.ent_off[at]) : 0u;
            }
            const uint32_t mine = ents[0] + ents[1] + ents[2] + ents[3], inc = warp_incl_scan(mine);
            if (lane == 31) warp_tot[warp] = inc;
            __syncthreads();
            uint32_t rel = run + inc - mine;
            for (int q = 0; q < kWarps; ++q) { if (q < warp) rel += warp_tot[q]; run += warp_tot[q]; }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (local[u] >= 0) export_offset(a, g, c + u, local[u], (int32_t)rel);
                rel += ents[u];
            }
        }
    }
    __syncthreads();
    // the others: a warp looks two consecutive bins up at once (lane = bin) and takes them one after the other
    int32_t* ids = reinterpret_cast<int32_t*>(map) + warp * kExportWarpKeys;
    for (int32_t b0 = ((int32_t)blockIdx.x * kWarps + warp) * kBinsPerWarp; b0 < n_bins; b0 += (int32_t)gridDim.x * kWarps * kBinsPerWarp) {
        int32_t my_seg = 0, my_start = 0, my_n = 0;
        uint32_t my_ents = 0;
        if (lane < kBinsPerWarp && b0 + lane < n_bins) {
            const int32_t bin = b0 + lane;
            my_seg = a.bin_seg[bin];
            my_start = bin == a.segs[my_seg].bin0 ? a.segs[my_seg].out0 : (int32_t)a.bin_end[bin - 1];
            my_n = (int32_t)a.bin_end[bin] - my_start;
            my_ents = a.bin_ents[bin];
        }
        for (int q = 0; q < kBinsPerWarp; ++q) {
            const int32_t n = __shfl_sync(0xFFFFFFFFu, my_n, q);
            if (n <= 0 || n > kExportWarpKeys) continue;
            const int32_t start = __shfl_sync(0xFFFFFFFFu, my_start, q);
            const ExportSeg g = a.segs[__shfl_sync(0xFFFFFFFFu, my_seg, q)];
            constexpr int kPer = kExportWarpKeys / 32;
            int2 key[kPer];
            int32_t rank[kPer];
#pragma unroll
            for (int r = 0; r < kPer; ++r) key[r] = r * 32 + lane < n ? a.keys[start + r * 32 + lane] : make_int2(INT32_MAX, 0);
#pragma unroll
            for (int r = 0; r < kPer; ++r) { ids[r * 32 + lane] = key[r].x; rank[r] = 0; }
            __syncwarp();
            for (int i = 0; i < n; i += 4) {
                const int4 v = *reinterpret_cast<const int4*>(ids + i);
#pragma unroll
                for (int r = 0; r < kPer; ++r)
                    if (r == 0 || n > r * 32) rank[r] += (v.x < key[r].x) + (v.y < key[r].x) + (v.z < key[r].x) + (v.w < key[r].x);
            }
            __syncwarp();
#pragma unroll
            for (int r = 0; r < kPer; ++r) if (r * 32 + lane < n) export_node(a, g, start + rank[r], key[r].x, key[r].y);
            if (g.hop == a.k) continue;
#pragma unroll
            for (int r = 0; r < kPer; ++r)
                if (r * 32 + lane < n) {
                    const int32_t at = g.in0 + key[r].y - g.lrow0;
                    ids[rank[r]] = a.ent_off[at + 1] - a.ent_off[at];
                }
            __syncwarp();
            uint32_t run = __shfl_sync(0xFFFFFFFFu, my_ents, q);
#pragma unroll
            for (int r = 0; r < kPer; ++r) {
                const uint32_t e = r * 32 + lane < n ? (uint32_t)ids[r * 32 + lane] : 0u;
                const uint32_t inc = warp_incl_scan(e);
                ids[r * 32 + lane] = (int32_t)(run + inc - e);
                run += __shfl_sync(0xFFFFFFFFu, inc, 31);
            }
            __syncwarp();
#pragma unroll
            for (int r = 0; r < kPer; ++r) if (r * 32 + lane < n) export_offset(a, g, start + rank[r], key[r].y, ids[rank[r]]);
            __syncwarp();
        }
    }
}

// A warp takes 32 sampled nodes (fewer where there would not be a warp for every slot of the SMs); their entries lie one behind the other in
// the arena and are read as one stream, four loads in flight per lane, each lane looking up whose its entry is.  They go to their place in the
// packed canonical entry list, the neighbours translated to canonical rows of the mini-batch.  (With 32 nodes per warp whatever their number, 100
// targets of 1,000 entries were four warps' work: 206 us, now 9; 8 mini-batches of 100 targets with 3,000 entries 9 -> 3.)
__global__ void __launch_bounds__(kThreads) k_export_many_entries(ExportManyArgs a) {
    constexpr int U = 4;
    const int lane = threadIdx.x & 31;
    const int32_t n_sampled = a.hop_base[a.k], npw = a.nodes_per_warp;
    const int64_t step = (int64_t)gridDim.x * (kThreads / 32) * npw;
    for (int64_t w0 = (blockIdx.x * (int64_t)(kThreads / 32) + (threadIdx.x >> 5)) * npw; w0 < n_sampled; w0 += step) {
        const int32_t i0 = (int32_t)w0, i = min(i0 + lane, n_sampled - 1);
        const int32_t off = lane < npw && i0 + lane < n_sampled ? a.ent_off[i] : INT32_MAX;
        const int32_t to = a.ent_to[i] - off, row0 = a.rowbase0[a.node_batch[i]];   // (lanes behind the last node: never asked for)
        const int32_t end = a.ent_off[min(i0 + npw, n_sampled)];
        for (int32_t e0 = __shfl_sync(0xFFFFFFFFu, off, 0); e0 < end; e0 += 32 * U) {
            int32_t nbr[U], row[U], at[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int32_t e = min(e0 + u * 32 + lane, end - 1);
                nbr[u] = a.ent_nbrs[e];
                row[u] = a.ent_repr[e];
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int32_t e = min(e0 + u * 32 + lane, end - 1);
                int owner = 0;   // the last node whose entries start at or before e
#pragma unroll
                for (int s = 16; s > 0; s >>= 1)
                    if (__shfl_sync(0xFFFFFFFFu, off, owner + s) <= e) owner += s;
                at[u] = __shfl_sync(0xFFFFFFFFu, to, owner) + e;
                row[u] = a.inv[__shfl_sync(0xFFFFFFFFu, row0, owner) + row[u]];
            }
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (e0 + u * 32 + lane < end) { a.o_nbrs[at[u]] = nbr[u]; a.o_repr[at[u]] = row[u]; }
        }
    }
}

// the five arrays of one mini-batch, one behind the other (mg_dense_arrays_copy); blockIdx.y = array, four loads in flight
struct ArraysCopy {
    const int32_t* src[5];
    int32_t len[5];
    int32_t align;   // every array starts at a multiple of this many elements (a power of two)
};
__global__ void __launch_bounds__(kThreads) k_copy_arrays(ArraysCopy a, int32_t* __restrict__ dst) {
    const int q = blockIdx.y;
    for (int p = 0; p < q; ++p) dst += ((int64_t)a.len[p] + a.align - 1) & -(int64_t)a.align;
    const int32_t* __restrict__ src = a.src[q];
    const int32_t n = a.len[q];
    for (int32_t i0 = blockIdx.x * 4 * kThreads + threadIdx.x; i0 < n; i0 += gridDim.x * 4 * kThreads) {
        int32_t v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) v[u] = i0 + u * kThreads < n ? src[i0 + u * kThreads] : 0;
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (i0 + u * kThreads < n) dst[i0 + u * kThreads] = v[u];
    }
}

int ilog2_ceil(int64_t x) {
    int b = 0;
    while (((int64_t)1 << b) < x) ++b;
    return b;
}

}  // namespace

// ---------------------------------------------------------------------------------------
// generic pieces other translation units use
// ---------------------------------------------------------------------------------------
size_t mg_sort_hist_elems(int64_t max_keys) { return (size_t)kBins * ((max_keys + kSortTile - 1) / kSortTile) + kBins; }
void mg_sort_params_host(SortParams* sp, int64_t n) {
    sp->zero = 0; sp->n = (int32_t)n; sp->ntiles = (int32_t)((n + kSortTile - 1) / kSortTile); sp->hist_len = kBins * sp->ntiles;
}

// LSD radix sort of 64-bit keys on bits [lo_bit, lo_bit + bits); sp (device) holds the key count.
// Keys start in buf[0]; *res_buf tells which buffer holds the result.
void mg_sort_u64(mg_ctx* ctx, uint64_t* const buf[2], const SortParams* sp, int lo_bit, int bits, uint32_t* hist,
                 uint32_t* scan_tmp, int* res_buf) {
    cudaStream_t st = ctx->stream;
    const int grid = mg_grid(ctx, 8);
    const int passes = (bits + kRadixBits - 1) / kRadixBits;
    ScanRange r{&sp->zero, &sp->hist_len, nullptr};
    mg_smem_limit(ctx, (const void*)k_radix_scatter, (int)kScatterSmem);   // (an error shows at the launch)
    int cur = 0;
    for (int p = 0; p < passes; ++p) {
        const int shift = lo_bit + kRadixBits * p;
        k_radix_hist<<<grid, kThreads, 0, st>>>(buf[cur], sp, shift, hist);
        k_scan_reduce<<<grid, kThreads, 0, st>>>(hist, r, scan_tmp);
        k_scan_tiles<<<1, 1024, 0, st>>>(scan_tmp, r, nullptr);
        k_scan_down<<<grid, kThreads, 0, st>>>(hist, r, scan_tmp);
        k_radix_scatter<<<grid, kThreads, kScatterSmem, st>>>(buf[cur], buf[cur ^ 1], sp, shift, hist);
        cur ^= 1;
    }
    ctx->launches += 5 * passes;
    *res_buf = cur;
}

// ---------------------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------------------
template <typename T>
static int dev_realloc(mg_ctx* ctx, T** p, size_t elems) {
    if (*p) cudaFree(*p);
    *p = nullptr;
    if (mg_malloc(ctx, (void**)p, std::max<size_t>(elems, 1) * sizeof(T)) != cudaSuccess) {
        cudaGetLastError();
        *p = nullptr;
        return mg_fail(ctx, MG_ERR_OOM, "device allocation of %zu bytes failed", elems * sizeof(T));
    }
    return MG_OK;
}

// tiles of a hop at most (tiles below 256 nodes: at most five per SM)
static size_t tile_states(const mg_ctx* ctx, int64_t cap_nodes) { return (size_t)cap_nodes / kThreads + (size_t)kHopBlocks * ctx->n_sms + 2; }

static int dense_alloc(mg_ctx* ctx, mg_dense* d, int32_t B, int32_t k, int64_t cap_nodes, int64_t cap_entries,
                       int32_t table_size, int32_t smem_nb) {
    int rc;
    if (!d->hdr && (rc = dev_realloc(ctx, &d->hdr, 1))) return rc;
    // scratch of the sort of one mini-batch and of the export's bins, segments and tiles: a tile per 4096 keys, and one more per (mini-batch,
    // delta) segment
    const int64_t want_sort_tiles = (std::max(cap_nodes, d->cap_nodes) + kSortTile - 1) / kSortTile + (int64_t)B * (k + 1);
    const bool grow_sort = d->cap_nodes < cap_nodes || d->cap_sort_tiles < want_sort_tiles;
    if (d->cap_nodes < cap_nodes) {
        d->cap_nodes = 0;
        if ((rc = dev_realloc(ctx, &d->nodes, (size_t)cap_nodes))) return rc;
        if ((rc = dev_realloc(ctx, &d->node_batch, (size_t)cap_nodes))) return rc;
        if ((rc = dev_realloc(ctx, &d->ent_off, (size_t)cap_nodes + 1))) return rc;
        const size_t n_states = tile_states(ctx, cap_nodes);
        if ((rc = dev_realloc(ctx, &d->tile_state, n_states))) return rc;
        MG_CUDA(ctx, cudaMemsetAsync(d->tile_state, 0, n_states * sizeof(uint64_t), ctx->stream));   // (no state carries epoch 0)
        d->epoch = 0;
        if ((rc = dev_realloc(ctx, &d->newlist[0], (size_t)cap_nodes))) return rc;
        if ((rc = dev_realloc(ctx, &d->newlist[1], (size_t)cap_nodes))) return rc;
        d->cap_nodes = cap_nodes;
    }
    if (grow_sort) {
        d->cap_sort_tiles = 0;
        const int64_t sort_tiles = want_sort_tiles;
        const int64_t scan_tiles = std::max<int64_t>((d->cap_nodes + kScanTile - 1) / kScanTile,
                                                     (kBins * sort_tiles + kScanTile - 1) / kScanTile);
        d->scan_tmp_elems = (size_t)scan_tiles + 16;
        if ((rc = dev_realloc(ctx, &d->scan_tmp, d->scan_tmp_elems))) return rc;
        d->sort_hist_elems = (size_t)kBins * sort_tiles + kBins;
        if ((rc = dev_realloc(ctx, &d->sort_hist, d->sort_hist_elems))) return rc;
        char* tables = static_cast<char*>(d->seg_tiles);   // the segments, then the tiles: there are no more of the former than of the latter
        if ((rc = dev_realloc(ctx, &tables, (size_t)sort_tiles * (sizeof(ExportSeg) + sizeof(int2))))) { d->seg_tiles = nullptr; return rc; }
        d->seg_tiles = tables;
        d->cap_sort_tiles = sort_tiles;
    }
    if (d->cap_entries < cap_entries) {
        d->cap_entries = 0;
        if ((rc = dev_realloc(ctx, &d->ent_nbrs, (size_t)cap_entries))) return rc;
        if ((rc = dev_realloc(ctx, &d->ent_repr, (size_t)cap_entries))) return rc;
        if ((rc = dev_realloc(ctx, &d->new_ids, (size_t)cap_entries))) return rc;
        d->cap_entries = cap_entries;
        d->cap_pairs = 0;
    }
    if (smem_nb > 0) {
        if (d->cap_pairs < d->cap_entries + d->cap_nodes) {   // (id, entry) of the last hop's entries, then (id, row) of the earlier nodes
            d->cap_pairs = 0;
            if ((rc = dev_realloc(ctx, &d->pairs, (size_t)(d->cap_entries + d->cap_nodes)))) return rc;
            d->cap_pairs = d->cap_entries + d->cap_nodes;
        }
        const int64_t need_share = 2 * (int64_t)B * smem_nb * (smem_nb + 1);
        if (d->cap_share < need_share) {
            d->cap_share = 0;
            if ((rc = dev_realloc(ctx, &d->share_off, (size_t)need_share))) return rc;
            d->cap_share = need_share;
        }
    }
    const int64_t need_table = (int64_t)B * table_size;
    if (d->alloc_table < need_table) {
        d->alloc_table = 0;
        if ((rc = dev_realloc(ctx, &d->hkeys, (size_t)need_table))) return rc;
        if ((rc = dev_realloc(ctx, &d->hvals, (size_t)need_table))) return rc;
        d->alloc_table = need_table;
    }
    const int64_t need_b = (int64_t)(MG_MAX_HOPS + 2) * (B + 1);
    if (d->alloc_batches < need_b) {
        d->alloc_batches = 0;
        if ((rc = dev_realloc(ctx, &d->node_off, (size_t)need_b))) return rc;
        if ((rc = dev_realloc(ctx, &d->cum, (size_t)need_b))) return rc;
        if ((rc = dev_realloc(ctx, &d->rowbase, (size_t)need_b))) return rc;
        if ((rc = dev_realloc(ctx, &d->d_ent_hop, (size_t)need_b))) return rc;
        if ((rc = dev_realloc(ctx, &d->d_seeds, (size_t)need_b))) return rc;
        if ((rc = dev_realloc(ctx, &d->batch_cnt, (size_t)need_b))) return rc;
        d->alloc_batches = need_b;
    }
    d->k = k;
    d->n_batches = B;
    d->table_size = table_size;
    return MG_OK;
}

static const char* status_text(uint32_t st) {
    if (st & ST_RANGE) return "a target id is outside [0, n_nodes)";
    if (st & ST_NONRESIDENT) return "a target lies in a partition that is not resident";
    if (st & ST_DUPLICATE) return "a batch lists a target twice";
    if (st & ST_CAP_ENTRIES) return "neighbour capacity (max_entries_total) exceeded";
    if (st & ST_CAP_NODES) return "node capacity (max_nodes_total) exceeded";
    if (st & ST_CAP_TABLE) return "per-batch node capacity (max_nodes_per_batch) exceeded";
    return "internal invariant violated";
}

static int status_code(uint32_t st) {
    if (st & ST_RANGE) return MG_ERR_ARG;
    if (st & ST_NONRESIDENT) return MG_ERR_NONRESIDENT;
    if (st & ST_DUPLICATE) return MG_ERR_DUPLICATE;
    if (st & (ST_CAP_ENTRIES | ST_CAP_NODES | ST_CAP_TABLE)) return MG_ERR_CAPACITY;
    return MG_ERR_CUDA;
}

// All sampling work is queued on the library's sampling stream, so that it can overlap a forward pass that is
// running on the context's stream.  The sampling stream first waits for whatever the caller had queued on the
// context's stream (e.g. the kernel that produced device-resident targets).
static int sample_begin_impl(mg_ctx* ctx, const int32_t* targets, int targets_on_device,
                             const int64_t* target_offsets, int32_t n_batches, const int32_t* fanouts,
                             int32_t k, const uint64_t* seeds, const mg_sample_caps* caps, mg_dense** out);

extern "C" int mg_sample_many_begin(mg_ctx* ctx, const int32_t* targets, int targets_on_device,
                                    const int64_t* target_offsets, int32_t n_batches, const int32_t* fanouts,
                                    int32_t k, const uint64_t* seeds, const mg_sample_caps* caps, mg_dense** out) {
    if (!ctx) return MG_ERR_ARG;
    cudaStream_t user = ctx->stream;
    if (cudaEventRecord(ctx->ev_user, user) == cudaSuccess) cudaStreamWaitEvent(ctx->sample_stream, ctx->ev_user, 0);
    ctx->stream = ctx->sample_stream;     // every helper launches on ctx->stream
    const int rc = sample_begin_impl(ctx, targets, targets_on_device, target_offsets, n_batches, fanouts, k, seeds, caps, out);
    ctx->stream = user;
    return rc;
}

extern "C" int mg_sample_many_end(mg_ctx* ctx, mg_dense* d) {
    if (!ctx) return MG_ERR_ARG;
    if (!d) return mg_fail(ctx, MG_ERR_ARG, "null mg_dense");
    if (!d->pending) return mg_fail(ctx, MG_ERR_STATE, "no sample in flight on this mg_dense");
    MG_CUDA(ctx, cudaSetDevice(ctx->device));
    d->pending = false;
    MG_CUDA(ctx, cudaEventSynchronize(d->ev_sampled));
    const int B = d->n_batches, k = d->k;
    const int32_t* p = d->h_stage + d->h_summary_at;
    memcpy(&d->h_hdr, p, sizeof(DenseHeader)); p += (sizeof(DenseHeader) + 3) / 4;
    d->h_cum.assign(p, p + (size_t)B * (k + 2)); p += (size_t)B * (k + 2);
    d->h_node_off.assign(p, p + (size_t)(k + 1) * (B + 1)); p += (size_t)(k + 1) * (B + 1);
    d->h_rowbase.assign(p, p + (size_t)(k + 1) * (B + 1)); p += (size_t)(k + 1) * (B + 1);
    d->h_ent_hop.assign(p, p + (size_t)k * (B + 1));
    for (int l = 0; l <= k; ++l) d->h_hdr.rows_total[l] = d->h_rowbase[(size_t)l * (B + 1) + B];
    if (d->h_hdr.status) return mg_fail(ctx, status_code(d->h_hdr.status), "%s", status_text(d->h_hdr.status));
    d->valid = true;
    d->perm_batch = -1;
    return MG_OK;
}

extern "C" int mg_sample_many(mg_ctx* ctx, const int32_t* targets, int targets_on_device,
                              const int64_t* target_offsets, int32_t n_batches, const int32_t* fanouts,
                              int32_t k, const uint64_t* seeds, const mg_sample_caps* caps, mg_dense** out) {
    const int rc = mg_sample_many_begin(ctx, targets, targets_on_device, target_offsets, n_batches, fanouts, k, seeds, caps, out);
    if (rc) return rc;
    return mg_sample_many_end(ctx, *out);
}


// dynamic shared-memory limits of the sampler's kernels (not inside a stream capture)
// The instance for a fanout, and for as many nodes per tile as the hop may have: the narrowest group of lanes that holds the fanout among
// those that waste at most two lanes of a warp; a thread per node where the hop fills larger tiles.
#define MG_HOP_KERNELS k_hop<2, false>, k_hop<3, false>, k_hop<4, false>, k_hop<5, false>, k_hop<6, false>, k_hop<8, false>, k_hop<10, false>, k_hop<16, false>, \
                       k_hop<32, false>, k_hop<2, true>, k_hop<3, true>, k_hop<4, true>, k_hop<5, true>, k_hop<6, true>, k_hop<8, true>, k_hop<10, true>, k_hop<16, true>, k_hop<20, true>
typedef void (*HopKernel)(HopArgs);
static HopKernel hop_kernel(int f, bool thread) {
    if (thread)
        return f <= 2 ? k_hop<2, true> : f == 3 ? k_hop<3, true> : f == 4 ? k_hop<4, true> : f == 5 ? k_hop<5, true> : f == 6 ? k_hop<6, true> : f <= 8 ? k_hop<8, true>
               : f <= 10 ? k_hop<10, true> : f <= 16 ? k_hop<16, true> : k_hop<20, true>;
    return f <= 2 ? k_hop<2, false> : f == 3 ? k_hop<3, false> : f == 4 ? k_hop<4, false> : f == 5 ? k_hop<5, false> : f == 6 ? k_hop<6, false> : f <= 8 ? k_hop<8, false>
           : f <= 10 ? k_hop<10, false> : f <= 16 ? k_hop<16, false> : f <= 32 ? k_hop<32, false> : k_hop<0, false>;
}

// of k_hop at most: a tile with both directions, the mini-batches' tables, the picks of a thread per node
constexpr int kHopSmem = kTileMax * (12 + 24) + 8 * MG_MAX_BATCHES + kThreads * kThreadPicks * 2 * 4;
static int sample_kernel_limits(mg_ctx* ctx) {
    MG_CUDA(ctx, mg_smem_limit(ctx, (const void*)k_dedupe_last<1024>, (int)(kDedupMaxSlots * 2 * sizeof(int32_t))));
    MG_CUDA(ctx, mg_smem_limit(ctx, (const void*)k_dedupe_last<512>, kDedupSlots512 * 2 * (int)sizeof(int32_t)));
    MG_CUDA(ctx, mg_smem_limit(ctx, (const void*)k_hop<0, false>, (int)((size_t)(kThreads / 32) * 2 * MG_MAX_FANOUT * sizeof(uint32_t)) + kHopSmem));
    return MG_OK;
}

// ... and of the others where the mini-batches' tables of k_hop, beside its tile, come to more than a kernel has without asking
static int hop_kernel_limits(mg_ctx* ctx, int32_t n_batches, bool inout) {
    if (kTileMax * hop_node_bytes(inout) + 8 * n_batches + (int)hop_pick_bytes(kThreadPicks, inout) <= 47 * 1024) return MG_OK;   // (48 KiB, of which k_hop has some for itself)
    const HopKernel hops[] = {MG_HOP_KERNELS};
    for (const HopKernel hop : hops) MG_CUDA(ctx, mg_smem_limit(ctx, (const void*)hop, kHopSmem));
    return MG_OK;
}

static int sample_begin_impl(mg_ctx* ctx, const int32_t* targets, int targets_on_device,
                             const int64_t* target_offsets, int32_t n_batches, const int32_t* fanouts,
                             int32_t k, const uint64_t* seeds, const mg_sample_caps* caps, mg_dense** out) {
    if (!ctx) return MG_ERR_ARG;
    if (!out || !target_offsets || !fanouts || !seeds) return mg_fail(ctx, MG_ERR_ARG, "null argument");
    if (n_batches <= 0 || n_batches > MG_MAX_BATCHES) return mg_fail(ctx, MG_ERR_ARG, "n_batches must be in [1, %d]", MG_MAX_BATCHES);
    if (k <= 0 || k > MG_MAX_HOPS) return mg_fail(ctx, MG_ERR_ARG, "k must be in [1, %d]", MG_MAX_HOPS);
    for (int h = 0; h < k; ++h)
        if (fanouts[h] <= 0 || fanouts[h] > MG_MAX_FANOUT) return mg_fail(ctx, MG_ERR_ARG, "fanouts must be in [1, %d]", MG_MAX_FANOUT);
    if (!ctx->row_off) return mg_fail(ctx, MG_ERR_STATE, "no graph loaded");
    if (!ctx->view_off) return mg_fail(ctx, MG_ERR_NONRESIDENT, "no partition is resident");
    const bool inout = ctx->sample_inout;
    if (inout && !ctx->view_off_out) return mg_fail(ctx, MG_ERR_STATE, "no outgoing edge list loaded");
    if (target_offsets[0] != 0) return mg_fail(ctx, MG_ERR_ARG, "target_offsets[0] must be 0");
    for (int b = 0; b < n_batches; ++b)
        if (target_offsets[b + 1] < target_offsets[b]) return mg_fail(ctx, MG_ERR_ARG, "target_offsets must be non-decreasing");
    const int64_t T = target_offsets[n_batches];
    if (T > 0 && !targets) return mg_fail(ctx, MG_ERR_ARG, "null targets");
    if (T >= (1ll << 31)) return mg_fail(ctx, MG_ERR_ARG, "too many targets");
    MG_CUDA(ctx, cudaSetDevice(ctx->device));

    // capacities: worst case unless the caller bounds them
    const int64_t N = ctx->n_nodes;
    int64_t worst_nodes_total = 0, worst_entries_total = 0, worst_nodes_batch = 0;
    for (int b = 0; b < n_batches; ++b) {
        double level = (double)(target_offsets[b + 1] - target_offsets[b]);  // nodes that can be new at this hop
        double nodes = level, entries = 0;
        for (int h = 0; h < k; ++h) {
            level = std::min(level, (double)N) * fanouts[h] * (ctx->sample_inout ? 2 : 1);
            entries += level;
            nodes += level;
        }
        const int64_t nb = (int64_t)std::min(nodes, (double)N);
        worst_nodes_total += nb;
        worst_entries_total += (int64_t)std::min(entries, 4.0e18);
        worst_nodes_batch = std::max(worst_nodes_batch, nb);
    }
    // Worst-case bounds follow the number of targets: they are rounded up on a geometric grid (steps of 1/8), so
    // that calls of similar size share allocations, table size and the captured graph.
    auto grid_up = [](int64_t v) {
        int64_t q = 1024;
        while (q < v) q += std::max<int64_t>(q / 8, 1);
        return q >= (1ll << 31) - 1 ? v : q;   // never round a legal bound out of range
    };
    int64_t cap_nodes = (caps && caps->max_nodes_total > 0) ? caps->max_nodes_total : grid_up(worst_nodes_total);
    int64_t cap_entries = (caps && caps->max_entries_total > 0) ? caps->max_entries_total : grid_up(worst_entries_total);
    int64_t cap_batch = (caps && caps->max_nodes_per_batch > 0) ? caps->max_nodes_per_batch : worst_nodes_batch;
    if (!(caps && caps->max_nodes_per_batch > 0)) cap_batch = std::min<int64_t>(grid_up(cap_batch), std::max<int64_t>(N, 1));
    cap_nodes = std::max<int64_t>({cap_nodes, T, 1});   // even an empty call needs its (one-element) arrays
    cap_batch = std::max<int64_t>(cap_batch, 1);
    for (int b = 0; b < n_batches; ++b) cap_batch = std::max<int64_t>(cap_batch, target_offsets[b + 1] - target_offsets[b]);
    if (cap_nodes >= (1ll << 31) - 1 || cap_entries >= (1ll << 31) - 1)
        return mg_fail(ctx, MG_ERR_CAPACITY, "capacities must stay below 2^31 (nodes %lld, entries %lld): pass tighter mg_sample_caps or fewer batches",
                       (long long)cap_nodes, (long long)cap_entries);
    // id table of a mini-batch: 1.625 slots per node it may hold (load factor <= 0.62 for linear probing), any size:
    // its traffic is random 32-byte sectors, so every slot that is not needed costs DRAM bandwidth
    // (sized below, once it is known whether the last hop goes through it)
    // The last hop is deduplicated in shared memory (k_bucket_entries, k_dedupe_last) when a mini-batch's nodes fit the
    // tables of 16 blocks.  Above, the global tables are the faster way (16 mini-batches of room for 480,000 nodes, 320,000 in
    // use: the sample's kernels take 698 us with k_insert, 723 us with 20 and more blocks per mini-batch).
    int64_t min_nb = (cap_batch + kDedupMaxSlots - 1) / kDedupMaxSlots;
    while (min_nb <= kDedupMaxTables && dedup_slots_for((cap_batch + min_nb - 1) / min_nb) > kDedupMaxSlots) ++min_nb;
    const int64_t dedup_nb = min_nb <= kDedupMaxTables ? dedup_buckets(n_batches, cap_batch, min_nb, ctx->n_sms) : min_nb;
    // Room for tables half as large again as they have to be, where blocks have 1,024 threads and there is that much: the probes are shorter (32 mini-batches of
    // 84,500 nodes in as much room 106 -> 65 us, 128 357 -> 245; the smaller blocks gain nothing, 49 -> 50).  k_dedupe_last takes of it what its ids need.
    const int32_t dedup_least = (int32_t)std::min<int64_t>(dedup_slots_for((cap_batch + dedup_nb - 1) / dedup_nb), kDedupMaxSlots);
    const int32_t dedup_slots = dedup_least > kDedupSlots512 ? std::min(kDedupMaxSlots, (dedup_least * 3 / 2 + 127) / 128 * 128) : dedup_least;
    const bool smem_fits = min_nb <= kDedupMaxTables && dedup_nb * n_batches < (1ll << 24) && cap_entries + cap_nodes < (1ll << 31);
    // Small samples go through the global tables in any case: these stay in L2, and k_insert takes one launch where the shared tables
    // take two (room for 14,000 nodes: the whole call 94 -> 84 us, 80,000: 192 -> 175 us, 8 x 83,000: 893 -> 883 us, 64 x 42,000:
    // equal, 37 x 100,000: 867 us with the shared tables, 880 without).
    const bool smem_last = smem_fits && (int64_t)n_batches * cap_batch > kDedupMinNodes && !getenv("MG_GLOBAL_TABLES");
    // With the last hop deduplicated in shared memory the global tables only ever hold the nodes that are sampled from
    // (targets and the inner deltas): a caller who bounds those gets tables several times smaller.  (The bound holds either way.)
    int64_t inner_nodes = cap_batch;
    if (smem_fits && caps && caps->max_inner_nodes_per_batch > 0) {
        inner_nodes = std::min<int64_t>(cap_batch, caps->max_inner_nodes_per_batch);
        for (int b = 0; b < n_batches; ++b) inner_nodes = std::max<int64_t>(inner_nodes, target_offsets[b + 1] - target_offsets[b]);
    }
    const int64_t table_nodes = smem_last ? inner_nodes : cap_batch;
    // (1.625 slots per node; four where all tables together stay within 8 MB: a sparse table saves a small hop the long probes,
    // 34 -> 17 us for the two inner hops of one mini-batch)
    auto slots_for = [](int64_t nodes) { return std::max<int64_t>(16, (nodes + nodes / 2 + nodes / 8 + 7) / 8 * 8); };
    const int32_t inner_limit = (int32_t)std::min<int64_t>(slots_for(inner_nodes), INT32_MAX);
    int64_t want_slots = slots_for(table_nodes);
    if (4 * table_nodes * n_batches <= 2ll << 20) want_slots = std::max<int64_t>(16, (4 * table_nodes + 7) / 8 * 8);
    if (want_slots > (1ll << MG_SLOT_BITS)) return mg_fail(ctx, MG_ERR_CAPACITY, "max_nodes_per_batch above %d", (int)((1ll << MG_SLOT_BITS) * 8 / 13));
    const int32_t table_size = (int32_t)want_slots;
    if ((int64_t)table_size * n_batches >= (1ll << 31))
        return mg_fail(ctx, MG_ERR_CAPACITY, "n_batches x id-table size must stay below 2^31: pass a smaller max_nodes_per_batch or fewer batches");

    mg_dense* d = *out;
    const bool created = (d == nullptr);
    if (created) { d = new mg_dense(); d->ctx = ctx; d->device = ctx->device; }
    else if (d->ctx != ctx) return mg_fail(ctx, MG_ERR_ARG, "mg_dense belongs to another context");
    d->valid = false;
    d->pending = false;
    d->export_valid = false;
    if (ctx->last_fwd_dense == d) ctx->last_fwd_dense = nullptr;   // (that pass was of the sample that ends here: mg_backward may not follow it)
    if (d->ev_read_done) MG_CUDA(ctx, cudaStreamWaitEvent(ctx->stream, d->ev_read_done, 0));
    int rc = dense_alloc(ctx, d, n_batches, k, cap_nodes, std::max<int64_t>(cap_entries, 1), table_size, smem_last ? (int32_t)dedup_nb : 0);
    if (rc) { if (created) mg_dense_free(d); return rc; }
    *out = d;
    for (int h = 0; h < k; ++h) d->fanouts[h] = fanouts[h];
    d->n_targets_total = T;
    d->n_nodes = N;
    d->resident_serial = ctx->resident_serial;
    d->slot_of_part_at_sample = ctx->slot_of_part;

    cudaStream_t st = ctx->stream;
    const int B = n_batches;
    const TableGeom tg{table_size};

    // Host-known part of the header, the per-batch tables and the seeds go through a pinned staging block of the
    // sample handle, so that the device work below reads nothing but fixed addresses: it can then be captured once
    // in a CUDA graph and replayed for every later call with the same shape.
    // (mapped, so that no copy engine is involved.)  Up to kStageTargets targets in host memory travel in it too; more are copied.
    static_assert(sizeof(DenseHeader) % 8 == 0, "the header is staged as 32-bit words");
    const size_t hdr_ints = sizeof(DenseHeader) / 4;
    const size_t seeds_at = (hdr_ints + (size_t)(B + 1) + (size_t)B * (k + 2) + 1) & ~(size_t)1;
    const size_t targets_at = seeds_at + 2 * (size_t)B;
    const void* mapped = nullptr;
    const HostMemory kind = targets_on_device || T == 0 ? HOST_PAGEABLE : mg_host_memory(targets, sizeof(int32_t) * (size_t)T, &mapped);
    const size_t n_staged = !targets_on_device && T <= kStageTargets && kind == HOST_PAGEABLE ? kStageTargets : 0;
    const size_t n_summary = hdr_ints + (size_t)B * (k + 2) + 2 * (size_t)(k + 1) * (B + 1) + (size_t)k * (B + 1);
    const size_t summary_at = targets_at + n_staged;
    if (d->h_stage_ints < summary_at + n_summary) {
        if (d->h_stage) cudaFreeHost(d->h_stage);
        d->h_stage = nullptr; d->h_stage_ints = 0;
        const size_t ints = summary_at + n_summary;
        if (cudaHostAlloc((void**)&d->h_stage, ints * sizeof(int32_t), cudaHostAllocMapped) != cudaSuccess ||
            cudaHostGetDevicePointer((void**)&d->h_stage_dev, d->h_stage, 0) != cudaSuccess) {
            cudaGetLastError();
            return mg_fail(ctx, MG_ERR_OOM, "pinned host allocation failed");
        }
        d->h_stage_ints = ints;
    }
    d->h_summary_at = summary_at;
    DenseHeader* st_hdr = reinterpret_cast<DenseHeader*>(d->h_stage);
    int32_t* st_off = d->h_stage + hdr_ints;
    int32_t* st_cum = st_off + (B + 1);
    memset(st_hdr, 0, sizeof(DenseHeader));
    st_hdr->hop_base[0] = 0;
    st_hdr->hop_base[1] = (int32_t)T;
    if (++d->epoch >= 1u << 27) {   // (27 bits of a tile state's tag; a handle gets here after 134 million samples)
        MG_CUDA(ctx, cudaMemsetAsync(d->tile_state, 0, tile_states(ctx, d->cap_nodes) * sizeof(uint64_t), st));
        d->epoch = 1;
    }
    st_hdr->epoch = d->epoch;
    memset(st_cum, 0, sizeof(int32_t) * (size_t)B * (k + 2));
    for (int b = 0; b <= B; ++b) st_off[b] = (int32_t)target_offsets[b];
    for (int b = 0; b < B; ++b) st_cum[(size_t)b * (k + 2) + 1] = st_off[b + 1] - st_off[b];
    memcpy(d->h_stage + seeds_at, seeds, sizeof(uint64_t) * B);
    if (targets_on_device) st_hdr->targets = (uint64_t)(uintptr_t)targets;
    else if (n_staged) {
        if (T > 0) memcpy(d->h_stage + targets_at, targets, sizeof(int32_t) * T);
        st_hdr->targets = (uint64_t)(uintptr_t)(d->h_stage_dev + targets_at);
    } else if (kind == HOST_MAPPED && T <= kStageTargets) {
        st_hdr->targets = (uint64_t)(uintptr_t)mapped;
    } else {
        MG_CUDA(ctx, cudaMemcpyAsync(d->newlist[1], targets, sizeof(int32_t) * T, cudaMemcpyHostToDevice, st));
        st_hdr->targets = (uint64_t)(uintptr_t)d->newlist[1];
    }
    if ((rc = sample_kernel_limits(ctx))) return rc;
    if ((rc = hop_kernel_limits(ctx, B, inout))) return rc;

    // Grids follow what a hop can hold at most (the number of targets rounded up to a power of two, so that calls of similar
    // size share the captured graph): blocks without work cost the small calls as much as the work itself.
    int64_t T_bound = 1;
    while (T_bound < T) T_bound <<= 1;
    int64_t nodes_bound[MG_MAX_HOPS + 1], entries_bound[MG_MAX_HOPS];
    nodes_bound[0] = std::min<int64_t>(T_bound, d->cap_nodes);
    for (int h = 0; h < k; ++h) {
        entries_bound[h] = std::min<int64_t>(nodes_bound[h] * fanouts[h] * (inout ? 2 : 1), d->cap_entries);
        nodes_bound[h + 1] = std::min<int64_t>({entries_bound[h], d->cap_nodes, (int64_t)B * cap_batch});
    }
    auto blocks_for = [&](int64_t items, int per_block, int ctas_per_sm) {
        return (unsigned)std::max<int64_t>(1, std::min<int64_t>((items + per_block - 1) / per_block, mg_grid(ctx, ctas_per_sm)));
    };

    // ---- everything the device does for this sample ----
    auto enqueue = [&]() -> int {
    uint32_t* batch_cnt = d->batch_cnt;   // new nodes per (hop, mini-batch)
    {
        ProfScope ps(ctx, PH_SAMPLE_INIT);
        BeginArgs a{d->h_stage_dev, (int32_t)hdr_ints, B + 1, B * (k + 2), 2 * B, (int32_t)seeds_at, k * B, (int64_t)B * table_size / 4,
                    reinterpret_cast<int32_t*>(d->hdr), d->node_off, d->cum, reinterpret_cast<int32_t*>(d->d_seeds),
                    reinterpret_cast<int32_t*>(batch_cnt), reinterpret_cast<int4*>(d->hkeys)};
        k_begin<<<blocks_for(a.n_table4, 4 * kThreads, 8), kThreads, 0, st>>>(a);
        ctx->launches++;
    }
    for (int h = 0; h < k; ++h) {
        const int32_t f = fanouts[h];
        const bool smem_hop = smem_last && h == k - 1;
        {
            ProfScope ps(ctx, PH_SAMPLE_PICK);
            const HopLaunch l = hop_launch(f, nodes_bound[h], ctx->n_sms, inout, h > 0 ? 8 * (size_t)B : 0);
            HopArgs a{d->hdr, h, f, d->nodes, d->node_batch, {ctx->view_off, inout ? ctx->view_off_out : nullptr},
                      {ctx->view_nbrs, ctx->view_nbrs_out}, d->ent_off, d->ent_nbrs, d->ent_repr, smem_hop ? 0 : 1, d->d_seeds, d->cap_entries, d->tile_state,
                      l.tile_cap, ctx->n_sms, l.per_sm, B, k, d->new_ids, batch_cnt + (size_t)(h > 0 ? h - 1 : 0) * B, d->cap_nodes,
                      inner_limit, d->cum, d->node_off, d->node_off, d->hkeys, d->hvals, tg, ctx->n_nodes, mg_feat_geom(ctx)};
            // (a thread per node: no block waits for another one to end just to find no tile left, 42,000 nodes of 3 12.1 -> 10.8 us)
            const unsigned grid = blocks_for(nodes_bound[h], 32, l.thread ? l.per_sm : 8);
            const HopKernel kern = hop_kernel(f, l.thread);
            kern<<<grid, kThreads, l.smem, st>>>(a);
            ctx->launches++;
        }
        {
            ProfScope ps(ctx, PH_SAMPLE_RELABEL);
            if (smem_hop) {
                DedupArgs da{d->hdr, h, B, k, (int32_t)dedup_nb, dedup_slots, d->nodes, d->node_off, d->ent_off, d->ent_nbrs,
                             d->ent_repr, d->pairs, d->share_off, d->cum, batch_cnt + (size_t)h * B, d->new_ids,
                             (int32_t)cap_batch, d->cap_entries};
                k_bucket_entries<<<(unsigned)(B * dedup_nb), kBucketThreads, 0, st>>>(da);
                // (threads by table size: registers let six blocks of 256 threads onto an SM, three of 512 and two of 1,024, tables as many of the
                // first two and, above 113 KB, one of the last)
                const unsigned grid = (unsigned)(B * dedup_nb);
                const size_t sm = (size_t)dedup_slots * 2 * sizeof(int32_t);
                if (dedup_slots > kDedupSlots512) k_dedupe_last<1024><<<grid, 1024, sm, st>>>(da);
                else if (dedup_slots > kDedupSlots256) k_dedupe_last<512><<<grid, 512, sm, st>>>(da);
                else k_dedupe_last<256><<<grid, 256, sm, st>>>(da);
                ctx->launches += 2;
            } else {
                InsertArgs ia{d->hdr, h, d->ent_nbrs, d->ent_repr, d->hkeys, tg, d->new_ids, B, k, d->node_off, d->ent_off,
                              d->cum, d->hvals, batch_cnt + (size_t)h * B, (int32_t)cap_batch};
                // many short blocks (64 threads: 340 us for the 254 of the large mini-batches, the counters are the limit then; 256: 255);
                // an entry per thread where the SMs hold all of the hop's at once that way (the three hops of one mini-batch 23 -> 15 us,
                // of a tiny graph 9.6 -> 7.4; with 12M entries it takes twice the time of four per thread)
                if (entries_bound[h] <= (int64_t)mg_grid(ctx, kInsertBlocks) * kInsertThreads)
                    k_insert<1><<<blocks_for(entries_bound[h], kInsertThreads, kInsertBlocks), kInsertThreads, 0, st>>>(ia);
                else
                    k_insert<kInsertPerThread><<<blocks_for(entries_bound[h], kInsertThreads * kInsertPerThread, 64), kInsertThreads, 0, st>>>(ia);
                ctx->launches++;
            }
        }
    }
    {
        ProfScope ps(ctx, PH_SAMPLE_PLACE);
        const int in_table = smem_last ? k - 1 : k;
        int64_t table_entries = 0;
        for (int h = 0; h < in_table; ++h) table_entries += entries_bound[h];
        PlaceArgs pa{d->hdr, d->new_ids, batch_cnt + (size_t)(k - 1) * B, d->cap_nodes, d->nodes, d->node_batch, d->hvals, in_table, (int32_t)cap_batch,
                     d->ent_repr, B, k, d->cum, d->node_off, (int32_t)hdr_ints, d->ent_off, d->rowbase, d->d_ent_hop, d->h_stage_dev + summary_at};
        const size_t sm = 2 * (size_t)B * sizeof(int32_t);   // 32 KiB at the largest number of mini-batches
        k_place<<<blocks_for(std::max(nodes_bound[k], table_entries), kThreads, 8) + 1, kThreads, sm, st>>>(pa);
        ctx->launches++;
    }
    MG_CUDA(ctx, cudaGetLastError());
    return MG_OK;
    };   // enqueue

    // Replay the captured graph when nothing that the device work depends on has changed since it was captured;
    // capture it (again) otherwise.  Profiling runs the launches one by one (its events do not belong in a graph).
    SampleSignature sig;
    memset(&sig, 0, sizeof(sig));
    sig.B = B; sig.k = k; sig.T_bound = T_bound; sig.table_size = table_size; sig.cap_batch = cap_batch;
    sig.cap_nodes = d->cap_nodes; sig.cap_entries = d->cap_entries; sig.n_nodes = ctx->n_nodes; sig.part_size = ctx->part_size;
    sig.inout = (inout ? 1 : 0) | (smem_last ? 2 + 4 * dedup_nb : 0) | ((int64_t)inner_limit << 16);
    for (int h = 0; h < k; ++h) sig.fanouts[h] = fanouts[h];
    const void* ptrs[] = {d->hdr, d->nodes, d->node_batch, d->ent_off, d->tile_state, d->newlist[0], d->newlist[1],
                          d->ent_nbrs, d->ent_repr, d->hkeys, d->hvals, d->node_off, d->cum, d->rowbase, d->batch_cnt,
                          d->d_ent_hop, d->d_seeds, d->h_stage_dev, d->h_stage_dev + summary_at, ctx->view_off, ctx->view_nbrs, ctx->d_slot_of_part, st,
                          ctx->d_part_of_node, inout ? (const void*)ctx->view_off_out : nullptr, inout ? (const void*)ctx->view_nbrs_out : nullptr,
                          d->pairs, d->share_off, d->new_ids};
    static_assert(sizeof(ptrs) <= sizeof(sig.ptrs), "signature too small");
    memcpy(sig.ptrs, ptrs, sizeof(ptrs));
    const bool use_graph = ctx->sample_graphs && !ctx->prof_on && !getenv("MG_NO_SAMPLE_GRAPH");
    if (use_graph) {
        if (!d->graph_exec || memcmp(&sig, &d->graph_sig, sizeof(sig)) != 0) {
            if (d->graph_exec) { cudaGraphExecDestroy(d->graph_exec); d->graph_exec = nullptr; }
            const int64_t launches0 = ctx->launches;
            MG_CUDA(ctx, cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal));
            const int erc = enqueue();
            cudaGraph_t graph = nullptr;
            const cudaError_t ce = cudaStreamEndCapture(st, &graph);
            d->graph_launches = ctx->launches - launches0;
            ctx->launches = launches0;
            if (erc || ce != cudaSuccess || !graph) {
                if (graph) cudaGraphDestroy(graph);
                cudaGetLastError();
                return erc ? erc : mg_fail(ctx, MG_ERR_CUDA, "capture of the sampler failed: %s", cudaGetErrorString(ce));
            }
            const cudaError_t ie = cudaGraphInstantiate(&d->graph_exec, graph, 0);
            cudaGraphDestroy(graph);
            if (ie != cudaSuccess) { d->graph_exec = nullptr; cudaGetLastError(); return mg_fail(ctx, MG_ERR_CUDA, "cudaGraphInstantiate: %s", cudaGetErrorString(ie)); }
            d->graph_sig = sig;
        }
        MG_CUDA(ctx, cudaGraphLaunch(d->graph_exec, st));
        ctx->launches += d->graph_launches;
    } else {
        const int erc = enqueue();
        if (erc) return erc;
    }
    if (!d->ev_sampled) MG_CUDA(ctx, cudaEventCreateWithFlags(&d->ev_sampled, cudaEventDisableTiming));
    MG_CUDA(ctx, cudaEventRecord(d->ev_sampled, st));
    d->pending = true;
    return MG_OK;
}

extern "C" int mg_sample(mg_ctx* ctx, const int32_t* targets, int targets_on_device, int32_t n_targets,
                         const int32_t* fanouts, int32_t k, uint64_t seed, const mg_sample_caps* caps, mg_dense** out) {
    if (!ctx) return MG_ERR_ARG;
    if (n_targets < 0) return mg_fail(ctx, MG_ERR_ARG, "negative n_targets");
    const int64_t off[2] = {0, n_targets};
    return mg_sample_many(ctx, targets, targets_on_device, off, 1, fanouts, k, &seed, caps, out);
}

extern "C" int mg_dense_counts(const mg_dense* d, int32_t* n_batches, int32_t* k, int64_t* nodes_per_hop,
                               int64_t* entries_per_hop) {
    if (!d) return MG_ERR_ARG;
    if (!d->valid) return MG_ERR_STATE;
    const int B = d->n_batches, K = d->k;
    if (n_batches) *n_batches = B;
    if (k) *k = K;
    if (nodes_per_hop)
        for (int b = 0; b < B; ++b)
            for (int h = 0; h <= K; ++h)
                nodes_per_hop[(size_t)b * (K + 1) + h] = d->h_cum[(size_t)b * (K + 2) + h + 1] - d->h_cum[(size_t)b * (K + 2) + h];
    if (entries_per_hop)
        for (int b = 0; b < B; ++b)
            for (int h = 0; h < K; ++h)
                entries_per_hop[(size_t)b * K + h] = d->h_ent_hop[(size_t)h * (B + 1) + b + 1] - d->h_ent_hop[(size_t)h * (B + 1) + b];
    return MG_OK;
}


static void batch_geom(const mg_dense* d, int b, BatchGeom* g) {
    const int k = d->k, B = d->n_batches;
    memset(g, 0, sizeof(*g));
    g->k = k;
    for (int h = 0; h <= k + 1; ++h) g->cum[h] = d->h_cum[(size_t)b * (k + 2) + h];
    for (int h = 0; h <= k; ++h) g->node_off[h] = d->h_node_off[(size_t)h * (B + 1) + b];
    g->V = g->cum[k + 1];
    g->n_targets = g->cum[1];
}

// perm / inv of mini-batch b (device arrays owned by d, valid until the next call for another batch or sample)
int mg_dense_batch_perm(mg_ctx* ctx, mg_dense* d, int b, const int32_t** perm, const int32_t** inv) {
    BatchGeom g;
    batch_geom(d, b, &g);
    int rc = mg_ensure(ctx, &d->perm_buf, &d->perm_elems, 2 * (size_t)g.V + 8);
    if (rc) return rc;
    *perm = d->perm_buf;
    *inv = d->perm_buf + g.V;
    if (d->perm_batch == b) return MG_OK;
    d->perm_batch = -1;
    cudaStream_t st = ctx->stream;
    if (d->export_pending) MG_CUDA(ctx, cudaStreamWaitEvent(st, d->ev_exported, 0));   // the export uses the same sort scratch
    const int32_t n = g.V - g.n_targets;
    const int id_bits = std::max(1, ilog2_ceil(d->n_nodes)), hop_bits = std::max(1, ilog2_ceil(g.k + 1));
    const int grid = std::max(1, std::min(mg_grid(ctx, 4), (g.V + kThreads - 1) / kThreads));
    int res = 0;
    if (n > 0) {
        SortParams* sp = (SortParams*)(d->scan_tmp + d->scan_tmp_elems - 8);   // tail of the scratch block, as in mg_dense_export_many
        SortParams h_sp;
        mg_sort_params_host(&h_sp, n);
        MG_CUDA(ctx, cudaMemcpyAsync(sp, &h_sp, sizeof(h_sp), cudaMemcpyHostToDevice, st));
        k_perm_keys<<<grid, kThreads, 0, st>>>(g, d->nodes, id_bits, d->newlist[0]);
        mg_sort_u64(ctx, d->newlist, sp, MG_SLOT_BITS, id_bits + hop_bits, d->sort_hist, (uint32_t*)d->scan_tmp, &res);
        ctx->launches++;
    }
    if (g.V > 0) {
        k_perm_fill<<<grid, kThreads, 0, st>>>(g, d->newlist[res], d->perm_buf, d->perm_buf + g.V);
        ctx->launches++;
    }
    MG_CUDA(ctx, cudaGetLastError());
    MG_CUDA(ctx, cudaStreamSynchronize(st));   // h_sp is a stack variable
    d->perm_batch = b;
    return MG_OK;
}

extern "C" int mg_dense_view(mg_ctx* ctx, mg_dense* d, int32_t batch, mg_dense_arrays* out) {
    if (!ctx) return MG_ERR_ARG;
    if (!d || !out) return mg_fail(ctx, MG_ERR_ARG, "null argument");
    if (!d->valid) return mg_fail(ctx, MG_ERR_STATE, "mg_dense holds no completed sample");
    if (batch < 0 || batch >= d->n_batches) return mg_fail(ctx, MG_ERR_ARG, "batch out of range");
    MG_CUDA(ctx, cudaSetDevice(ctx->device));
    const int k = d->k, B = d->n_batches, b = batch;
    ExportArgs a;
    memset(&a, 0, sizeof(a));
    batch_geom(d, b, &a.g);
    int rc = mg_dense_batch_perm(ctx, d, b, &a.perm, &a.inv);
    if (rc) return rc;
    // canonical Delta_j = hop k - j
    a.nio[0] = 0;
    for (int j = 0; j <= k; ++j) a.nio[j + 1] = a.nio[j] + (a.g.cum[k - j + 1] - a.g.cum[k - j]);
    a.n0 = a.nio[1];
    int32_t n_entries = 0;
    for (int h = 0; h < k; ++h) n_entries += d->h_ent_hop[(size_t)h * (B + 1) + b + 1] - d->h_ent_hop[(size_t)h * (B + 1) + b];
    const int32_t n_s = a.g.V - a.n0;
    const size_t need = (size_t)a.g.V + (k + 2) + 2 * (size_t)n_entries + (size_t)n_s + 1 + 16;
    rc = mg_ensure(ctx, &d->exp_buf, &d->exp_elems, need);
    if (rc) return rc;
    a.nodes = d->nodes; a.ent_off = d->ent_off; a.ent_nbrs = d->ent_nbrs; a.ent_repr = d->ent_repr;
    a.o_node_ids = d->exp_buf;
    a.o_nio = a.o_node_ids + a.g.V;
    a.o_nbrs = a.o_nio + (k + 2);
    a.o_nbr_off = a.o_nbrs + n_entries;
    a.o_repr = a.o_nbr_off + n_s + 1;
    MG_CUDA(ctx, mg_reads_wait(&ctx->array_reads, ctx->stream));   // (the last call's arrays may still be read)
    const int grid = std::max(1, std::min(mg_grid(ctx, 4), (a.g.V + kThreads - 1) / kThreads));
    k_export_nodes<<<grid, kThreads, 0, ctx->stream>>>(a);
    k_export_scan<<<1, 1024, 0, ctx->stream>>>(a.o_nbr_off, n_s);
    if (n_s > 0) k_export_entries<<<grid, kThreads, 0, ctx->stream>>>(a);
    ctx->launches += 3;
    MG_CUDA(ctx, cudaGetLastError());
    MG_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    out->k = k;
    out->n_nodes = a.g.V;
    out->n_sampled = n_s;
    out->n_entries = n_entries;
    out->node_ids = a.o_node_ids;
    out->node_id_offsets = a.o_nio;
    out->nbrs = a.o_nbrs;
    out->nbr_offsets = a.o_nbr_off;
    out->repr_map = a.o_repr;
    return MG_OK;
}

// Layout of the export buffer (int32 elements), from the sample's capacities so that it is allocated once per handle.
struct ExportLayout { size_t node_ids, nio, nbrs, repr, nbr_off, inv, ent_to, total; };
static ExportLayout export_layout(const mg_dense* d) {
    ExportLayout L;
    const size_t cn = (size_t)d->cap_nodes, ce = (size_t)d->cap_entries, B = (size_t)d->n_batches;
    size_t at = 0;
    L.node_ids = at; at += cn;
    L.nio = at; at += B * (MG_MAX_HOPS + 2);
    L.nbrs = at; at += ce;
    L.repr = at; at += ce;
    L.nbr_off = at; at += cn + B + 1;
    L.inv = at; at += cn;
    L.ent_to = at; at += cn;
    L.total = at + 16;
    return L;
}

extern "C" int mg_dense_export_many(mg_ctx* ctx, mg_dense* d) {
    if (!ctx) return MG_ERR_ARG;
    if (!d) return mg_fail(ctx, MG_ERR_ARG, "null mg_dense");
    if (d->ctx != ctx) return mg_fail(ctx, MG_ERR_ARG, "mg_dense belongs to another context");
    if (d->pending) return mg_fail(ctx, MG_ERR_STATE, "a sample is in flight on this mg_dense: call mg_sample_many_end first");
    if (!d->valid) return mg_fail(ctx, MG_ERR_STATE, "mg_dense holds no completed sample");
    MG_CUDA(ctx, cudaSetDevice(ctx->device));
    const int k = d->k, B = d->n_batches;
    const int32_t n_total = d->h_hdr.hop_base[k + 1];
    const int64_t n_segs = (int64_t)B * (k + 1);
    if ((int64_t)(n_total + kSortTile - 1) / kSortTile + n_segs > d->cap_sort_tiles)
        return mg_fail(ctx, MG_ERR_STATE, "the sort scratch of this mg_dense is too small for its sample");
    const ExportLayout L = export_layout(d);
    int rc = mg_ensure(ctx, &d->expm_buf, &d->expm_elems, L.total);
    if (rc) return rc;
    if (!d->ev_exported) MG_CUDA(ctx, cudaEventCreateWithFlags(&d->ev_exported, cudaEventDisableTiming));
    // on the sampling stream: behind the sample (and a later sample into d behind this), beside the layers
    cudaStream_t user = ctx->stream;
    cudaStream_t st = ctx->sample_stream;
    ExportManyArgs a;
    memset(&a, 0, sizeof(a));
    a.B = B; a.k = k; a.id_bits = std::max(1, ilog2_ceil(d->n_nodes));
    for (int h = 0; h <= k + 1; ++h) a.hop_base[h] = d->h_hdr.hop_base[h];
    a.nodes = d->nodes; a.node_batch = d->node_batch; a.node_off = d->node_off; a.cum = d->cum; a.rowbase0 = d->rowbase;
    a.ent_hop = d->d_ent_hop; a.ent_off = d->ent_off; a.ent_nbrs = d->ent_nbrs; a.ent_repr = d->ent_repr;
    a.o_node_ids = d->expm_buf + L.node_ids; a.o_nio = d->expm_buf + L.nio; a.o_nbrs = d->expm_buf + L.nbrs;
    a.o_repr = d->expm_buf + L.repr; a.o_nbr_off = d->expm_buf + L.nbr_off; a.inv = d->expm_buf + L.inv; a.ent_to = d->expm_buf + L.ent_to;
    a.segs = static_cast<ExportSeg*>(d->seg_tiles);
    a.tiles = reinterpret_cast<int2*>(a.segs + n_segs);
    a.n_bins_max = (int32_t)(n_segs + n_total / 32);   // (export_bins_log: a segment of more than 64 nodes has at most a bin for 32 of them)
    a.bin_end = d->sort_hist;                          // (kBins places for every tile that the scratch is sized for, and these are three for every bin)
    a.bin_ents = a.bin_end + a.n_bins_max;
    a.bin_seg = reinterpret_cast<int32_t*>(a.bin_ents + a.n_bins_max);
    a.counts = reinterpret_cast<ExportCounts*>(d->scan_tmp + d->scan_tmp_elems - 12);
    a.keys = reinterpret_cast<int2*>(d->newlist[0]);
    a.dense_bins = reinterpret_cast<int32_t*>(d->newlist[1]);
    d->export_valid = false;
    MG_CUDA(ctx, mg_reads_wait(&d->expm_reads, st));   // (the last export's arrays may still be read)
    MG_CUDA(ctx, mg_reads_wait(&ctx->array_reads, st));
    d->expm_reads.queued = false;
    if (n_total > 0) {
        const int64_t n_tiles_max = n_segs + n_total / kSortTile;
        auto blocks_for = [&](int64_t items, int per_block, int ctas_per_sm) {
            return (unsigned)std::max<int64_t>(1, std::min<int64_t>((items + per_block - 1) / per_block, mg_grid(ctx, ctas_per_sm)));
        };
        ctx->stream = st;   // (the phase events use ctx->stream)
        {
        ProfScope ps(ctx, PH_SAMPLE_SORT);
        k_export_begin<<<1 + blocks_for(a.n_bins_max + B, 1024, 1), 1024, 0, st>>>(a);
        k_export_count<<<blocks_for(n_tiles_max, 1, 8), kThreads, 0, st>>>(a);
        k_export_split<<<blocks_for(n_tiles_max, 1, 8), kThreads, 0, st>>>(a);
        k_export_order<<<blocks_for(a.n_bins_max, kThreads / 32, 8), kThreads, 0, st>>>(a);
        const int32_t n_sampled = d->h_hdr.hop_base[k];
        a.nodes_per_warp = 32;
        while (a.nodes_per_warp > 1 && n_sampled < (int64_t)a.nodes_per_warp * mg_grid(ctx, 8) * (kThreads / 32)) a.nodes_per_warp /= 2;
        k_export_many_entries<<<blocks_for(n_sampled, kThreads / 32 * a.nodes_per_warp, 8), kThreads, 0, st>>>(a);
        ctx->launches += 5;
        }
        ctx->stream = user;
    }
    MG_CUDA(ctx, cudaGetLastError());
    MG_CUDA(ctx, cudaEventRecord(d->ev_exported, st));
    d->export_pending = true;
    d->export_valid = true;
    d->perm_batch = -1;   // the per-batch permutation shares the sort scratch
    return MG_OK;
}

// where mini-batch `batch` stands in the last export
static int exported_arrays(mg_ctx* ctx, const mg_dense* d, int32_t batch, mg_dense_arrays* out) {
    if (!d || !out) return mg_fail(ctx, MG_ERR_ARG, "null argument");
    if (!d->valid || !d->export_valid) return mg_fail(ctx, MG_ERR_STATE, "no export of this sample: call mg_dense_export_many first");
    if (batch < 0 || batch >= d->n_batches) return mg_fail(ctx, MG_ERR_ARG, "batch out of range");
    const int k = d->k, B = d->n_batches, b = batch;
    const ExportLayout L = export_layout(d);
    const int32_t row0 = d->h_rowbase[b], V = d->h_rowbase[b + 1] - row0;
    const int32_t n0 = d->h_cum[(size_t)b * (k + 2) + k + 1] - d->h_cum[(size_t)b * (k + 2) + k];
    int64_t e_before = 0, e_mine = 0;   // entries are packed mini-batch after mini-batch in the export
    for (int h = 0; h < k; ++h) {
        const int32_t* at = d->h_ent_hop.data() + (size_t)h * (B + 1);
        e_before += at[b] - at[0];
        e_mine += at[b + 1] - at[b];
    }
    out->k = k;
    out->n_nodes = V;
    out->n_sampled = V - n0;
    out->n_entries = (int32_t)e_mine;
    out->node_ids = d->expm_buf + L.node_ids + row0;
    out->node_id_offsets = d->expm_buf + L.nio + (size_t)b * (k + 2);
    out->nbrs = d->expm_buf + L.nbrs + e_before;
    out->repr_map = d->expm_buf + L.repr + e_before;
    out->nbr_offsets = d->expm_buf + L.nbr_off + row0 + b;
    return MG_OK;
}

extern "C" int mg_dense_export_view(mg_ctx* ctx, mg_dense* d, int32_t batch, mg_dense_arrays* out) {
    if (!ctx) return MG_ERR_ARG;
    if (int rc = exported_arrays(ctx, d, batch, out)) return rc;
    MG_CUDA(ctx, cudaSetDevice(ctx->device));
    if (d->export_pending) { MG_CUDA(ctx, cudaEventSynchronize(d->ev_exported)); d->export_pending = false; }
    return MG_OK;
}

static int copy_arrays(mg_ctx* ctx, const mg_dense_arrays* v, int32_t* dst_dev, int32_t align, cudaStream_t st) {
    const ArraysCopy a{{v->node_ids, v->node_id_offsets, v->nbrs, v->nbr_offsets, v->repr_map},
                       {v->n_nodes, v->k + 2, v->n_entries, v->n_sampled + 1, v->n_entries}, align};
    const int longest = std::max(std::max(v->n_nodes, v->n_entries), v->n_sampled + 1);
    const int blocks = std::max(1, std::min(mg_grid(ctx, 2), (longest + 4 * kThreads - 1) / (4 * kThreads)));
    k_copy_arrays<<<dim3((unsigned)blocks, 5), kThreads, 0, st>>>(a, dst_dev);
    ctx->launches++;
    MG_CUDA(ctx, cudaGetLastError());
    return MG_OK;
}

static bool bad_align(int32_t align) { return align <= 0 || align > 1024 || (align & (align - 1)); }

extern "C" int mg_dense_export_copy_aligned(mg_ctx* ctx, mg_dense* d, int32_t batch, mg_dense_arrays* out, int32_t* dst_dev, int32_t align,
                                            void* stream) {
    if (!ctx) return MG_ERR_ARG;
    if (bad_align(align)) return mg_fail(ctx, MG_ERR_ARG, "align must be a power of two up to 1024");
    if (int rc = exported_arrays(ctx, d, batch, out)) return rc;
    if (!dst_dev) return MG_OK;
    MG_CUDA(ctx, cudaSetDevice(ctx->device));
    cudaStream_t st = (cudaStream_t)stream;
    if (d->export_pending) MG_CUDA(ctx, cudaStreamWaitEvent(st, d->ev_exported));
    if (int rc = copy_arrays(ctx, out, dst_dev, align, st)) return rc;
    MG_CUDA(ctx, mg_reads_add(&d->expm_reads, st));
    return MG_OK;
}

extern "C" int mg_dense_export_copy(mg_ctx* ctx, mg_dense* d, int32_t batch, mg_dense_arrays* out, int32_t* dst_dev, void* stream) {
    return mg_dense_export_copy_aligned(ctx, d, batch, out, dst_dev, 1, stream);
}

extern "C" int mg_dense_arrays_copy_aligned(mg_ctx* ctx, const mg_dense_arrays* v, int32_t* dst_dev, int32_t align, void* stream) {
    if (!ctx) return MG_ERR_ARG;
    if (!v || !dst_dev) return mg_fail(ctx, MG_ERR_ARG, "null argument");
    if (bad_align(align)) return mg_fail(ctx, MG_ERR_ARG, "align must be a power of two up to 1024");
    MG_CUDA(ctx, cudaSetDevice(ctx->device));
    if (int rc = copy_arrays(ctx, v, dst_dev, align, (cudaStream_t)stream)) return rc;
    MG_CUDA(ctx, mg_reads_add(&ctx->array_reads, (cudaStream_t)stream));
    return MG_OK;
}

extern "C" int mg_dense_arrays_copy(mg_ctx* ctx, const mg_dense_arrays* v, int32_t* dst_dev, void* stream) {
    return mg_dense_arrays_copy_aligned(ctx, v, dst_dev, 1, stream);
}

extern "C" int mg_dense_free(mg_dense* d) {
    if (!d) return MG_OK;
    cudaSetDevice(d->device);
    if (d->ctx && d->ctx->last_fwd_dense == d) d->ctx->last_fwd_dense = nullptr;
    cudaFree(d->hdr); cudaFree(d->nodes); cudaFree(d->node_batch); cudaFree(d->ent_off); cudaFree(d->tile_state); cudaFree(d->pairs); cudaFree(d->share_off);
    cudaFree(d->ent_nbrs); cudaFree(d->ent_repr); cudaFree(d->node_off); cudaFree(d->cum);
    cudaFree(d->rowbase); cudaFree(d->hkeys); cudaFree(d->hvals); cudaFree(d->newlist[0]); cudaFree(d->new_ids);
    cudaFree(d->newlist[1]); cudaFree(d->d_seeds); cudaFree(d->batch_cnt); cudaFree(d->scan_tmp); cudaFree(d->sort_hist); cudaFree(d->seg_tiles);
    cudaFree(d->exp_buf); cudaFree(d->perm_buf); cudaFree(d->d_ent_hop); cudaFree(d->expm_buf);
    if (d->ev_exported) cudaEventDestroy(d->ev_exported);
    mg_reads_free(&d->expm_reads);
    if (d->h_stage) cudaFreeHost(d->h_stage);
    if (d->graph_exec) cudaGraphExecDestroy(d->graph_exec);
    if (d->ev_sampled) cudaEventDestroy(d->ev_sampled);
    if (d->ev_read_done) cudaEventDestroy(d->ev_read_done);
    delete d;
    return MG_OK;
}
