// Tree-masked verification attention (Section 3.2, "Verification Phase": all tree
// tokens are scored by the target in one pass; Appendix D: the attention mask
// follows the tree).
//
// Split-KV flash-decode on the 5th-generation tensor cores.  The query rows of one
// KV head (tree token x the Hq/Hkv heads sharing it) are packed into 128-row tiles,
// so that Q K^T and P V are dense contractions: tcgen05.mma with the fp32
// accumulators (S and O) in tensor memory.  K/V tiles of 64 keys are staged by TMA
// (cp.async.bulk.tensor, one elected thread) into 128-byte-swizzled shared memory
// through mbarrier rings (four stages each for K and V), Q tiles likewise.
//
// A CTA runs two symmetric lanes that take the key tiles of its range in turn.  A lane is an
// MMA-issuing warp, a softmax warpgroup (one TMEM lane = one query row per thread) and a
// quarter of tensor memory (two S/P buffers and one O accumulator).  The softmax warpgroup
// scales, applies the ancestor bitmask (from registers, only on tiles that reach past the
// prefix), keeps the online softmax state and writes P back into the tensor-memory columns S
// came from, from where it is the A operand of P V.  P is kept as two bf16 terms (p = hi + lo):
// one bf16 rounding of the weights alone would cost up to 2^-9 per weight, about 1 % of an
// output row's rms in the worst element.  At the end the two lanes merge their results inside
// the CTA (a lane reads the other's accumulator straight from tensor memory).
//
// The work list depends only on the step parameters, which are the same for every layer of a
// step: a one-CTA kernel derives it once from the device-resident parameters and leaves it in
// the workspace as a table, so nothing about a launch depends on (TT, d, k, L) and a CTA learns
// its work from one load.  How the work is laid out is explained at the table.
//
// Every wait (mbarrier) is bounded: when it runs out the CTA raises
// RESPS_STATUS_WAIT_TIMEOUT, stops issuing work, drains its copies in flight, frees
// its tensor memory, meets the other CTAs of its cluster and returns.  Every barrier is used so
// that a waiter can never fall two phases behind (a parity wait would then never return).
#include <cuda.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>
#include <mutex>
#include <new>
#include <unordered_map>

#include "common.cuh"

namespace resps {
namespace {

constexpr int kBM = 128;           // rows per row tile (one TMEM lane each)
constexpr int kBN = 64;            // keys per tile
// Ring depths.  Both must be even: the lanes take alternate tiles and a lane waits for
// (and looks ahead at) the "full" barriers of its own tiles only, so the previous use of a stage
// must have been its own too -- with an odd depth it would be the other lane's, which this lane has
// not seen complete, and a parity wait cannot tell "not yet" from "one phase on".
constexpr int kStagesK = 4;
constexpr int kStagesV = 4;
static_assert(kStagesK % 2 == 0 && kStagesV % 2 == 0, "ring depths must be even");
constexpr int kLanes = 2;
constexpr int kSoftmaxThreads = 256;
constexpr int kPieceWarps = kSoftmaxThreads / 32;
constexpr int kProducerWarp = 8;   // K and Q tiles
constexpr int kMmaWarp0 = 9;       // lane x is issued by warp kMmaWarp0 + x
constexpr int kVProducerWarp = 11; // V tiles
constexpr int kAttnThreads = 384;
constexpr int kRegsSoftmax = 216;  // setmaxnreg: 256 x 216 + 128 x 72 = 384 x 168 <= 64 K registers
constexpr int kRegsIssue = 72;
constexpr int kMaxBatch = 256;
constexpr int kMaxCluster = 8;     // CTAs of a cluster (the portable limit)
constexpr int kMaxGrid = 256;      // clusters x CTAs (one per SM)
constexpr int kSnap = 4;           // mode stream: a cut this close to a group's edge (key tiles) is moved onto it
constexpr int kItemTiles = 4;      // what an item costs a CTA besides its tiles (its start and epilogue), in key tiles
constexpr int kMaxRounds = 4;      // mode even: most rounds of splits
constexpr int kPieceTiles = 5;     // mode whole: a group is cut where that takes more than this many key tiles off a CTA
// Two and more rounds are looked at from this many key tiles a CTA on, about 15 us a layer: below that they gain under
// 3 us a layer, and looking at them takes a step 3 us.
constexpr int kLongTiles = 24;
constexpr int kRereadNum = 5, kRereadDen = 4;
constexpr int kCutTiles = 6;       // what cut groups cost a call (partials, the combine kernel's round trips)
constexpr int kTmemCols = 512;
constexpr uint32_t kWaitLimitCycles = kWaitTest ? 2000000u : 0x70000000u;  // bounded waits give up after ~1 s of SM clocks
constexpr float kRescaleSlack = 8.0f;  // O is rescaled only when the running max grows by > 2^8
constexpr unsigned kFull = 0xFFFFFFFFu;

// How a layer's work is laid out, one of three ways:
//  whole   clusters of several CTAs, one group (sequence, KV head, row tile) per cluster.  The CTAs share
//          the group's key tiles, send each other normalised partial results through the cluster's shared
//          memory and merge a share of the rows x columns each: one kernel does the layer.  Where the tree at
//          hand has fewer groups than there are clusters (which are as many as the context's largest tree needs),
//          a group with enough key tiles is cut over several clusters, and of the warps that have merged the same
//          share in each of them the last one merges those (fp32 sums, in L2).
//  even    single CTAs; every group is cut into splits of at most T key tiles with the smallest T for which
//          the splits fit one round of the grid, or two to four (CTA c takes splits c, c + CTAs, ... in the order of
//          sequence, KV head, row tile and keys); a second, small kernel combines the partials.
//  stream  the same two kernels; the key tiles of all groups, one group after the other, are cut into equal
//          contiguous ranges, one per CTA (a CTA may end one group and begin another), or into ranges of whole
//          groups.
// Of even (each number of rounds) and stream the one with the smallest largest share is taken (tiles, items, cut
// groups).  In mode even the row tiles of a KV head go through the same keys at the same time, in mode stream at
// different times: where K and V do not stay in L2 meanwhile, every row tile reads them from HBM again, and 148 CTAs
// with 32 KB per 0.57 us ask for more than HBM has.  So the share of mode stream counts kRereadNum / kRereadDen times as
// much beyond `l2_tiles` key tiles (all KV heads of the sequences with several row tiles; head dimension 128).  In us a
// call, stream against the best of even: 8 x 24 000 keys, 80 nodes, 8B shape 416 / 351 (four rounds); 5 x 28 000 keys, 40-96
// nodes, 56 query heads 469 / 391 (four); 4 x 8192 keys, 96 nodes, 70B shape 141 / 128 (four); 16 x 4096 keys, 64 nodes, 8B
// shape 108 / 94 (two); 32 000 keys, 128 nodes 92 / 82 (one); 12 ragged sequences up to 16 000 keys, 28 query
// heads 108 / 88 (three).  With K and V that stay in L2: 8192 keys, 128 nodes 28.0 / 26.3, 8 x 2048 keys,
// 64 nodes 27.4 / 27.6.
constexpr int kModeWhole = 0, kModeEven = 1, kModeStream = 2;

struct alignas(16) PlanHead {
    int n_groups, pad[3];
};
// A cluster's (or CTA's) first item and its number of items.
struct alignas(8) PlanCluster {
    int first_item, n_items;
};
// For every item and CTA of the cluster everything the CTA needs to start.
struct alignas(16) PlanItem {
    int b_g;             // sequence | KV head << 16
    int tile_active;     // row tile of the KV head | CTAs that have key tiles of the item << 16
    int t_begin, t_end;  // this CTA's key tiles (none: t_begin == t_end)
    int n, L;            // the sequence's tree size and prefix length
    int pieces;          // items the group is cut into | (mode whole) the item's place among them << 16
    int place;           // where its partial goes (mode whole: the group's first cluster)
};
// For the combine kernel: the partials of a group are in consecutive places.
struct alignas(16) PlanGroup {
    int b_g, tile, n, first_place, pieces, pad[3];
};
static_assert(sizeof(PlanHead) == 16 && sizeof(PlanCluster) == 8 && sizeof(PlanItem) == 32 && sizeof(PlanGroup) == 32, "vector loads");

struct AttnArgs {
    const resps_step* steps;
    const int32_t* n_nodes;
    int batch;
    const __nv_bfloat16* q;
    __nv_bfloat16* o;
    float* lse;
    int64_t capacity;
    const uint64_t* mask;
    float scale_log2;
    int Hq, Hkv, max_tt;
    // Partials of the two-kernel modes (in mode whole the same goes into the cluster's shared memory).  O is stored
    // normalised (O / l, a convex combination of V rows) as fp16 times a power of two per half row that only differs
    // from 1 when a value would leave the fp16 range: half the bytes of fp32, and 11 significant bits per element
    // (2^-11, against the 2^-9 of the final bf16 rounding).
    uint4* part_o;    // [places][D/8][128 rows]  eight fp16 each
    float4* part_ml;  // [places][128 rows]   (running max m, running sum l, l * scale of each half row)
    int cluster;      // CTAs per cluster (1: modes even and stream)
    unsigned long long chunk_first;  // mode whole: first_chunk of every rank, 7 bits each
    int chunk_step;   // ... and the bytes a CTA's part takes in a stage
    int clusters;     // clusters the work list is cut for (at most gridDim / cluster)
    int max_items;
    int comb_chunk;   // partials the combine kernel fetches together
    int stream_gain;  // -1: own choice; 0: never mode even; else always where it fits (tests)
    int may_cut;      // mode whole: a group may be cut over several clusters
    int most_rounds;  // mode even: rounds that are looked at
    int rounds;       // mode even: 0: own choice; else this many rounds (tests)
    int l2_tiles;     // K and V of more key tiles (of a KV head) than this do not stay in L2
    int min_tiles;    // fewest key tiles a CTA is given (clusters: of items of more than kAloneTiles)
    int q_by_tma;     // 1: Q tiles come by TMA (128 % (Hq/Hkv) == 0), 0: by plain loads
    int log2_group;   // of Hq/Hkv, where Q tiles come by TMA
    int plan_after_wait;  // 1: the work list was written by the kernel just before this one
    int test_drop;        // test build only: 1 = the CTA's first V copy is left out
    float4* piece_acc;      // [clusters][4][128 x D/16 units] a cut group's merged share: 16 sums of a unit,
    float2* piece_ml;       // [clusters][units] (running max, running sum)
    unsigned* piece_count;  // [kMaxGrid][8] warps that have left theirs: of the group's first cluster, by CTA and warp
    int32_t* status;
    // The work list, written by attention_plan_kernel.
    PlanHead* plan_head;
    PlanCluster* plan_cluster;  // [kMaxGrid]
    PlanItem* plan_first;       // [kMaxGrid] every CTA's first item (one load instead of two in a row)
    PlanItem* plan_item;        // [max_items x cluster] the others
    PlanGroup* plan_group;      // [groups]
};

__host__ __device__ __forceinline__ int ceil_div(int a, int b) {  // a >= 0, b > 0: the unsigned division is the shorter one
    return static_cast<int>((static_cast<unsigned>(a) + static_cast<unsigned>(b) - 1u) / static_cast<unsigned>(b));
}

// CTAs of a cluster that get key tiles of an item with `tiles` of them: the fewest among which the fullest has as few
// tiles as it can (7 tiles in a cluster of 6: four CTAs 7.4 us a layer, six 7.6).  Up to kAloneTiles tiles stay in one CTA,
// which rounds nothing before O: split, a layer of the 8B shape with 32 nodes takes 5.9 to 6.1 us instead of 7.2 to 8.2, but
// its partials would be rounded to fp16; as fp32 they need more code than the calls of all other lengths can bear
// (8B shape at 1024 keys 8.3 / 8.7).
constexpr int kAloneTiles = 5;
__device__ __forceinline__ int active_ctas(int tiles, int cluster, int min_tiles) {
    if (tiles <= kAloneTiles) return 1;
    return ceil_div(tiles, max(ceil_div(tiles, cluster), min_tiles));
}

// ---------------------------------------------------------------------------- work list
// Bound by latency (one CTA, once per step): a scan over the sequences, a search, then a thread per CTA or
// item.  Positions are in key tiles of the sequence of groups (b, KV head, row tile).
struct PlanShared {
    unsigned long long start[kMaxBatch + 1];  // first position of a sequence, in key tiles ...
    unsigned long long cost0[kMaxBatch + 1];  // ... and with every group's kItemTiles
    int group0[kMaxBatch + 1];                // first group of a sequence
    int n[kMaxBatch], L[kMaxBatch], tiles[kMaxBatch], kt[kMaxBatch];
    // mode even, by rounds - 1 (a warp each)
    int item0[kMaxRounds][kMaxBatch + 1];     // first item of a sequence (also the first place of its partials)
    int splits[kMaxRounds][kMaxBatch];        // items a group is cut into
    unsigned long long cut[2][kMaxGrid + 1];
    int n_items[kMaxGrid];
    int even_share[kMaxRounds], even_cost[kMaxRounds];  // mode even: largest share of a CTA, and what comes on top
    int range_cost[2];                         // largest share of a CTA: ranges of whole groups, equal ranges
    int cut_groups;                            // mode whole: groups are cut over several clusters
    int reread;                                // K and V are read again by every row tile in mode stream
};
static_assert(kMaxGrid >= 32 * kMaxRounds, "a warp per number of rounds");

__global__ void __launch_bounds__(kMaxGrid) attention_plan_kernel(const AttnArgs a) {
    __shared__ PlanShared sh;
    const int tid = threadIdx.x, lane = tid & 31, G = a.Hq / a.Hkv;
    const int reach = min(32, a.batch);  // lanes that a scan over the sequences has to span
    pdl_wait();  // the step parameters and node counts are complete
    pdl_launch_dependents();
    if (tid < a.batch) {
        int n = min(max(a.n_nodes[tid], 0), a.max_tt);
        const int L = max(a.steps[tid].prefix_len, 0);
        if (static_cast<int64_t>(L) + n > a.capacity) {
            atomicOr(a.status, RESPS_STATUS_KV_OVERFLOW);
            n = 0;
        }
        sh.n[tid] = n, sh.L[tid] = L;
        sh.tiles[tid] = ceil_div(n * G, kBM);
        sh.kt[tid] = (n > 0) ? ceil_div(L + n, kBN) : 0;
    }
    __syncthreads();
    if (tid < 32 * kMaxRounds) {  // (each of these warps scans for itself, the first one keeps what it finds)
        const int w = tid >> 5;
        unsigned long long pos = 0;
        int group = 0;
#pragma unroll 1
        for (int b0 = 0; b0 < a.batch; b0 += 32) {
            const int b = b0 + lane;
            int groups = (b < a.batch) ? a.Hkv * sh.tiles[b] : 0;
            unsigned long long work = (b < a.batch) ? static_cast<unsigned long long>(groups) * sh.kt[b] : 0ull;
            const int own_groups = groups;
            const unsigned long long own_work = work;
#pragma unroll 1
            for (int d = 1; d < reach; d <<= 1) {
                const int g = __shfl_up_sync(kFull, groups, d);
                const unsigned long long before = __shfl_up_sync(kFull, work, d);
                if (lane >= d) groups += g, work += before;
            }
            if (w == 0 && b < a.batch) {
                sh.start[b] = pos + work - own_work, sh.group0[b] = group + groups - own_groups;
                sh.cost0[b] = sh.start[b] + static_cast<unsigned long long>(sh.group0[b]) * kItemTiles;
            }
            pos += __shfl_sync(kFull, work, min(31, a.batch - b0 - 1));
            group += __shfl_sync(kFull, groups, min(31, a.batch - b0 - 1));
        }
        if (tid == 0) {
            sh.start[a.batch] = pos, sh.group0[a.batch] = group;
            sh.cost0[a.batch] = pos + static_cast<unsigned long long>(group) * kItemTiles;
        }
        // ---- mode whole: the clusters that the groups leave are given to them by their key tiles; a group stays whole
        // where a piece saves a CTA too little ------------------------------------------------------------------------
        bool cut = false;
        if (w == 0 && a.may_cut && group < a.clusters) {
            const int gain = a.stream_gain > 0 ? 0 : kPieceTiles * a.cluster, spare = a.clusters - group;
            int base = 0;
#pragma unroll 1
            for (int b0 = 0; b0 < a.batch; b0 += 32) {
                const int b = b0 + lane, kt = (b < a.batch) ? sh.kt[b] : 0;
                int pieces = 1;
                if (kt > gain) {  // (fewer groups than CTAs, of at most 2^15 tiles: 32 bits hold the sum)
                    pieces += static_cast<int>(static_cast<unsigned>(spare * kt) / static_cast<unsigned>(pos));
                    pieces = min(pieces, kt);
                    if (kt - ceil_div(kt, pieces) <= gain) pieces = 1;
                }
                cut = cut || pieces > 1;
                const int own = (b < a.batch) ? a.Hkv * sh.tiles[b] * pieces : 0;
                int incl = own;
#pragma unroll 1
                for (int d = 1; d < reach; d <<= 1) {
                    const int v = __shfl_up_sync(kFull, incl, d);
                    if (lane >= d) incl += v;
                }
                if (b < a.batch) sh.splits[0][b] = pieces, sh.item0[0][b] = base + incl - own;
                base += __shfl_sync(kFull, incl, min(31, a.batch - b0 - 1));
            }
            cut = __any_sync(kFull, cut);
            if (lane == 0) sh.item0[0][a.batch] = base;
        }
        if (tid == 0) {
            sh.cut_groups = cut;
            sh.range_cost[0] = sh.range_cost[1] = 0;
            PlanHead h = {};
            h.n_groups = group;
            *a.plan_head = h;
        }
        if (a.cluster == 1) {
            // ---- mode even: the smallest T (in steps of T/16) for which the splits fit the rounds ----------------------
            const int rounds = w + 1, room = rounds * a.clusters;
            const bool is_long = pos >= static_cast<unsigned long long>(kLongTiles) * a.clusters;
            const bool looked_at = a.stream_gain != 0 &&
                (a.rounds > 0 ? a.rounds == rounds : rounds == 1 || (rounds <= a.most_rounds && is_long));
            int T = max(static_cast<int>(min((pos + room - 1) / room, 1ull << 24)), 1);
            bool fits = false;
#pragma unroll 1
            for (int tries = 0; tries < 40 && looked_at && !fits; ++tries) {
                unsigned count = 0;
#pragma unroll 1
                for (int b = lane; b < a.batch; b += 32)
                    count += static_cast<unsigned>(a.Hkv * sh.tiles[b] * ceil_div(sh.kt[b], max(T, a.min_tiles)));
                count = __reduce_add_sync(kFull, min(count, 1u << 20));
                fits = count <= static_cast<unsigned>(room);
                if (!fits) T += max(1, T >> 4);
            }
            T = max(T, a.min_tiles);
            int base = 0, tiles = 0, most = 0;
            bool split = false;
#pragma unroll 1
            for (int b0 = 0; b0 < a.batch && (fits || w == 0); b0 += 32) {
                const int b = b0 + lane, splits = (b < a.batch) ? ceil_div(sh.kt[b], T) : 0;
                int incl = (b < a.batch && fits) ? a.Hkv * sh.tiles[b] * splits : 0;
                split = split || splits > 1;
                most = max(most, splits > 0 ? ceil_div(sh.kt[b], splits) + kItemTiles : 0);
                if (b < a.batch && sh.tiles[b] > 1) tiles += min(a.Hkv * sh.kt[b], 1 << 22);
                const int own = incl;
#pragma unroll 1
                for (int d = 1; d < reach; d <<= 1) {
                    const int v = __shfl_up_sync(kFull, incl, d);
                    if (lane >= d) incl += v;
                }
                if (b < a.batch) sh.splits[w][b] = splits, sh.item0[w][b] = base + incl - own;
                base += __shfl_sync(kFull, incl, min(31, a.batch - b0 - 1));
            }
            tiles = __reduce_add_sync(kFull, min(tiles, 1 << 25));
            most = __reduce_max_sync(kFull, most);
            split = __any_sync(kFull, split);
            if (lane == 0) {
                sh.item0[w][a.batch] = base;
                const bool allowed = fits && base <= a.max_items;
                // (one item, or items of one sequence, the same to a tile; else the CTAs' sums are looked at below)
                sh.even_share[w] = (a.batch == 1 || rounds == 1) ? ceil_div(base, a.clusters) * most : 0;
                sh.even_cost[w] = !allowed ? 1 << 30 : (split ? kCutTiles : 0) - (a.stream_gain > 0 ? 1 << 28 : 0);  // besides the share
                if (w == 0) sh.reread = tiles > a.l2_tiles;
            }
        }
    }
    __syncthreads();
    auto last_at_or_before = [&](const int* first, int x) {  // the last sequence whose entry is <= x
        int lo = 0, hi = a.batch;
#pragma unroll 1
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (first[mid] <= x) lo = mid; else hi = mid;
        }
        return lo;
    };
    auto item_of = [&](int b, int local) {  // what all pieces of a group share
        PlanItem p = {};
        const int head = static_cast<int>(static_cast<unsigned>(local) / static_cast<unsigned>(sh.tiles[b]));
        p.b_g = static_cast<int>(static_cast<unsigned>(b) | (static_cast<unsigned>(head) << 16));
        p.tile_active = static_cast<int>(static_cast<unsigned>(local - head * sh.tiles[b]) | (1u << 16));
        p.n = sh.n[b], p.L = sh.L[b], p.pieces = 1;
        return p;
    };
    auto write_group = [&](int group, const PlanItem& p) {  // by the group's first item
        PlanGroup q = {};
        q.b_g = p.b_g, q.tile = p.tile_active & 0xFFFF, q.n = p.n, q.first_place = p.place, q.pieces = p.pieces;
        a.plan_group[group] = q;
    };
    // ---- ranges ---------------------------------------------------------------------------------------
    // (of a position before the end; `extra` units of every group come before its tiles)
    auto locate = [&](const unsigned long long* first, unsigned long long pos, int extra, int& b, int& local, int& t) {
        int lo = 0, hi = a.batch;  // last sequence that starts at or before pos (and is not empty there)
#pragma unroll 1
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (first[mid] <= pos) lo = mid; else hi = mid;
        }
        b = lo;
        const unsigned off = static_cast<unsigned>(pos - first[b]);  // < groups x length of a group: fits 32 bits
        const unsigned len = static_cast<unsigned>(sh.kt[b] + extra);
        local = static_cast<int>(off / len);
        t = max(static_cast<int>(off - static_cast<unsigned>(local) * len) - extra, 0);
    };
    int b = 0, local = 0, t = 0;
    if (a.cluster == 1) {
        if (tid <= a.clusters) {
            const unsigned long long cost = sh.cost0[a.batch];
            const unsigned long long at = cost * static_cast<unsigned long long>(tid) / static_cast<unsigned long long>(a.clusters);
            unsigned long long whole = sh.start[a.batch], equal = whole;
            if (at < cost) {
                locate(sh.cost0, at, kItemTiles, b, local, t);
                const int behind = sh.kt[b] - t;
                const unsigned long long g0 = sh.start[b] + static_cast<unsigned long long>(local) * sh.kt[b];
                whole = g0 + (t <= behind ? 0 : sh.kt[b]);
                // a piece shorter than its own epilogue is not worth a cut; nor are ranges of less than a tile (several CTAs
                // would begin at one place, and the pieces of a group are counted by its CTAs)
                equal = (min(t, behind) <= kSnap || cost < static_cast<unsigned long long>(a.clusters)) ? whole : g0 + t;
            }
            sh.cut[0][tid] = whole, sh.cut[1][tid] = equal;
        }
        __syncthreads();
        if (tid < a.clusters) {
#pragma unroll 1
            for (int w = 0; w < 2; ++w) {
                const unsigned long long begin = sh.cut[w][tid], end = sh.cut[w][tid + 1];
                if (begin == end) continue;
                int b1, local1, t1;
                locate(sh.start, end - 1, 0, b1, local1, t1);
                locate(sh.start, begin, 0, b, local, t);
                const int items = sh.group0[b1] + local1 - sh.group0[b] - local + 1;
                atomicMax(&sh.range_cost[w], static_cast<int>(end - begin) + items * kItemTiles + (w ? kCutTiles : 0));
            }
            // (sequences of different lengths give items of different lengths: a CTA's real sum counts)
#pragma unroll 1
            for (int w = 1; w < kMaxRounds && a.batch > 1; ++w) {
                if (sh.even_cost[w] == 1 << 30) continue;
                const int n = sh.item0[w][a.batch];
                int share = 0;
#pragma unroll 1
                for (int item = tid; item < n; item += a.clusters) {
                    const int b = last_at_or_before(sh.item0[w], item);
                    share += ceil_div(sh.kt[b], sh.splits[w][b]) + kItemTiles;
                }
                atomicMax(&sh.even_share[w], share);
            }
        }
        __syncthreads();
    }
    const int ranges = sh.range_cost[1] < sh.range_cost[0] ? 1 : 0;
    int mode = kModeWhole, even = 0;
    if (a.cluster == 1) {
#pragma unroll 1
        for (int w = 1; w < kMaxRounds; ++w)
            if (sh.even_cost[w] + sh.even_share[w] < sh.even_cost[even] + sh.even_share[even]) even = w;
        const long long range_cost = static_cast<long long>(sh.range_cost[ranges]) * (sh.reread ? kRereadNum : kRereadDen);
        mode = static_cast<long long>(sh.even_cost[even] + sh.even_share[even]) * kRereadDen <= range_cost ? kModeEven : kModeStream;
    }
    if (mode == kModeEven) {
        // ---- CTA c takes items c, c + CTAs, ... --------------------------------------------------------------------
        const int n = sh.item0[even][a.batch], rounds = ceil_div(n, a.clusters);  // (that are used)
        if (tid < a.clusters) {
            PlanCluster c;
            c.first_item = tid * rounds, c.n_items = 0;
#pragma unroll 1
            for (int item = tid; item < n; item += a.clusters, ++c.n_items) {
                const int b = last_at_or_before(sh.item0[even], item), splits = sh.splits[even][b], kt = sh.kt[b];
                const int at = item - sh.item0[even][b], local = static_cast<int>(static_cast<unsigned>(at) / static_cast<unsigned>(splits));
                const int sp = at - local * splits;
                PlanItem p = item_of(b, local);
                p.t_begin = kt * sp / splits, p.t_end = kt * (sp + 1) / splits;  // (kt <= 2^15, splits <= 2^10)
                p.pieces = splits, p.place = item;
                *(c.n_items == 0 ? a.plan_first + tid : a.plan_item + c.first_item + c.n_items) = p;
                if (sp == 0) write_group(sh.group0[b] + local, p);
            }
            a.plan_cluster[tid] = c;
        }
        return;
    }
    if (mode == kModeWhole) {
        // ---- a group, or a piece of one, per cluster (more than clusters only if a tree is larger than the context's
        // limits allow) ----------------------------------------------------------------------------------------------
        const bool cut = sh.cut_groups != 0;
        const int* const first = cut ? sh.item0[0] : sh.group0;
        const int n = first[a.batch];
        if (tid < a.clusters) {
            PlanCluster c;
            c.first_item = static_cast<int>(static_cast<unsigned>(n) * tid / a.clusters);
            c.n_items = static_cast<int>(static_cast<unsigned>(n) * (tid + 1) / a.clusters) - c.first_item;
            if (n <= a.clusters) c.first_item = tid, c.n_items = (tid < n) ? 1 : 0;
            a.plan_cluster[tid] = c;
#pragma unroll 1
            for (int i = 0; i < c.n_items; ++i) {
                const int item = c.first_item + i, b = last_at_or_before(first, item);
                int local = item - first[b], pieces = 1, piece = 0, t0 = 0, kt = sh.kt[b];
                if (cut && sh.splits[0][b] > 1) {
                    pieces = sh.splits[0][b];
                    piece = local, local = static_cast<int>(static_cast<unsigned>(local) / static_cast<unsigned>(pieces));
                    piece -= local * pieces;
                    t0 = kt * piece / pieces, kt = kt * (piece + 1) / pieces - t0;
                }
                PlanItem p = item_of(b, local);
                const int act = active_ctas(kt, a.cluster, a.min_tiles);
                p.tile_active = (p.tile_active & 0xFFFF) | (act << 16);
                p.pieces = pieces | (piece << 16), p.place = item - piece;
                p.t_end = t0;
#pragma unroll 1
                for (int r = 0; r < a.cluster; ++r) {
                    p.t_begin = p.t_end;
                    if (r < act) p.t_end = t0 + kt * (r + 1) / act;
                    *(i == 0 ? a.plan_first + tid * a.cluster + r : a.plan_item + item * a.cluster + r) = p;
                }
            }
        }
        return;
    }
    const unsigned long long* const cuts = sh.cut[ranges];
    if (tid < a.clusters) {
        int count = 0;
        if (cuts[tid] < cuts[tid + 1]) {
            int b1, local1, t1;
            locate(sh.start, cuts[tid + 1] - 1, 0, b1, local1, t1);
            locate(sh.start, cuts[tid], 0, b, local, t);
            count = sh.group0[b1] + local1 - sh.group0[b] - local + 1;
        }
        sh.n_items[tid] = count;
    }
    __syncthreads();
    if (tid < a.clusters) {
        int first = 0;
#pragma unroll 4
        for (int i = 0; i < tid; ++i) first += sh.n_items[i];
        const int count = min(sh.n_items[tid], max(a.max_items - first, 0));
        const unsigned long long begin = cuts[tid], end = cuts[tid + 1];
        auto cluster_of = [&](unsigned long long pos) {  // the last CTA that begins at or before pos
            int lo = 0, hi = a.clusters;
#pragma unroll 1
            while (hi - lo > 1) {
                const int mid = (lo + hi) >> 1;
                if (cuts[mid] <= pos) lo = mid; else hi = mid;
            }
            return lo;
        };
        unsigned long long pos = begin;
#pragma unroll 1
        for (int i = 0; i < count; ++i) {
            const unsigned long long g0 = pos - static_cast<unsigned>(t), g1 = g0 + static_cast<unsigned>(sh.kt[b]);  // the group
            const unsigned long long stop = g1 < end ? g1 : end;
            const int c0 = (g0 >= begin) ? tid : cluster_of(g0), c1 = (g1 <= end) ? tid : cluster_of(g1 - 1);
            PlanItem p = item_of(b, local);
            p.t_begin = t, p.t_end = static_cast<int>(stop - g0), p.pieces = c1 - c0 + 1, p.place = first + i;
            *(i == 0 ? a.plan_first + tid : a.plan_item + first + i) = p;
            if (t == 0) write_group(sh.group0[b] + local, p);
            // on to the next group
            pos = stop, t = 0;
            if (++local == a.Hkv * sh.tiles[b]) {
                local = 0;
                do ++b; while (b < a.batch && sh.kt[b] == 0);
            }
        }
        PlanCluster c;
        c.first_item = first, c.n_items = count;
        a.plan_cluster[tid] = c;
    }
}

// A CTA's view of one item.
struct Item {
    int b, g, n, L, M, row_base;
    int t_begin, t_end;  // this CTA's key tiles (none: t_begin == t_end)
    int active;          // CTAs of the cluster that have tiles of the item
    int pieces, place;
};

__device__ __forceinline__ Item load_item(const PlanItem* entry, int G) {
    const int4* src = reinterpret_cast<const int4*>(entry);
    const int4 lo = __ldcg(src), hi = __ldcg(src + 1);
    Item it;
    it.b = lo.x & 0xFFFF, it.g = static_cast<int>(static_cast<unsigned>(lo.x) >> 16);
    it.row_base = (lo.y & 0xFFFF) * kBM, it.active = static_cast<int>(static_cast<unsigned>(lo.y) >> 16);
    it.t_begin = lo.z, it.t_end = lo.w;
    it.n = hi.x, it.L = hi.y, it.pieces = hi.z & 0xFFFF, it.place = hi.w;
    it.M = it.n * G;
    return it;
}

// ---------------------------------------------------------------------------- PTX wrappers
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
// Never suspends the thread (a try_wait may): for looking ahead.
__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
// Behind arrivals from other CTAs of the cluster.
__device__ __forceinline__ bool mbar_try_cluster(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
// Arrives on the barrier at the same place in the shared memory of CTA `rank` of the cluster.
__device__ __forceinline__ void mbar_arrive_remote(uint32_t bar, int rank) {
    asm volatile(
        "{\n\t.reg .b32 remote;\n\t"
        "mapa.shared::cluster.u32 remote, %0, %1;\n\t"
        "mbarrier.arrive.release.cluster.shared::cluster.b64 _, [remote];\n\t}" ::"r"(bar), "r"(rank)
        : "memory");
}
// Sixteen bytes into the shared memory of a CTA of the cluster; they count on the mbarrier beside them there.
__device__ __forceinline__ void store_async(uint32_t dst, uint4 v, uint32_t bar) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(dst), "r"(v.x),
                 "r"(v.y), "r"(v.z), "r"(v.w), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ uint32_t at_rank(uint32_t local, int rank) {
    uint32_t remote;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(local), "r"(rank));
    return remote;
}
// Bounded wait: false when this wait ran out (about a second of SM clocks) or another thread of
// the CTA has given up.  Kept to a few instructions, because it is inlined at every wait: a role runs
// through its code once per launch, most of it cold, and what it costs to fetch is about a cycle per 4
// bytes.  The caller records the failure in its `alive` flag, and the status word is written once, at
// the end of the kernel.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
    if (mbar_try(bar, parity)) return true;  // the common case does not even read the clock
    const uint32_t t0 = static_cast<uint32_t>(clock());
#pragma unroll 1
    while (!mbar_try(bar, parity))  // the 32-bit cycle counter wraps after two seconds; it is read far more often than that
        if (static_cast<uint32_t>(clock()) - t0 > kWaitLimitCycles || *abort_flag) return false;
    return true;
}
__device__ __forceinline__ bool cluster_bar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
    const uint32_t t0 = static_cast<uint32_t>(clock());
#pragma unroll 1
    while (!mbar_try_cluster(bar, parity))
        if (static_cast<uint32_t>(clock()) - t0 > kWaitLimitCycles || *abort_flag) return false;
    return true;
}
// For the tear-down: a copy this thread issued must have landed before the CTA gives up its shared
// memory, whatever else went wrong, so this wait looks at nothing but its own barrier and clock.
__device__ __forceinline__ bool drain_wait(uint32_t bar, uint32_t parity) {
    const uint32_t t0 = static_cast<uint32_t>(clock());
    uint32_t spins = 0;
    while (!mbar_try(bar, parity))
        if ((++spins & 255u) == 0u && static_cast<uint32_t>(clock()) - t0 > kWaitLimitCycles) return false;
    return true;
}
// Same, with a warp-uniform answer (the callers go on to warp-collective TMEM instructions).
__device__ __forceinline__ bool warp_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
    const bool ok = mbar_wait(bar, parity, abort_flag);
    return __all_sync(0xFFFFFFFFu, ok);
}
// One lane of a converged warp.
__device__ __forceinline__ bool elect_one() {
    uint32_t pred;
    asm volatile(
        "{\n\t.reg .pred P;\n\t"
        "elect.sync _|P, 0xFFFFFFFF;\n\t"
        "selp.u32 %0, 1, 0, P;\n\t}"
        : "=r"(pred));
    return pred != 0;
}
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// TMA: one box of a 5-D view into shared memory.  The last dimension of every view is the
// 64-element column panel, so that one copy brings all panels of a tile, each in its own
// 128-byte-swizzled block (the innermost coordinate is always 0).
__device__ __forceinline__ void tma_load_5d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0,
                                            int c1, int c2, int c3, int c4) {
    asm volatile(
        "cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4, %5, %6}], [%7];" ::"r"(dst),
        "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4), "r"(bar)
        : "memory");
}

// Shared-memory matrix descriptor, 128-byte swizzle (layout type 2), descriptor version 1: the low word has the start
// address (in 16 bytes; in a cluster an address has more bits than the field) and the leading offset, the high word
// never changes (8 rows of 128 bytes from group to group).
__device__ __forceinline__ constexpr uint32_t desc_lo(uint32_t addr, uint32_t lbo_bytes) { return (addr & 0x3FFFFu) >> 4 | (lbo_bytes >> 4) << 16; }
constexpr uint32_t kDescHi = (1024u >> 4) | 1u << 14 | 2u << 29;
// Instruction descriptor: bf16 x bf16 -> fp32, M = 128, A K-major.
__host__ __device__ constexpr uint32_t instr_desc(int n, bool b_mn_major) {
    return (1u << 4) | (1u << 7) | (1u << 10) | (b_mn_major ? (1u << 16) : 0u) |
           (static_cast<uint32_t>(n >> 3) << 17) | (static_cast<uint32_t>(kBM >> 4) << 24);
}
template <uint32_t kIdesc, bool kAccumulate>
__device__ __forceinline__ void umma(uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 a, b;\n\t"
        "mov.b64 a, {%1, %3};\n\tmov.b64 b, {%2, %3};\n\tsetp.ne.b32 p, %5, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %4, p;\n\t}" ::"r"(d_tmem),
        "r"(a_lo), "r"(b_lo), "n"(kDescHi), "n"(kIdesc), "n"(kAccumulate ? 1 : 0)
        : "memory");
}
// A operand from tensor memory (lane = row, two bf16 per 32-bit column).
template <uint32_t kIdesc>
__device__ __forceinline__ void umma_ts(uint32_t d_tmem, uint32_t a_tmem, uint32_t b_lo, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 b;\n\t"
        "mov.b64 b, {%2, %3};\n\tsetp.ne.b32 p, %5, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], b, %4, p;\n\t}" ::"r"(d_tmem),
        "r"(a_tmem), "r"(b_lo), "n"(kDescHi), "n"(kIdesc), "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void umma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
                 : "memory");
}

__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
          "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]),
          "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]),
          "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
        "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
        "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};" ::"r"(taddr),
        "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]),
        "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]),
        "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]),
        "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
        : "memory");
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// Packed fp32 pairs (one instruction for two lanes of arithmetic) and the 3-input maximum.
__device__ __forceinline__ unsigned long long pack2(float lo, float hi) {
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(unsigned long long v, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c) {
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ unsigned long long add2(unsigned long long a, unsigned long long b) {
    unsigned long long d;
    asm("add.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ unsigned long long sub2(unsigned long long a, unsigned long long b) {
    unsigned long long d;
    asm("sub.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ float max3(float a, float b, float c) {
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&v);
}
__device__ __forceinline__ uint32_t pack_half2(float lo, float hi) {
    __half2 v = __floats2half2_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&v);
}


// ---------------------------------------------------------------------------- merge in a cluster
// A partial (128 rows x D columns) is cut into chunks of 32 rows x 16 columns, row block by row block, and CTA `rank` of
// the cluster merges the chunks [first_chunk(rank), first_chunk(rank + 1)), a warp a chunk.  All CTAs send them their parts
// of these chunks: the warp that holds rows and columns stores fp16 pairs and the rows' (max, sum, sum x scale) into the
// merging CTA's shared memory (st.async, bytes counted by its mbarrier), so that nobody reads what is far away and no
// fence waits for stores.
// Bound by the way between SMs: 32 KB from each of 6 CTAs to the others are there 1480 clocks after the first store (8
// CTAs 1300, 3 1540); plain remote stores behind a releasing arrival 2740 (3100, 2120), bulk copies 2950.  Through
// L2 (partials written, a meeting, read back) the 8B shape spent 3.5 us between its merged lanes and O.
__host__ __device__ constexpr int chunks_of(int D) { return kBM / 32 * (D / 16); }
__host__ __device__ constexpr int first_chunk(int D, int cluster, int rank) { return (chunks_of(D) * rank + cluster - 1) / cluster; }
static_assert(chunks_of(128) < 128 && 7 * (kMaxCluster + 1) <= 64, "AttnArgs::chunk_first");
// (from the launch's table: a division by the cluster's size takes a hundred clocks, and there were a dozen on the way)
__device__ __forceinline__ int chunk_at(const AttnArgs& a, int rank) { return static_cast<int>(a.chunk_first >> (7 * rank)) & 127; }
// a chunk's place: 32 rows x 2 units of eight fp16, then the rows' (max, sum, sum x scale) where it is the first chunk of
// its rows and half of the columns that the CTA merges
constexpr int kChunkBytes = 32 * 32, kRowBytes = 32 * 16, kSlotBytes = kChunkBytes + kRowBytes;
__host__ __device__ constexpr int chunks_most(int D, int cluster) { return (chunks_of(D) + cluster - 1) / cluster; }
constexpr int most_staged(int D) {
    int most = 0;
    for (int c = 2; c <= kMaxCluster; ++c) most = most < c * chunks_most(D, c) ? c * chunks_most(D, c) : most;
    return most;
}

// ---------------------------------------------------------------------------- shared memory map
template <int D>
struct Smem {
    static constexpr int kPanels = D / 64;                   // 64-element (128-byte) column panels
    static constexpr int kQPanel = kBM * 128;                // one panel of a Q row tile
    static constexpr int kQTile = kPanels * kQPanel;
    static constexpr int kKVPanel = kBN * 128;
    static constexpr int kKVTile = kPanels * kKVPanel;
    static constexpr int kOffQ = 0;
    static constexpr int kOffK = kOffQ + kQTile;
    static constexpr int kOffV = kOffK + kStagesK * kKVTile;
    static constexpr int kOffBar = kOffV + kStagesV * kKVTile;
    static constexpr int kNumBars = 2 * (kStagesK + kStagesV) + 2 + kLanes * 6 + 4;
    static constexpr int kOffMisc = kOffBar + 8 * 40;
    static constexpr int kOffMerge = kOffMisc + 64;          // (max, sum) of every row of both lanes
    static constexpr int kUsed = kOffMerge + kLanes * kBM * 8;
    // Mode whole: what the CTAs of the cluster send for this CTA's share of the merge, [CTA][chunk of the share].
    static constexpr int kOffStage = kOffMerge + kLanes * kBM * 8;
    static constexpr int kStage = most_staged(D) * kSlotBytes;
    // Never less than 120 KB, more than half of an SM's shared memory: one CTA per SM, so the
    // 512-column TMEM allocation can never wait for a neighbour.
    static constexpr int kBytes = kUsed > 120 * 1024 ? kUsed : 120 * 1024;
    static_assert(kNumBars <= 40, "barrier area");
    static_assert(2 * kBytes > 228 * 1024, "two CTAs must not fit on one SM");
    static constexpr int kClusterBytes = kUsed + kStage > kBytes ? kUsed + kStage : kBytes;
    static_assert(kClusterBytes <= 227 * 1024, "shared memory of a CTA");
};

// barrier indices
__device__ __forceinline__ constexpr int bar_kfull(int s) { return s; }
__device__ __forceinline__ constexpr int bar_vfull(int s) { return kStagesK + s; }
// K and V stages are released separately: a K tile is dead once its Q K^T has completed, long
// before the P V of the same tile, and the next K can be on its way meanwhile.
__device__ __forceinline__ constexpr int bar_kempty(int s) { return kStagesK + kStagesV + s; }
__device__ __forceinline__ constexpr int bar_vempty(int s) { return 2 * kStagesK + kStagesV + s; }
constexpr int kBar0 = 2 * (kStagesK + kStagesV);  // first barrier after the ring's
__device__ __forceinline__ constexpr int bar_qfull() { return kBar0; }
__device__ __forceinline__ constexpr int bar_qempty() { return kBar0 + 1; }
// Lane m's S and P share a TMEM buffer (its j-th tile uses buffer j & 1) and each buffer has its own
// barriers: a buffer's next phase cannot complete before the other side has observed the
// current one (QK(j+2) is issued after PV(j), which is issued after pfull(j) was seen), so a
// parity wait never falls two phases behind.  One pfull barrier for both buffers would: the
// softmax warps can finish tile j+1 while the MMA thread still waits for V(j).
// pvdone likewise: whoever has seen S(j) knows that PV(j-2) has completed (QK(j) was issued behind it),
// so PV(j) and PV(j-1) may be waited for without having looked at every tile's.
__device__ __forceinline__ constexpr int bar_sfull(int m, int buf) { return kBar0 + 2 + m * 6 + buf; }
__device__ __forceinline__ constexpr int bar_pfull(int m, int buf) { return kBar0 + 2 + m * 6 + 2 + buf; }
__device__ __forceinline__ constexpr int bar_pvdone(int m, int buf) { return kBar0 + 2 + m * 6 + 4 + buf; }
constexpr int kBar1 = kBar0 + 2 + kLanes * 6;
// the softmax warpgroups have read an item's O: the next item's P V may overwrite it (its Q K^T need not wait)
__device__ __forceinline__ constexpr int bar_item() { return kBar1; }
// both softmax warpgroups have their partial result (and its PV completions) behind them
__device__ __forceinline__ constexpr int bar_merge() { return kBar1 + 1; }
// everything the CTA merges is in its shared memory: its own warps' arrivals, the other CTAs' bytes
__device__ __forceinline__ constexpr int bar_meet() { return kBar1 + 2; }
// every warp of the cluster has merged its share of the item: the next item's may be sent
__device__ __forceinline__ constexpr int bar_free() { return kBar1 + 3; }

// Sixteen columns of a row: O, and with the first ones the row's log-sum-exp.
// (row of a KV head -> token; heads in a group: a power of two where Q comes by TMA)
template <bool kPow2>
__device__ __forceinline__ unsigned token_of(const AttnArgs& a, unsigned R, int G) {
    return kPow2 ? R >> a.log2_group : R / static_cast<unsigned>(G);
}
template <bool kPow2>
__device__ __forceinline__ int64_t output_row(const AttnArgs& a, const Item& it, int r, int G) {
    const unsigned R = it.row_base + r, t = token_of<kPow2>(a, R, G), h = it.g * G + (R - t * G);
    return (static_cast<int64_t>(it.b) * a.max_tt + t) * a.Hq + h;
}
template <int D>
__device__ __forceinline__ void write_unit(const AttnArgs& a, int64_t row, int c16, float Mx, float den, const float (&acc)[16]) {
    const float inv = 1.f / den;
    uint32_t o[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) o[e] = pack_bf16(acc[2 * e] * inv, acc[2 * e + 1] * inv);
    uint4* dst = reinterpret_cast<uint4*>(a.o + row * D + c16 * 16);
    dst[0] = make_uint4(o[0], o[1], o[2], o[3]);
    dst[1] = make_uint4(o[4], o[5], o[6], o[7]);
    if (a.lse && c16 == 0) a.lse[row] = (Mx + log2f(den)) * 0.6931471805599453f;
}
// The chunk that a warp merges, and where the row of the lane goes.
struct MergeAt {
    int q, r;       // chunk; row of the tile (past the valid ones: nothing to do)
    int data, rows; // its places in the stage
    int64_t out;    // row of O
};
template <int D, bool kPow2>
__device__ __forceinline__ MergeAt merge_at(const AttnArgs& a, const Item& it, int q, int q0, int lane, int G) {
    MergeAt m;
    m.q = q, m.r = q / (D / 16) * 32 + lane;
    m.data = (q - q0) * kSlotBytes + lane * 16;
    m.rows = (max(q / (D / 32) * (D / 32), q0) - q0) * kSlotBytes + kChunkBytes + lane * 16;
    m.out = output_row<kPow2>(a, it, m.r, G);
    return m;
}
// Merges a chunk of the partials in the CTA's shared memory, O = sum_p w_p O_p / sum_p w_p l_p with
// w_p = 2^(m_p - max m).  kPiece: the group is cut over several
// clusters, the sums go to the workspace.  (Copies of the code, so that the common ones have nothing to skip.)
template <int D, bool kPiece>
__device__ __forceinline__ void merge_chunk(const AttnArgs& a, const Item& it, const unsigned char* stage, const MergeAt& m, int lane,
                                            unsigned cluster_id) {
    constexpr int kUnits = kBM * (D / 16);
    if (it.row_base + m.r >= it.M) return;
    float Mx = -INFINITY, den = 0.f;
#pragma unroll
    for (int p = 0; p < kMaxCluster; ++p)
        Mx = fmaxf(Mx, *reinterpret_cast<const float*>(stage + m.rows + min(p, it.active - 1) * a.chunk_step));
    unsigned long long acc2[8] = {};
#pragma unroll 2
    for (int p = 0; p < it.active; ++p) {
        const unsigned char* const src = stage + p * a.chunk_step;
        const float4 ml = *reinterpret_cast<const float4*>(src + m.rows);
        const uint4 v0 = *reinterpret_cast<const uint4*>(src + m.data), v1 = *reinterpret_cast<const uint4*>(src + m.data + 512);
        const float w = ml.x == -INFINITY ? 0.f : ex2_approx(ml.x - Mx);  // an empty partial is zeros
        den += ml.y * w;
        const float wo = ml.z * w;  // O_p = Ohat * l * scale
        const uint32_t hw[8] = {v0.x, v0.y, v0.z, v0.w, v1.x, v1.y, v1.z, v1.w};
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&hw[e]));
            acc2[e] = fma2(pack2(f.x, f.y), pack2(wo, wo), acc2[e]);
        }
    }
    float acc[16];
#pragma unroll
    for (int e = 0; e < 8; ++e) unpack2(acc2[e], acc[2 * e], acc[2 * e + 1]);
    if (!kPiece) {
        write_unit<D>(a, m.out, m.q % (D / 16), Mx, den, acc);
    } else {
        const unsigned u = m.q * 32 + lane;
#pragma unroll
        for (int e = 0; e < 4; ++e)
            __stcg(a.piece_acc + (cluster_id * 4 + e) * kUnits + u,
                   make_float4(acc[4 * e], acc[4 * e + 1], acc[4 * e + 2], acc[4 * e + 3]));
        __stcg(a.piece_ml + cluster_id * kUnits + u, make_float2(Mx, den));
    }
}
// A group that is cut over several clusters: the same warp of the same CTA of each has merged the same units.  It
// says so (nobody waits), and the one that finds that all others have done so merges the pieces: two round trips to L2
// more on the way of a cut group, 2.5 to 3 us, against 0.6 us for each key tile that it takes off a CTA (kPieceTiles).
// Under a context for 128 nodes on the 8B shape (32 clusters of 4), in us a layer uncut / cut / the two kernels with the
// same context: 16 nodes at 4096 keys 14.6 / 12.9 / 14.1, at 8192 22.7 / 15.4 / 16.7, at 12 288 30.9 / 17.7 / 19.2;
// 64 nodes 15.0 / 13.7 / 15.6, 23.1 / 18.4 / 19.4, 31.2 / 22.6 / 23.2.
template <int D, bool kPow2>
__device__ __forceinline__ void merge_pieces(const AttnArgs& a, const Item& it, int rank, int tid, int G) {
    constexpr unsigned kUnits = kBM * (D / 16);
    const int lane = tid & 31, nv = min(kBM, it.M - it.row_base);
    const int q0 = chunk_at(a, rank) + (tid >> 5), q1 = chunk_at(a, rank + 1);
    bool any = false;
    for (int q = q0; q < q1; q += kPieceWarps) any = any || q / (D / 16) * 32 < nv;
    if (!any) return;  // the warp has no units (in no piece)
    unsigned* const count = a.piece_count + (it.place * a.cluster + rank) * kPieceWarps + (tid >> 5);
    unsigned before = 0;
    __syncwarp();  // (orders the lanes' sums before the first one's arrival)
    if ((tid & 31) == 0) asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], 1;" : "=r"(before) : "l"(count) : "memory");
    before = __shfl_sync(kFull, before, 0);
    if (before + 1u != static_cast<unsigned>(it.pieces)) return;
    if ((tid & 31) == 0) __stcg(count, 0u);  // for the next layer
    __syncwarp();
#pragma unroll 1
    for (int q = q0; q < q1; q += kPieceWarps) {
        const int r = q / (D / 16) * 32 + lane;
        if (r >= nv) continue;
        const unsigned u = q * 32 + lane;
        float Mx = -INFINITY, den = 0.f;
        float acc[16] = {};
#pragma unroll 2
        for (int p = 0; p < it.pieces; ++p) {
            const unsigned cluster = static_cast<unsigned>(it.place + p);
            const float2 ml = __ldcg(a.piece_ml + cluster * kUnits + u);
            float4 v[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) v[e] = __ldcg(a.piece_acc + (cluster * 4 + e) * kUnits + u);
            if (ml.x == -INFINITY) continue;  // nothing of the piece is visible to the row
            const float mx = fmaxf(Mx, ml.x), c = ex2_approx(Mx - mx), w = ex2_approx(ml.x - mx);
            Mx = mx, den = den * c + ml.y * w;
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                acc[4 * e] = acc[4 * e] * c + v[e].x * w, acc[4 * e + 1] = acc[4 * e + 1] * c + v[e].y * w;
                acc[4 * e + 2] = acc[4 * e + 2] * c + v[e].z * w, acc[4 * e + 3] = acc[4 * e + 3] * c + v[e].w * w;
            }
        }
        write_unit<D>(a, output_row<kPow2>(a, it, r, G), q % (D / 16), Mx, den, acc);
    }
}

__device__ __forceinline__ int cluster_index() {
    int c;
    asm("mov.u32 %0, %%clusterid.x;" : "=r"(c));
    return c;
}
// What of the kernel a launch needs: the two-kernel modes, mode whole, mode whole where groups may be cut; Q by TMA or
// by plain loads.  A launch runs through most of its code once, and an SM keeps 32 KB of it: straight code of up to
// 24 KB takes a clock an instruction, in the next launch too, of 48 KB and more 2.1 clocks wherever it is in its loops.  One
// kernel for all forms had 76 KB (head dimension 128); these have 39, 55 and 64 with uniform warp indexes, constant base
// addresses and 32-bit descriptor words.  In us a call before / now, the cluster's exchange included: 8B shape at 1024
// keys 9.35 / 7.9, 128 nodes at 2048 keys 13.4 / 11.6, 13B shape 15.1 / 13.6, 28 heads of two users 12.6 / 10.0, 70B
// shape 22.4 / 20.4, 8 ragged sequences 60.1 / 55.8, 32 000 keys 31.6 / 29.5, 4 heads of 64 5.06 / 4.5.
enum Form { kSingles, kWhole, kCut };
template <int D, int kForm, bool kQByTma>
__global__ void __launch_bounds__(kAttnThreads, 1)
tree_attention_kernel(const AttnArgs a, const __grid_constant__ CUtensorMap map_k,
                      const __grid_constant__ CUtensorMap map_v, const __grid_constant__ CUtensorMap map_q) {
    using S = Smem<D>;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    const uint32_t base = smem_u32(smem_raw);
    unsigned char* base_ptr = smem_raw;
    const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(kFull, tid >> 5, 0);  // (known to be the same for the warp)
    const int G = a.Hq / a.Hkv;
    constexpr bool kClusters = kForm != kSingles;
    const int cluster_id = kClusters ? cluster_index() : static_cast<int>(blockIdx.x);
    const int rank = kClusters ? static_cast<int>(cluster_rank()) : 0;
    const uint32_t bars = base + S::kOffBar;
    auto bar = [&](int i) { return bars + 8u * i; };
    volatile int* abort_flag = reinterpret_cast<volatile int*>(base_ptr + S::kOffMisc + 8);

    // ---- one-time set-up ---------------------------------------------------------------
    // A lane a barrier, by several warps side by side (one thread after the other took 450 clocks longer); the producers'
    // barriers by the producers themselves: their first copies go out before the cluster meets.
    const bool is_producer = warp == kProducerWarp || warp == kVProducerWarp;
    {
        static_assert(kStagesK == 4 && kStagesV == 4 && kLanes == 2, "places by lane");
        int i = -1;
        uint32_t count = 1;
        if (is_producer) {
            if (lane < 8) i = (lane & 3) + (lane >> 2) * 8 + (warp == kVProducerWarp ? 4 : 0);  // full and empty, K's and V's in turn
            if (warp == kProducerWarp && (lane >> 1) == 4) i = bar_qfull() + (lane & 1), count = lane & 1 ? kLanes : kQByTma ? 1 : kSoftmaxThreads;
        } else if (warp == 5) {
            if (lane < 8) i = bar_sfull(lane >> 2, lane & 1) + (lane & 2) * 2;  // S, P V
        } else if (warp == 6) {
            if (lane < 4) i = bar_pfull(lane >> 1, lane & 1), count = kBM / 32;  // one arrival per warp
        } else if (warp == 7) {
            if (lane < 4) i = bar_item() + lane, count = lane < 2 ? kSoftmaxThreads : lane == 2 ? kPieceWarps : a.cluster * kPieceWarps;
        }
        if (i >= 0) {
            mbar_init(bar(i), count);
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        }
        if (is_producer) fence_proxy_async();
        if (tid == 0) *abort_flag = 0;
    }
    if (warp == kMmaWarp0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         base + S::kOffMisc),
                     "r"(kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (warp == kMmaWarp0 + 1 && lane == 0) {
        asm volatile("prefetch.tensormap [%0];" ::"l"(&map_k) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&map_v) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&map_q) : "memory");
    }
    // The work list was written once for the whole step.  From the second layer on it is at least
    // two kernels old: this kernel can only have started after its predecessor had started, which
    // can only have started after every CTA of the kernel before that one had passed its own
    // dependency wait, i.e. after the kernel that wrote the list had completed and flushed.  (That kernel before
    // is an attention kernel, or comes behind one: the first call's follows the list's writer at once and signals
    // its dependents only after its own wait.  The combine kernel signals before its wait.)  So the
    // list is read before the wait, under the tail of the preceding kernel; only when the list was
    // written by the kernel immediately before this one does the read have to follow the wait.
    // Behind the set-up, which then overlaps the list's writer too: work list and first layer of the 8B shape at 1024 keys
    // 10.8 us a call with the wait in front of the set-up, 10.5 so; 4 heads of 64 7.55 / 7.05, 70B shape 24.8 / 24.45; layers
    // that find the list made 8.0 / 8.0, 4.7 / 4.7, 20.7 / 20.7.  (Read twice, in front of the set-up where the list is old: 10.55,
    // 7.2, 24.6, and 28 heads 9.4 / 9.3 with a list made.)
    // Every thread reads the CTA's first item for itself: no role waits for another.
    if (a.plan_after_wait) pdl_wait();
    int first_item = 0, n_items = 0;
    Item first_it = {};
    if (cluster_id < a.clusters) {
        const int2 c = __ldcg(reinterpret_cast<const int2*>(a.plan_cluster + cluster_id));
        first_it = load_item(a.plan_first + blockIdx.x, G);
        first_item = c.x, n_items = c.y;
    }
    // Everything so far touches no global memory but the work list, so under programmatic dependent launch it overlaps the
    // tail of the preceding kernel.  The barriers are visible in the cluster behind the pair of arrival and wait (other CTAs
    // arrive on this one's barriers), what else there is in the CTA behind its own barrier: the arrival need not release
    // anything (one that does waits for the work list's loads, 500 to 900 clocks; from a CTA's first instruction to here
    // 1800 clocks before, for the CTAs that start last on the way of every call).
    tc_fence_before();
    __syncwarp();
    if constexpr (kClusters) asm volatile("barrier.cluster.arrive.relaxed;" ::: "memory");
    __syncthreads();
    tc_fence_after();
    pdl_wait();
    pdl_launch_dependents();
    auto load_q = [&](const Item& it) {
        mbar_expect_tx(bar(bar_qfull()), S::kQTile);
        tma_load_5d(base + S::kOffQ, &map_q, bar(bar_qfull()), 0, 0, it.g, it.b * a.max_tt + it.row_base / G, 0);
    };
    auto load_tile = [&](const Item& it, int t, uint32_t use, bool v) {
        const int s = use % kStagesK;
        const uint32_t full = bar(v ? bar_vfull(s) : bar_kfull(s));
        mbar_expect_tx(full, S::kKVTile);
        tma_load_5d(base + (v ? S::kOffV : S::kOffK) + s * S::kKVTile, v ? &map_v : &map_k, full, 0, t * kBN, it.g, it.b, 0);
    };
    static_assert(kStagesK == kStagesV, "load_tile");
    // The producers issue the first copies of the CTA's first item at once.
    const bool early = n_items > 0 && first_it.t_begin < first_it.t_end;
    if (early && lane == 0 && (warp == kProducerWarp || warp == kVProducerWarp)) {
        const bool is_v = warp == kVProducerWarp;
        // (in the wait test's build the CTA's first V copy may be left out)
        if (!(kWaitTest && is_v && (a.test_drop & 1))) load_tile(first_it, first_it.t_begin, 0, is_v);
        if (!is_v && kQByTma) load_q(first_it);
    }
    __syncwarp();
    if constexpr (kClusters) cluster_wait();
    constexpr uint32_t tmem = 0;  // all columns are allocated: they begin at 0
    // The list must still describe the step parameters it is used with (the caller changes them only
    // through the library, or asks for a new list): one thread compares its item's sequence.
    bool stale = false;
    if (tid == 0 && n_items > 0) {
        const int n_live = min(max(a.n_nodes[first_it.b], 0), a.max_tt), L_live = max(a.steps[first_it.b].prefix_len, 0);
        stale = (n_live != first_it.n) || (L_live != first_it.L);
    }
    auto get_item = [&](int i) { return i == 0 ? first_it : load_item(a.plan_item + (first_item + i) * (kClusters ? a.cluster : 1) + rank, G); };

    // Running use counts of the barrier families.  Every role walks the same items and tiles in
    // the same order, so each keeps its own copy.
    uint32_t kt_run = 0;     // K/V ring uses (all tiles of all items)
    uint32_t jx = 0;         // tiles this lane has taken (S/P buffers, PV completions)
    uint32_t items_run = 0;  // items with tiles for this CTA
    bool alive = true;

    // Registers follow the roles: the softmax warpgroups hold a tile of S, a tile of P and a row of
    // O; the warpgroup of the producers and MMA issuers needs few (384 x 168 at launch).
    if (warp >= kProducerWarp) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsIssue));
    if (warp == kProducerWarp || warp == kVProducerWarp) {
        // ================================ TMA producers: K tiles and Q; V tiles ==============
        if (lane == 0) {
            const bool is_v = warp == kVProducerWarp;
#pragma unroll 1
            for (int i = 0; i < n_items && alive; ++i) {
                const Item it = get_item(i);
#pragma unroll 1
                for (int t = it.t_begin; t < it.t_end; ++t, ++kt_run) {
                    const int s = kt_run % kStagesK;
                    if (kt_run == 0 && early) {  // went out during the set-up, and the item's Q with it
                        ++items_run;
                        continue;
                    }
                    // the first use of a stage finds it free
                    if (kt_run >= kStagesK && !mbar_wait(bar(is_v ? bar_vempty(s) : bar_kempty(s)),
                                                         ((kt_run / kStagesK) & 1u) ^ 1u, abort_flag)) {
                        alive = false;
                        break;
                    }
                    load_tile(it, t, kt_run, is_v);
                    if (t == it.t_begin && !is_v && kQByTma) {
                        // Q follows the first K tile: K and Q are what the first MMA needs.  The Q
                        // tile of the previous item is free once its last QK^T has completed.
                        if (!mbar_wait(bar(bar_qempty()), (items_run & 1u) ^ 1u, abort_flag)) {
                            alive = false;
                            ++kt_run;
                            break;
                        }
                        load_q(it);
                        ++items_run;
                    }
                }
            }
            // Drain: every copy this thread issued has landed before the CTA may exit (each one is
            // waited for, also after an earlier wait has run out).
            bool landed = is_v || !(kQByTma && items_run > 0) || drain_wait(bar(bar_qfull()), (items_run - 1u) & 1u);
            const uint32_t issued = kt_run;
#pragma unroll 1
            for (uint32_t u = (issued > kStagesK ? issued - kStagesK : 0u); u < issued; ++u)
                landed = drain_wait(bar(is_v ? bar_vfull(u % kStagesK) : bar_kfull(u % kStagesK)), (u / kStagesK) & 1u) && landed;
            alive = alive && landed;
        }
    } else {
        // ================================ MMA issuer of lane x ============================
        // The whole warp walks the loop and waits (so that every value stays warp-uniform);
        // one elected lane issues.  The MMAs of one thread execute in issue order: QK of this
        // lane's tile j+1 is issued before PV of tile j, so the tensor pipe has S(j+1) to work on
        // while the softmax warps turn S(j) into P(j), and QK(j+2) cannot overwrite the TMEM
        // buffer j & 1 before PV(j) has read P(j) from it.
        // The MMAs of a tile are unrolled: one elected thread issues them, and what it needs per instruction is on
        // the chain of every tile.  As loops (QK by two, PV rolled) a call took, in us: 70B shape at 4096 keys 24.6
        // against 22.7, at 32 000 143.5 / 130.4, 8B shape with 128 nodes at 32 000 105 / 98, the 13B shape 16.0 / 15.5;
        // calls of one or two tiles a lane, where code is fetched cold, the same (9.6 / 9.5).
        const int x = warp - kMmaWarp0;
        constexpr uint32_t kIdescQK = instr_desc(kBN, false);
        constexpr uint32_t kIdescPV = instr_desc(D, true);
        const uint32_t q_lo = desc_lo(base + S::kOffQ, 16), k_lo0 = desc_lo(base + S::kOffK, 16), v_lo0 = desc_lo(base + S::kOffV, S::kKVPanel);
        const uint32_t s_t0 = tmem + x * 256, o_t = s_t0 + 128;
        uint32_t k_seen = 0xFFFFFFFFu;  // ring use whose K tile this warp has already seen arrive
#pragma unroll 1
        for (int i = 0; i < n_items && alive; ++i) {
            const Item it = get_item(i);
            if (it.t_begin == it.t_end) continue;
            alive = warp_wait(bar(bar_qfull()), items_run & 1u, abort_flag);
            tc_fence_after();
            bool first_pv = true;
            // The lane's tiles are t_begin + x, + 2, ...; one round issues Q K^T of a tile and P V of the one
            // before (the last round P V only).
            const int n_tiles = __shfl_sync(kFull, it.t_end - it.t_begin, 0), mine = (n_tiles - x + 1) >> 1;
            const uint32_t use0 = kt_run + static_cast<uint32_t>(x);
#pragma unroll 1
            for (int j = 0; j <= mine && mine > 0 && alive; ++j) {
                if (j < mine) {
                    const uint32_t use = use0 + 2u * j;
                    const int s = use % kStagesK;
                    if (k_seen != use && !warp_wait(bar(bar_kfull(s)), (use / kStagesK) & 1u, abort_flag)) {
                        alive = false;
                        break;
                    }
                    tc_fence_after();
                    if (elect_one()) {
                        const uint32_t k_lo = k_lo0 + s * (S::kKVTile >> 4), s_t = s_t0 + (jx & 1u) * kBN;
                        umma<kIdescQK, false>(s_t, q_lo, k_lo);
#pragma unroll
                        for (int ks = 1; ks < D / 16; ++ks)
                            umma<kIdescQK, true>(s_t, q_lo + (ks >> 2) * (S::kQPanel >> 4) + (ks & 3) * 2,
                                                 k_lo + (ks >> 2) * (S::kKVPanel >> 4) + (ks & 3) * 2);
                        umma_commit(bar(bar_sfull(x, jx & 1u)));
                        umma_commit(bar(bar_kempty(s)));
                    }
                    __syncwarp();
                    ++jx;
                }
                if (j > 0) {
                    // P V of the lane's previous tile.  While it waits for P it looks (without blocking) at
                    // the K tile of the lane's next Q K^T, whose wait would otherwise sit between P V and
                    // the next Q K^T: the chain that decides when the softmax warps get their next S.
                    const uint32_t prev_use = use0 + 2u * (j - 1), prev_j = jx - (j < mine ? 2u : 1u);
                    const uint32_t next_use = use0 + 2u * (j + 1);
                    const int s = prev_use % kStagesV;
                    alive = warp_wait(bar(bar_vfull(s)), (prev_use / kStagesV) & 1u, abort_flag);
                    if (!alive) break;
                    if (j + 1 < mine &&
                        __all_sync(kFull, mbar_test(bar(bar_kfull(next_use % kStagesK)), (next_use / kStagesK) & 1u)))
                        k_seen = next_use;
                    alive = warp_wait(bar(bar_pfull(x, prev_j & 1u)), (prev_j >> 1) & 1u, abort_flag);
                    if (alive && first_pv && items_run > 0)
                        alive = warp_wait(bar(bar_item()), (items_run - 1u) & 1u, abort_flag);
                    if (!alive) break;
                    tc_fence_after();
                    if (elect_one()) {
                        const uint32_t v_lo = v_lo0 + s * (S::kKVTile >> 4);
                        // P of keys 32h .. 32h+31: hi in columns 32h .. 32h+15, lo in 32h+16 .. 32h+31
                        const uint32_t p_t = s_t0 + (prev_j & 1u) * kBN;
#pragma unroll
                        for (int kk = 0; kk < kBN / 16; ++kk) {
                            const uint32_t a_t = p_t + (kk >> 1) * 32 + (kk & 1) * 8;
                            umma_ts<kIdescPV>(o_t, a_t, v_lo + kk * (2048 >> 4), (first_pv && kk == 0) ? 0u : 1u);
                            umma_ts<kIdescPV>(o_t, a_t + 16, v_lo + kk * (2048 >> 4), 1u);
                        }
                        umma_commit(bar(bar_pvdone(x, prev_j & 1u)));
                        umma_commit(bar(bar_vempty(s)));
                    }
                    __syncwarp();
                    first_pv = false;
                }
                // Q is free for the next item once the last QK^T of both lanes has completed
                if (j + 1 == mine && elect_one()) umma_commit(bar(bar_qempty()));
                __syncwarp();
            }
            if (alive && mine == 0 && elect_one()) umma_commit(bar(bar_qempty()));
            __syncwarp();
            kt_run += static_cast<uint32_t>(n_tiles);
            ++items_run;
        }
    }
    } else {
        // ================================ softmax warpgroup of lane x =====================
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsSoftmax));
        constexpr int kHalf = D / 2;                   // columns of a row that a lane merges
        const int x = warp >> 2;
        const int r = (warp & 3) * 32 + lane;          // row inside the tile = TMEM lane
        const uint32_t lane_sel = static_cast<uint32_t>((warp & 3) * 32) << 16;
        const uint32_t s_t = tmem + lane_sel + x * 256, o_t = s_t + 128;
        uint32_t merges = 0, meets = 0, frees = 0;     // uses of the end-of-item barriers
        bool in_use = false;                           // the cluster may still be merging the item before
        auto wait_free = [&]() {
            if (in_use) alive = __all_sync(kFull, cluster_bar_wait(bar(bar_free()), frees++ & 1u, abort_flag));
            in_use = false;
        };
#pragma unroll 1
        for (int i = 0; i < n_items && alive; ++i) {
            const Item it = get_item(i);
            const int n_tiles = it.t_end - it.t_begin;
            const bool direct = it.pieces == 1 && it.active == 1;  // one CTA has the whole group
            if (n_tiles > 0) {
                // ---- Q tile -> shared memory in the swizzled K-major layout (only when the group size does not
                // allow the TMA view): every thread's pieces are in flight together (one at a time they
                // took 8 us) --------------------------------------------------------------------------
                if constexpr (!kQByTma) {
                    constexpr int kChunks = D / 8, kPer = kBM * kChunks / kSoftmaxThreads;  // 16-byte pieces of a row, of a thread
                    uint4 v[kPer];
                    const int c = tid % kChunks;
#pragma unroll
                    for (int e = 0; e < kPer; ++e) {
                        const unsigned Rq = it.row_base + tid / kChunks + e * (kSoftmaxThreads / kChunks);
                        const unsigned t = Rq / static_cast<unsigned>(G), h = it.g * G + (Rq - t * G);
                        v[e] = make_uint4(0u, 0u, 0u, 0u);
                        if (Rq < static_cast<unsigned>(it.M))
                            v[e] = __ldg(reinterpret_cast<const uint4*>(
                                a.q + ((static_cast<int64_t>(it.b) * a.max_tt + t) * a.Hq + h) * D + c * 8));
                    }
#pragma unroll
                    for (int e = 0; e < kPer; ++e) {
                        const int row = tid / kChunks + e * (kSoftmaxThreads / kChunks);
                        *reinterpret_cast<uint4*>(base_ptr + S::kOffQ + (c >> 3) * S::kQPanel + row * 128 +
                                                  (((c & 7) ^ (row & 7)) << 4)) = v[e];
                    }
                    fence_proxy_async();
                    mbar_arrive(bar(bar_qfull()));
                }

                const int R = it.row_base + r;
                const bool row_ok = R < it.M;
                unsigned long long mlo = 0ull, mhi = 0ull;
                if (row_ok) {
                    const int t = token_of<kQByTma>(a, R, G);
                    mlo = a.mask[(static_cast<int64_t>(it.b) * a.max_tt + t) * 2 + 0];
                    mhi = a.mask[(static_cast<int64_t>(it.b) * a.max_tt + t) * 2 + 1];
                    // only nodes of this tree can be visible
                    if (it.n < 64) {
                        mlo &= (1ull << it.n) - 1ull;
                        mhi = 0ull;
                    } else if (it.n < 128) {
                        mhi &= (1ull << (it.n - 64)) - 1ull;
                    }
                }
                float m_ref = -INFINITY, l_run = 0.f;
                const int kv_len = it.L + it.n;
                bool first = true, s_loaded = false;
                uint32_t sr[2][32];
                auto load_s = [&](uint32_t buf) {
                    tc_fence_after();
                    tmem_ld32(s_t + buf * kBN, sr[0]);
                    tmem_ld32(s_t + buf * kBN + 32, sr[1]);
                };
#pragma unroll 1
                for (int t = it.t_begin + x; t < it.t_end; t += kLanes) {
                    const uint32_t buf = jx & 1u;
                    if (!s_loaded) {
                        alive = warp_wait(bar(bar_sfull(x, buf)), (jx >> 1) & 1u, abort_flag);
                        if (!alive) break;
                        load_s(buf);
                    }
                    tmem_wait_ld();

                    // ---- ancestor mask (tiles that reach past the prefix only), row maximum -------
                    const int j0 = t * kBN;
                    if (j0 + kBN > it.L) {
                        const int off = j0 - it.L;  // tile start relative to the first tree slot
                        unsigned long long allowed;
                        if (off >= 64)
                            allowed = mhi >> (off - 64);
                        else if (off > 0)
                            allowed = (mlo >> off) | (mhi << (64 - off));
                        else if (off == 0)
                            allowed = mlo;
                        else  // -64 < off < 0: the first -off keys are prefix
                            allowed = (mlo << (-off)) | ((1ull << (-off)) - 1ull);
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const uint32_t bits = static_cast<uint32_t>(allowed >> (32 * h));
#pragma unroll
                            for (int c = 0; c < 32; ++c)
                                if (!((bits >> c) & 1u)) sr[h][c] = 0xFF800000u;  // -inf
                        }
                    }
                    float t4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};  // four independent chains
#pragma unroll
                    for (int h = 0; h < 2; ++h)
#pragma unroll
                        for (int c = 0; c < 32; c += 2)
                            t4[(c >> 1) & 3] = max3(t4[(c >> 1) & 3], __uint_as_float(sr[h][c]), __uint_as_float(sr[h][c + 1]));
                    // the scale is positive: max(scale * s) = scale * max(s)
                    const float tmax = fmaxf(fmaxf(t4[0], t4[1]), fmaxf(t4[2], t4[3])) * a.scale_log2;
                    const float m_new = fmaxf(m_ref, tmax);
                    // Lazy rescale: O and l keep the old reference maximum while the true one
                    // grew by less than 2^kRescaleSlack (fp32 accumulators have the head-room).
                    const bool need = !first && (m_new > m_ref + kRescaleSlack);
                    if (first) m_ref = m_new;
                    if (__any_sync(kFull, need)) {
                        // O may only be touched once PV of the previous tile has completed
                        alive = warp_wait(bar(bar_pvdone(x, buf ^ 1u)), ((jx - 1u) >> 1) & 1u, abort_flag);
                        if (!alive) break;
                        const float corr = need ? ex2_approx(m_ref - m_new) : 1.f;
                        if (need) m_ref = m_new;
                        l_run *= corr;
                        tc_fence_after();
#pragma unroll 1
                        for (int c0 = 0; c0 < D; c0 += 32) {
                            uint32_t orr[32];
                            tmem_ld32(o_t + c0, orr);
                            tmem_wait_ld();
#pragma unroll
                            for (int c = 0; c < 32; ++c) orr[c] = __float_as_uint(__uint_as_float(orr[c]) * corr);
                            tmem_st32(o_t + c0, orr);
                        }
                        tmem_wait_st();
                    }
                    const float m_use = (m_ref == -INFINITY) ? 0.f : m_ref;

                    // ---- stale V rows of the sequence's last tile must not reach the MMA ----------
                    const bool clear_v = j0 + kBN > kv_len;
                    if (clear_v) {
                        const uint32_t use = kt_run + static_cast<uint32_t>(t - it.t_begin);
                        const int s = use % kStagesV;
                        alive = warp_wait(bar(bar_vfull(s)), (use / kStagesV) & 1u, abort_flag);
                        if (!alive) break;
                        const int valid = kv_len - j0;
                        unsigned char* vt = base_ptr + S::kOffV + s * S::kKVTile;
#pragma unroll 1
                        for (int e = r; e < (kBN - valid) * 8 * S::kPanels; e += kBM) {
                            const int row = valid + e / (8 * S::kPanels), cc = e % (8 * S::kPanels);
                            *reinterpret_cast<uint4*>(vt + (cc >> 3) * S::kKVPanel + row * 128 + ((cc & 7) << 4)) =
                                make_uint4(0u, 0u, 0u, 0u);
                        }
                        fence_proxy_async();
                    }

                    // ---- P = exp2(scale * S - m) as bf16 hi + lo, back into the columns S came from.
                    // hi is p truncated to bf16, so p - hi is exact and lo = bf16(p - hi) leaves an
                    // error of 2^-16 p.  Packed fp32 pairs halve the instruction count.  Each half of the
                    // tile (32 keys) becomes 16 columns of hi and 16 of lo in place of its own 32 columns
                    // of S, stored as soon as it is ready so that the store overlaps the other half.
                    {
                        const unsigned long long sc2 = pack2(a.scale_log2, a.scale_log2);
                        const unsigned long long nm2 = pack2(-m_use, -m_use);
                        unsigned long long psum2 = pack2(0.f, 0.f);
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            uint32_t w[32];
#pragma unroll
                            for (int c = 0; c < 16; ++c) {
                                float x0, x1;
                                unpack2(fma2(pack2(__uint_as_float(sr[h][2 * c]), __uint_as_float(sr[h][2 * c + 1])), sc2, nm2),
                                        x0, x1);
                                const float p0 = ex2_approx(x0), p1 = ex2_approx(x1);
                                const unsigned long long p2 = pack2(p0, p1);
                                psum2 = add2(psum2, p2);
                                const uint32_t b0 = __float_as_uint(p0), b1 = __float_as_uint(p1);
                                w[c] = __byte_perm(b0, b1, 0x7632);
                                float l0, l1;
                                unpack2(sub2(p2, pack2(__uint_as_float(b0 & 0xFFFF0000u), __uint_as_float(b1 & 0xFFFF0000u))),
                                        l0, l1);
                                w[16 + c] = pack_bf16(l0, l1);
                            }
                            tmem_st32(s_t + buf * kBN + h * 32, w);
                        }
                        float ps0, ps1;
                        unpack2(psum2, ps0, ps1);
                        l_run += ps0 + ps1;
                    }
                    // P is handed over at once (the tensor pipe waits for it); then S of the lane's next
                    // tile is fetched, if it has arrived (sr is free now).
                    tmem_wait_st();
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar(bar_pfull(x, buf)));
                    ++jx;
                    first = false;
                    s_loaded = t + kLanes < it.t_end &&
                               __all_sync(kFull, mbar_test(bar(bar_sfull(x, buf ^ 1u)), (jx >> 1) & 1u));
                    if (s_loaded) load_s(buf ^ 1u);
                }
                if (!alive) break;
                kt_run += static_cast<uint32_t>(n_tiles);

                // ---- end of the CTA's share.  The two lanes hold partial results over different keys for the
                // same rows; they exchange (max, sum) through shared memory and each merges one half of
                // the columns, reading the other lane's accumulator straight from tensor memory.
                const bool use_self = !first, use_oth = x == 1 || n_tiles > 1;
                if (use_self) alive = warp_wait(bar(bar_pvdone(x, (jx - 1u) & 1u)), ((jx - 1u) >> 1) & 1u, abort_flag);
                if (!alive) break;
                const float m_self = (l_run > 0.f) ? m_ref : -INFINITY;
                float2* xch = reinterpret_cast<float2*>(base_ptr + S::kOffMerge);
                xch[x * kBM + r] = make_float2(m_self, l_run);
                tc_fence_before();
                mbar_arrive(bar(bar_merge()));
                // The half row stays in registers: its largest magnitude decides the scale of a partial before
                // anything is sent.  (In pieces, in a rolled loop, with such rows sent again through the workspace:
                // 8B shape 9.0 us, 13B shape 14.9.)
                // (a lane without tiles has nothing in tensor memory: the other's is read in its place, with weight 0)
                const uint32_t both_t = tmem + lane_sel + 128 + x * kHalf;
                const uint32_t self_t = both_t + (use_self ? x : x ^ 1) * 256, oth_t = both_t + (use_oth ? x ^ 1 : x) * 256;
                // (while the other lane's result is waited for) where the chunks of the warp's rows and columns go
                uint32_t there[kHalf / 16], meet[kHalf / 16];
                if constexpr (kClusters) {
                    const uint32_t stage = base + S::kOffStage + lane * 16 + rank * a.chunk_step;
#pragma unroll
                    for (int i = 0; i < kHalf / 16; ++i) {
                        const int q = (warp & 3) * (D / 16) + x * (D / 32) + i, to = static_cast<unsigned>(q * a.cluster) / chunks_of(D);
                        there[i] = at_rank(stage + (q - chunk_at(a, to)) * kSlotBytes, to);
                        meet[i] = at_rank(bar(bar_meet()), to);
                    }
                }
                alive = warp_wait(bar(bar_merge()), merges & 1u, abort_flag);
                ++merges;
                if (!alive) break;
                tc_fence_after();
                const float2 oth = xch[(x ^ 1) * kBM + r];
                const float m_tot = fmaxf(m_self, oth.x);
                float w_self = (m_self == -INFINITY) ? 0.f : ex2_approx(m_self - m_tot);
                float w_oth = (oth.x == -INFINITY) ? 0.f : ex2_approx(oth.x - m_tot);
                const float l_tot = l_run * w_self + oth.y * w_oth;
                const float inv = (l_tot > 0.f) ? 1.f / l_tot : 0.f;
                w_self *= inv, w_oth *= inv;
                if (direct) {
                    // (in 16-column pieces, a loop of few instructions: through the registers of the other case a call of one
                    // CTA a group took 0.6 us longer)
                    const int64_t out_row = output_row<kQByTma>(a, it, r, G);
                    if (row_ok && a.lse && x == 0) a.lse[out_row] = (m_tot + log2f(l_tot)) * 0.6931471805599453f;
                    const unsigned long long ws2 = pack2(w_self, w_self), wo2 = pack2(w_oth, w_oth);
                    uint4* to = reinterpret_cast<uint4*>(a.o + out_row * D + x * kHalf);
#pragma unroll 1
                    for (int c = 0; c < kHalf; c += 16, to += 2) {
                        uint32_t r0[16], r1[16], v[8];
                        tmem_ld16(self_t + c, r0);
                        tmem_ld16(oth_t + c, r1);
                        tmem_wait_ld();
#pragma unroll
                        for (int e = 0; e < 8; ++e) {
                            const unsigned long long s2 = pack2(__uint_as_float(r0[2 * e]), __uint_as_float(r0[2 * e + 1]));
                            const unsigned long long o2 = pack2(__uint_as_float(r1[2 * e]), __uint_as_float(r1[2 * e + 1]));
                            float g0, g1;
                            unpack2(fma2(o2, wo2, fma2(s2, ws2, pack2(0.f, 0.f))), g0, g1);
                            v[e] = pack_bf16(g0, g1);
                        }
                        if (row_ok) {
                            __stcg(to, make_uint4(v[0], v[1], v[2], v[3]));
                            __stcg(to + 1, make_uint4(v[4], v[5], v[6], v[7]));
                        }
                    }
                    // O has been read: the next item's P V may overwrite it
                    tc_fence_before();
                    mbar_arrive(bar(bar_item()));
                } else {
                    float scale = 1.f;  // O = Ohat * l * scale, a scale for each half of the columns
                    uint32_t g[kHalf / 32][32];
                    // (a second time where |O / l| of a partial would leave fp16's range: the weights take a scale then)
#pragma unroll 1
                    while (true) {
                        const unsigned long long ws2 = pack2(w_self, w_self), wo2 = pack2(w_oth, w_oth);
                        float amax = 0.f;
#pragma unroll
                        for (int c = 0; c < kHalf / 32; ++c) {
                            uint32_t other[32];
                            tmem_ld32(self_t + 32 * c, g[c]);
                            tmem_ld32(oth_t + 32 * c, other);
                            tmem_wait_ld();
#pragma unroll
                            for (int e = 0; e < 32; e += 2) {
                                const unsigned long long s2 = pack2(__uint_as_float(g[c][e]), __uint_as_float(g[c][e + 1]));
                                const unsigned long long o2 = pack2(__uint_as_float(other[e]), __uint_as_float(other[e + 1]));
                                float g0, g1;
                                unpack2(fma2(o2, wo2, fma2(s2, ws2, pack2(0.f, 0.f))), g0, g1);
                                g[c][e] = __float_as_uint(g0), g[c][e + 1] = __float_as_uint(g1);
                                amax = fmaxf(fmaxf(amax, fabsf(g0)), fabsf(g1));
                            }
                        }
                        // (`!direct` holds here and only steers the compiler: without it head dimension 64 in single CTAs
                        // spills 36 bytes for 24, 16 sequences of up to 8000 keys 86.9 -> 89.1 us)
                        // (not behind an infinity: a scale for it would take the row's other values out of fp16 at the lower end)
                        const bool large = row_ok && !direct && amax > 16384.f && amax < INFINITY && scale == 1.f;
                        if (!__any_sync(kFull, large)) break;
                        if (large) {  // the next power of two above |O / l|, 2^14 down; its reciprocal by the exponent too
                            scale = __uint_as_float((__float_as_uint(amax) & 0x7F800000u) - (13u << 23));
                            const float down = __uint_as_float((254u << 23) - __float_as_uint(scale));
                            w_self *= down, w_oth *= down;
                        }
                    }
                    // O has been read: the next item's P V may overwrite it
                    tc_fence_before();
                    mbar_arrive(bar(bar_item()));
                    if (kClusters) wait_free();
                    if (!alive) break;
                    uint32_t v[kHalf / 2];
#pragma unroll
                    for (int e = 0; e < kHalf / 2; ++e)
                        v[e] = pack_half2(__uint_as_float(g[e >> 4][(2 * e) & 31]), __uint_as_float(g[e >> 4][(2 * e + 1) & 31]));
                    if constexpr (!kClusters) {
                        uint4* const po = a.part_o + static_cast<int64_t>(it.place) * (D / 8) * kBM + r + x * (kHalf / 8) * kBM;
                        float* const ml = reinterpret_cast<float*>(a.part_ml + static_cast<int64_t>(it.place) * kBM + r);
                        if (row_ok) {
#pragma unroll
                            for (int i = 0; i < kHalf / 8; ++i)
                                __stcg(po + i * kBM, make_uint4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]));
                            if (x == 0) {
                                __stcg(reinterpret_cast<float2*>(ml), make_float2(m_tot, l_tot));
                                __stcg(ml + 2, l_tot * scale);
                            } else {
                                __stcg(ml + 3, l_tot * scale);
                            }
                        }
                    } else if (it.row_base + (r & ~31) < it.M) {
                        const uint4 ml = make_uint4(__float_as_uint(m_tot), __float_as_uint(l_tot), __float_as_uint(l_tot * scale), 0u);
#pragma unroll
                        for (int i = 0; i < kHalf / 16; ++i) {
                            const int q = (warp & 3) * (D / 16) + x * (D / 32) + i, to = static_cast<unsigned>(q * a.cluster) / chunks_of(D);
                            // (with the first of the chunks that go to a CTA)
                            const bool with_rows = i == 0 || static_cast<unsigned>((q - 1) * a.cluster) / chunks_of(D) != to;
                            const uint4 v0 = make_uint4(v[8 * i], v[8 * i + 1], v[8 * i + 2], v[8 * i + 3]);
                            const uint4 v1 = make_uint4(v[8 * i + 4], v[8 * i + 5], v[8 * i + 6], v[8 * i + 7]);
                            if (to == rank) {
                                uint4* const p = reinterpret_cast<uint4*>(base_ptr + S::kOffStage + lane * 16 + rank * a.chunk_step +
                                                                          (q - chunk_at(a, rank)) * kSlotBytes);
                                p[0] = v0, p[32] = v1;
                                if (with_rows) p[64] = ml;
                            } else {
                                store_async(there[i], v0, meet[i]);
                                store_async(there[i] + 512, v1, meet[i]);
                                if (with_rows) store_async(there[i] + kChunkBytes, ml, meet[i]);
                            }
                        }
                    }
                }
            }

            if (kClusters && !direct) {
                // ---- the CTA's warps have left their own parts, the other CTAs' bytes are counted; then it merges its
                // share of all of them ----------------------------------------------------------------------
                wait_free();  // (a CTA without tiles has not waited yet)
                if (!alive) break;
                __syncwarp();
                const int q0 = chunk_at(a, rank), q1 = chunk_at(a, rank + 1);
                if (warp == 0) {
                    const int q = q0 + lane;
                    const bool own = q < q1 && it.row_base + q / (D / 16) * 32 < it.M;
                    const bool rows = own && (lane == 0 || q % (D / 32) == 0);
                    const int senders = it.active - (n_tiles > 0 ? 1 : 0);
                    const int bytes = senders * __reduce_add_sync(kFull, (own ? kChunkBytes : 0) + (rows ? kRowBytes : 0));
                    if (lane == 0) mbar_expect_tx(bar(bar_meet()), static_cast<uint32_t>(bytes));
                } else if (lane == 0) {
                    mbar_arrive(bar(bar_meet()));
                }
                MergeAt m = merge_at<D, kQByTma>(a, it, q0 + warp, q0, lane, G);
                asm volatile("" ::"r"(m.data), "r"(m.rows), "l"(m.out));  // (computed while the bytes are on their way)
                alive = __all_sync(kFull, cluster_bar_wait(bar(bar_meet()), meets & 1u, abort_flag));
                if (!alive) break;
                const unsigned char* const stage = base_ptr + S::kOffStage;
                const bool whole = kForm == kWhole || it.pieces == 1;
#pragma unroll 1
                while (m.q < q1) {
                    if (kForm == kCut && !whole) merge_chunk<D, true>(a, it, stage, m, lane, static_cast<unsigned>(cluster_id));
                    else merge_chunk<D, false>(a, it, stage, m, lane, 0u);
                    if (m.q + kPieceWarps >= q1) break;
                    m = merge_at<D, kQByTma>(a, it, m.q + kPieceWarps, q0, lane, G);
                }
                if (kForm == kCut && !whole) merge_pieces<D, kQByTma>(a, it, rank, tid, G);
                ++meets;
                if (i + 1 < n_items) {
                    __syncwarp();
                    if (lane < a.cluster) mbar_arrive_remote(bar(bar_free()), lane);
                    in_use = true;
                }
            }
            if (n_tiles > 0) {
                // (long complete: only keeps a thread from running an item ahead of the others)
                if (i + 1 < n_items) alive = warp_wait(bar(bar_item()), items_run & 1u, abort_flag);
                ++items_run;
            }
        }
        if (kClusters && alive) wait_free();  // (nobody arrives at a CTA that has left)
    }

    // ---- tear-down: every role arrives here, whatever happened ------------------------------
    if (!alive) {
        *abort_flag = 1;
        atomicOr(a.status, RESPS_STATUS_WAIT_TIMEOUT);
    }
    if (stale) atomicOr(a.status, RESPS_STATUS_STALE_PLAN);
    tc_fence_before();
    __syncthreads();
    // (the addresses count on it: the test build looks whether the swizzled tiles and tensor memory begin where they do)
    if (kWaitTest && tid == 0 && ((base & 1023u) != 0 || *reinterpret_cast<volatile uint32_t*>(base_ptr + S::kOffMisc) != tmem))
        atomicOr(a.status, RESPS_STATUS_WAIT_TIMEOUT);
    if (warp == kMmaWarp0) {
        __syncwarp();
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
    }
    // A CTA that has met the others has received their last arrival and may leave.  Where a wait has run
    // out, nobody leaves while another CTA of the cluster may still arrive on its barriers.
    if (kClusters && !alive) {
        cluster_arrive();
        cluster_wait();
        // (what the last of them sent just before it left may still be on its way: 17 us, 1500 clocks are usual)
        const uint32_t t0 = static_cast<uint32_t>(clock());
        while (static_cast<uint32_t>(clock()) - t0 < 32768u) {}
    }
}

// Combines the partials of every group that is cut into several items (modes even and stream):
// O = sum_p w_p O_p / sum_p w_p l_p with w_p = 2^(m_p - max m).
//
// The kernel is two dependent round trips to L2 (partials in, O out) behind a dependency wait, so
// what counts is how many memory requests an SM has to issue: with plain loads a warp-load is four
// 128-byte requests and an SM can only keep so many in flight.  Here a CTA takes one group x two 8-column
// pieces and lets the copy engine fetch its share of every partial (one bulk copy per partial and column
// piece, one for the (max, sum, scales) of the rows) into shared memory: a few dozen requests per CTA, all
// in flight at once.  What a CTA has to do is one entry of the work list, fetched before the wait.
constexpr int kCombineThreads = 256;
constexpr int kCombChunk = 8;       // partials fetched together; with few groups, when a CTA has an SM to itself,
constexpr int kCombChunkMost = 32;  // all of a group's up to this many
constexpr int kCombPieces = 2;  // 8-column pieces per CTA
constexpr int kCombSlotBytes = (kCombPieces + 1) * kBM * 16;  // per partial: the pieces, then (max, sum, scales)

template <int D>
__global__ void __launch_bounds__(kCombineThreads) attention_combine_kernel(const AttnArgs a) {
    constexpr int kPieces = D / 8;                    // 16-byte pieces of a row
    constexpr int kShares = kPieces / kCombPieces;    // units of work per group
    static_assert(kCombineThreads == kCombPieces * kBM, "thread = (row, piece)");
    extern __shared__ __align__(128) unsigned char comb_smem[];  // [comb_chunk][kCombSlotBytes]
    __shared__ __align__(8) unsigned long long s_bar;
    pdl_launch_dependents();
    const int tid = threadIdx.x, r = tid % kBM, cc = tid / kBM;
    const int G = a.Hq / a.Hkv;
    const uint32_t bar = smem_u32(&s_bar);
    // (the list is at least two kernels old when this kernel starts: see the note at the attention kernel)
    const int units = __ldcg(&a.plan_head->n_groups) * kShares;
    auto entry = [&](int unit, int4& lo, int& pieces) {
        const int* p = reinterpret_cast<const int*>(a.plan_group + static_cast<unsigned>(unit) / kShares);
        lo = __ldcg(reinterpret_cast<const int4*>(p)), pieces = __ldcg(p + 4);
    };
    if (static_cast<int>(blockIdx.x) >= units) return;
    int4 lo;
    int pieces;
    entry(blockIdx.x, lo, pieces);
    if (tid == 0) {
        mbar_init(bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    pdl_wait();  // the attention kernel has finished and its partials are visible
    uint32_t phase = 0;
#pragma unroll 1
    for (int unit = blockIdx.x; unit < units; unit += gridDim.x) {
        if (unit != static_cast<int>(blockIdx.x)) entry(unit, lo, pieces);
        if (pieces <= 1) continue;  // the group wrote O directly
        const int b = lo.x & 0xFFFF, g = static_cast<int>(static_cast<unsigned>(lo.x) >> 16);
        const int R0 = lo.y * kBM, nv = min(kBM, lo.z * G - R0);  // valid rows
        const int c8_0 = static_cast<int>(static_cast<unsigned>(unit) % kShares) * kCombPieces;
        float Mx = -INFINITY, den = 0.f;
        float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
        for (int p0 = 0; p0 < pieces; p0 += a.comb_chunk) {
            const int np = min(a.comb_chunk, pieces - p0);
            // one copy per thread, so that they are issued side by side: a partial's column pieces and
            // its (max, sum, scales), each nv x 16 contiguous bytes
            if (tid == 0) mbar_expect_tx(bar, static_cast<uint32_t>(np * (kCombPieces + 1) * nv * 16));
            if (tid < np * (kCombPieces + 1)) {
                const int u = tid / (kCombPieces + 1), c = tid % (kCombPieces + 1);
                const int64_t place = lo.w + p0 + u;
                const uint32_t dst = smem_u32(comb_smem + u * kCombSlotBytes + c * kBM * 16);
                const void* src = (c < kCombPieces) ? static_cast<const void*>(a.part_o + (place * kPieces + c8_0 + c) * kBM)
                                                    : static_cast<const void*>(a.part_ml + place * kBM);
                asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                             "l"(src), "r"(nv * 16), "r"(bar)
                             : "memory");
            }
            // bounded: on expiry the status word is flagged and the CTA leaves without a result
            bool ok = mbar_try(bar, phase);
            const uint32_t t0 = static_cast<uint32_t>(clock());
#pragma unroll 1
            while (!ok && static_cast<uint32_t>(clock()) - t0 <= kWaitLimitCycles) ok = mbar_try(bar, phase);
            phase ^= 1u;
            if (!__syncthreads_and(ok)) {
                if (tid == 0) atomicOr(a.status, RESPS_STATUS_WAIT_TIMEOUT);
                return;
            }
            if (r < nv) {
                float mx = Mx;
#pragma unroll 1
                for (int u = 0; u < np; ++u)
                    mx = fmaxf(mx, reinterpret_cast<const float4*>(comb_smem + u * kCombSlotBytes + kCombPieces * kBM * 16)[r].x);
                if (mx != -INFINITY) {
                    const float corr = ex2_approx(Mx - mx);  // 0 on the first chunk
                    den *= corr;
#pragma unroll
                    for (int e = 0; e < 8; ++e) acc[e] *= corr;
                    Mx = mx;
#pragma unroll 1
                    for (int u = 0; u < np; ++u) {
                        const unsigned char* sl = comb_smem + u * kCombSlotBytes;
                        const float4 ml = reinterpret_cast<const float4*>(sl + kCombPieces * kBM * 16)[r];
                        const float w = ex2_approx(ml.x - Mx);  // 0 for an empty partial, which stores zeros
                        den += ml.y * w;
                        const float wo = (c8_0 + cc < kPieces / 2 ? ml.z : ml.w) * w;  // O_p = Ohat * l * scale of this half
                        const uint4 v = reinterpret_cast<const uint4*>(sl + cc * kBM * 16)[r];
                        const uint32_t hw[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&hw[e]));
                            acc[2 * e] += f.x * wo, acc[2 * e + 1] += f.y * wo;
                        }
                    }
                }
            }
            __syncthreads();  // the next copies overwrite the staging area
        }
        if (r < nv) {
            const float inv = 1.f / den;
            const int R = R0 + r, t = R / G, h = g * G + (R - t * G);
            const int64_t row = (static_cast<int64_t>(b) * a.max_tt + t) * a.Hq + h;
            uint4 out;
            out.x = pack_bf16(acc[0] * inv, acc[1] * inv);
            out.y = pack_bf16(acc[2] * inv, acc[3] * inv);
            out.z = pack_bf16(acc[4] * inv, acc[5] * inv);
            out.w = pack_bf16(acc[6] * inv, acc[7] * inv);
            *reinterpret_cast<uint4*>(a.o + row * D + (c8_0 + cc) * 8) = out;
            if (a.lse && c8_0 + cc == 0) a.lse[row] = (Mx + log2f(den)) * 0.6931471805599453f;
        }
    }
}

// cuTensorMapEncodeTiled, resolved at run time so that the library has no link-time
// dependency on the driver (it must load on a machine without one).
using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                   const cuuint64_t*, const cuuint32_t*, const cuuint32_t*,
                                   CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                                   CUtensorMapFloatOOBfill);

EncodeTiledFn encode_tiled_fn() {
    static EncodeTiledFn fn = [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            p = nullptr;
        return reinterpret_cast<EncodeTiledFn>(p);
    }();
    return fn;
}

// (element, slot, head, sequence, panel) view of a bf16 cache; a box is 64 slots of all panels.
bool make_kv_map(CUtensorMap* map, const void* basep, int D, int64_t capacity, int Hkv, int batch,
                 int64_t s_tok, int64_t s_head, int64_t s_seq) {
    EncodeTiledFn fn = encode_tiled_fn();
    if (!fn) return false;
    // a dimension of extent 1 never uses its stride; give it a valid one
    if (s_head <= 0) s_head = capacity * s_tok;
    if (s_seq <= 0) s_seq = s_head * Hkv;
    const cuuint32_t panels = static_cast<cuuint32_t>(D / 64);
    const cuuint64_t dims[5] = {64, static_cast<cuuint64_t>(capacity), static_cast<cuuint64_t>(Hkv),
                                static_cast<cuuint64_t>(batch), panels};
    const cuuint64_t strides[4] = {static_cast<cuuint64_t>(s_tok) * 2, static_cast<cuuint64_t>(s_head) * 2,
                                   static_cast<cuuint64_t>(s_seq) * 2, 128};
    const cuuint32_t box[5] = {64, static_cast<cuuint32_t>(kBN), 1, 1, panels};
    const cuuint32_t estr[5] = {1, 1, 1, 1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void*>(basep), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// (element, head in group, KV head, token of any sequence, panel) view of Q [batch][max_tt][Hq][D]:
// a box of 64 elements x G heads x 128/G tokens x all panels is one 128-row tile in (token, head)
// row order.  The sequences are folded into the token dimension (they are contiguous), so rows
// past a sequence's max_tt read the next sequence's; such rows are never valid.
bool make_q_map(CUtensorMap* map, const void* basep, int D, int G, int Hkv, int max_tt, int batch) {
    EncodeTiledFn fn = encode_tiled_fn();
    if (!fn) return false;
    const cuuint64_t Hq = static_cast<cuuint64_t>(G) * Hkv;
    const cuuint32_t panels = static_cast<cuuint32_t>(D / 64);
    const cuuint64_t dims[5] = {64, static_cast<cuuint64_t>(G), static_cast<cuuint64_t>(Hkv),
                                static_cast<cuuint64_t>(max_tt) * batch, panels};
    const cuuint64_t strides[4] = {static_cast<cuuint64_t>(D) * 2, static_cast<cuuint64_t>(G) * D * 2, Hq * D * 2, 128};
    const cuuint32_t box[5] = {64, static_cast<cuuint32_t>(G), 1, static_cast<cuuint32_t>(kBM / G), panels};
    const cuuint32_t estr[5] = {1, 1, 1, 1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void*>(basep), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Tensor maps are kept per context, keyed by everything that goes into them: a decode loop calls
// with the same few buffers over and over, and encoding a map is a driver call.
struct MapKey {
    const void* base;
    int64_t a, b, c, d;  // K/V: token, head, sequence strides and capacity; Q: G, max_tt, 0, 0
    int hkv, batch, kind;  // kind 0: K/V cache, 1: Q
    bool operator==(const MapKey& o) const {
        return base == o.base && a == o.a && b == o.b && c == o.c && d == o.d && hkv == o.hkv && batch == o.batch &&
               kind == o.kind;
    }
};
struct MapKeyHash {
    size_t operator()(const MapKey& k) const {
        uint64_t h = reinterpret_cast<uintptr_t>(k.base) * 0x9E3779B97F4A7C15ull;
        h ^= (static_cast<uint64_t>(k.a) * 31 + k.b) * 0xBF58476D1CE4E5B9ull + k.c + k.d * 7 + k.batch * 131 + k.kind +
             k.hkv * 8191;
        return static_cast<size_t>(h ^ (h >> 29));
    }
};
struct HostState {
    std::mutex mu;
    std::unordered_map<MapKey, CUtensorMap, MapKeyHash> maps;
    // The work list in the workspace was made for these arguments ...
    bool plan_valid = false;
    const resps_step* plan_steps = nullptr;
    const int32_t* plan_n_nodes = nullptr;
    int plan_batch = 0;
    int64_t plan_capacity = 0;
    cudaStream_t plan_stream = nullptr;
    // ... and this many kernels of the library have been enqueued behind the one that wrote it.
    int plan_age = 0;
    int resident[kMaxCluster + 1] = {};  // clusters of each size that are resident at once
};
constexpr size_t kMaxCachedMaps = 4096;

HostState* host_state(const resps_ctx* ctx) { return static_cast<HostState*>(ctx->attn_host); }

// Copies the map into `out`: a map inserted later may clear the table.  False where the map cannot be encoded or
// there is no host memory for its entry (no exception may leave the C entry points).
bool cached_map(HostState* hs, const MapKey& key, int D, CUtensorMap* out) {
    const auto it = hs->maps.find(key);
    if (it != hs->maps.end()) {
        *out = it->second;
        return true;
    }
    const bool ok = key.kind == 0 ? make_kv_map(out, key.base, D, key.d, key.hkv, key.batch, key.a, key.b, key.c)
                                  : make_q_map(out, key.base, D, static_cast<int>(key.a), key.hkv,
                                               static_cast<int>(key.b), key.batch);
    if (!ok) return false;
    if (hs->maps.size() >= kMaxCachedMaps) hs->maps.clear();
    try {
        hs->maps.emplace(key, *out);
    } catch (const std::bad_alloc&) {
        return false;
    }
    return true;
}

// CTAs per cluster for mode whole, or 1 for the two-kernel modes.  The launch shape is fixed before the tree and the
// prefix are known (a captured step is replayed for any), so it goes by what both can be: `groups` of the largest tree
// of the context and the longest prefix of the cache.  Mode whole saves the second kernel and pays with CTAs that stay
// without work: clusters of C CTAs for `groups` (smaller trees have their groups cut over the clusters left).  For kt
// key tiles that is kt (1 / C - groups / SMs) tiles a CTA.  Measured, whole / two kernels, in us a layer (largest tree
// of each context, prefix 1024, 2048, 4096, 8192):
//    8 groups, C = 8    7.8 /  9.1    9.1 / 10.5   11.4 / 12.4   16.0 / 14.9
//   12         8        9.5 / 10.6   10.7 / 11.6   12.6 / 13.3   16.9 / 16.4   (Q by plain loads)
//   16         6        8.3 /  9.7    9.8 / 11.0   12.6 / 13.2   18.5 / 17.0
//   24         5        9.0 / 11.4   10.5 / 13.3   14.3 / 16.0   20.7 / 21.7   (28.4 / 28.3 at 12 288)
//   32         4        9.4 / 11.8   11.5 / 13.8   15.8 / 17.9   24.8 / 26.1   (35.0 / 36.2)
//   40         3       11.1 / 11.9   14.0 / 14.9   20.1 / 21.1   33.7 / 35.3   (47.8 / 48.0)
// At the longest prefix that 5, 6 and 7 lost tiles admit (a cache without room beyond it), whole / two kernels:
//    8 groups   11.0 / 12.7   12.1 / 13.3   13.1 / 14.0  (6240 keys)
//   12          15.8 / 15.9   17.0 / 17.0   18.5 / 18.0  (10 129)
//   16          14.6 / 14.4   16.0 / 15.5   17.8 / 16.7  (7556; Q by plain loads 15.9 / 15.5, 17.1 / 16.6, 18.7 / 17.6)
//   24          21.4 / 22.1   24.3 / 24.9   28.2 / 27.5  (11 744)
//   32          27.5 / 28.7   32.3 / 34.1   37.1 / 38.6  (13 120)
//   40          23.7 / 25.8   26.6 / 30.0   29.6 / 33.8  (7056)
// With 7 a call at that limit takes up to 6 % longer than the two kernels would (16 groups), and one of 1024 keys in such a
// cache, where calls usually are well below its end, 11 to 21 % less (16 groups 8.2 / 9.6, 24 9.1 / 11.5).
constexpr double kWholeGainTiles = 7.0;
// In a batch the cache may hold one long sequence among short ones, which only its own clusters work on.  (Four equal
// sequences of 8 groups: 10.4 / 12.9 us at 1024 keys, 40.5 / 43.6 at 12 288.)
int choose_cluster(const int* resident, int sm_count, int groups, int batch, int kt_most) {
    for (int c : {8, 6, 5, 4, 3, 2}) {
        if (resident[c] < groups) continue;
        const double lost = 1.0 / c - static_cast<double>(groups / batch) / sm_count;
        if (lost * kt_most <= kWholeGainTiles) return c;
    }
    return 1;
}
// K and V of this many bytes are taken to stay in L2 between the row tiles of a head (measured between 67 and 131 MB).
// With a head dimension of 64 it does not matter where they are: 148 CTAs with 16 KB per 0.6 us ask for 4 TB/s, below
// HBM's rate, where 32 KB per 0.57 us ask for 8.5.  (16 sequences up to 32 000 keys, 546 MB, ranges / the best of two to four
// rounds of equal splits: trees of up to 32 nodes 135.7 / 138.5, 135.6 / 143.8, 135.2 / 146 us, up to 96 nodes 248 / 244,
// 279 / 307, 314 / 302.  Four of six lose 2 to 10 %, two gain 2 to 4 %, so rounds are not looked at there.)
constexpr int64_t kL2Bytes = 96 << 20;
int forced_cluster(const int* resident, int cluster, int groups) {
    while (cluster > 1 && resident[cluster] < groups) --cluster;
    return cluster;
}
// Nodes of the largest tree a context builds: min(max_tt, 1 + n_cand).
int most_nodes(const resps_shape& s) {
    return static_cast<int>(std::min<int64_t>(s.max_tt, 1 + s.max_k + static_cast<int64_t>(s.max_depth - 1) * s.max_k * s.max_k));
}

// Clusters of C CTAs that are resident at once with this kernel's shared memory (index C; the GPCs are not
// multiples of every size), asked for once per device.  One answer serves all forms of a head dimension: they have the
// same threads, registers (the launch bound's) and shared memory, of which one CTA takes more than half an SM's.
struct Residency {
    int clusters[kMaxCluster + 1] = {};
    bool known = false;
};
std::mutex g_residency_mu;
Residency g_residency[2][64];  // [head dim 64, 128][device]

// Q tiles come by TMA where a row tile is whole tokens.
bool group_by_tma(int G) { return G <= kBM && kBM % G == 0; }

using AttnKernel = void (*)(AttnArgs, CUtensorMap, CUtensorMap, CUtensorMap);
template <int D>
AttnKernel form_of(int form, bool q_by_tma) {
    switch (form) {
        case kSingles: return q_by_tma ? tree_attention_kernel<D, kSingles, true> : tree_attention_kernel<D, kSingles, false>;
        case kWhole: return q_by_tma ? tree_attention_kernel<D, kWhole, true> : tree_attention_kernel<D, kWhole, false>;
        default: return q_by_tma ? tree_attention_kernel<D, kCut, true> : tree_attention_kernel<D, kCut, false>;
    }
}

template <int D>
cudaError_t launch_for_dim(const resps_ctx* ctx, const AttnArgs& a, int grid, const CUtensorMap& mk, const CUtensorMap& mv,
                           const CUtensorMap& mq, cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid), cfg.blockDim = dim3(kAttnThreads), cfg.stream = st;
    cfg.dynamicSmemBytes = a.cluster > 1 ? Smem<D>::kClusterBytes : Smem<D>::kBytes;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = static_cast<unsigned>(a.cluster), attr[1].val.clusterDim.y = 1, attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr, cfg.numAttrs = a.cluster > 1 ? 2 : 1;
    cudaError_t e = cudaLaunchKernelEx(&cfg, form_of<D>(a.cluster == 1 ? kSingles : a.may_cut ? kCut : kWhole, a.q_by_tma != 0), a, mk, mv, mq);
    if (e != cudaSuccess || a.cluster > 1) return e;
    // the units of work of the largest trees, at most one resident round of CTAs
    const int64_t units = static_cast<int64_t>(a.batch) * a.Hkv * ((a.max_tt * (a.Hq / a.Hkv) + kBM - 1) / kBM) * (D / 8 / kCombPieces);
    const int combine_grid = static_cast<int>(std::min<int64_t>(units, 4 * ctx->sm_count));
    return launch_pdl(attention_combine_kernel<D>, dim3(combine_grid), dim3(kCombineThreads), a.comb_chunk * kCombSlotBytes, st, a);
}

template <int D>
cudaError_t setup_for_dim(int device, int sm_count, bool q_by_tma, int* clusters) {
    cudaError_t e = cudaSuccess;
    for (int form : {kSingles, kWhole, kCut}) {
        e = cudaFuncSetAttribute(form_of<D>(form, q_by_tma), cudaFuncAttributeMaxDynamicSharedMemorySize, Smem<D>::kClusterBytes);
        if (e != cudaSuccess) return e;
    }
    e = cudaFuncSetAttribute(attention_combine_kernel<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, kCombChunkMost * kCombSlotBytes);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lock(g_residency_mu);
    Residency local;
    Residency& r = (device >= 0 && device < 64) ? g_residency[D == 128][device] : local;
    if (!r.known) {
        r.clusters[1] = std::min(sm_count, kMaxGrid);
        for (int c = 2; c <= kMaxCluster; ++c) {
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(static_cast<unsigned>(sm_count / c * c)), cfg.blockDim = dim3(kAttnThreads);
            cfg.dynamicSmemBytes = Smem<D>::kClusterBytes;
            cudaLaunchAttribute attr[1];
            attr[0].id = cudaLaunchAttributeClusterDimension;
            attr[0].val.clusterDim.x = static_cast<unsigned>(c), attr[0].val.clusterDim.y = 1, attr[0].val.clusterDim.z = 1;
            cfg.attrs = attr, cfg.numAttrs = 1;
            int n = 0;
            e = cudaOccupancyMaxActiveClusters(&n, form_of<D>(kWhole, q_by_tma), &cfg);
            if (e != cudaSuccess) return e;
            r.clusters[c] = std::min(n, kMaxGrid / c);
        }
        r.known = true;
    }
    for (int c = 1; c <= kMaxCluster; ++c) clusters[c] = r.clusters[c];
    return cudaSuccess;
}

}  // namespace

cudaError_t attention_setup(resps_ctx* ctx) {
    HostState* hs = new (std::nothrow) HostState();
    if (!hs) return cudaErrorMemoryAllocation;
    ctx->attn_host = hs;
    const bool q_by_tma = group_by_tma(ctx->shape.n_q_heads / ctx->shape.n_kv_heads);
    return ctx->shape.head_dim == 128 ? setup_for_dim<128>(ctx->device, ctx->sm_count, q_by_tma, hs->resident)
                                      : setup_for_dim<64>(ctx->device, ctx->sm_count, q_by_tma, hs->resident);
}

void attention_teardown(resps_ctx* ctx) {
    delete host_state(ctx);
    ctx->attn_host = nullptr;
}

// The step parameters or node counts behind `steps` may have changed (or the scheduling knobs
// have): the next attention call derives its work list anew.
void attention_plan_invalidate(resps_ctx* ctx, const void* steps_or_null) {
    HostState* hs = host_state(ctx);
    if (!hs) return;
    std::lock_guard<std::mutex> lock(hs->mu);
    if (steps_or_null == nullptr || steps_or_null == hs->plan_steps || steps_or_null == hs->plan_n_nodes)
        hs->plan_valid = false;
}

cudaError_t launch_tree_attention(const resps_ctx* ctx, const resps_step* d_steps,
                                  const int32_t* d_n_nodes, int batch, const __nv_bfloat16* q,
                                  __nv_bfloat16* o, float* lse, const __nv_bfloat16* k_cache,
                                  const __nv_bfloat16* v_cache, int64_t stride_seq,
                                  int64_t stride_head, int64_t stride_tok, int64_t capacity,
                                  const uint64_t* mask, float scale, cudaStream_t st) {
    const Workspace& w = ctx->ws;
    AttnArgs a;
    a.steps = d_steps, a.n_nodes = d_n_nodes, a.batch = batch;
    a.q = q, a.o = o, a.lse = lse;
    a.capacity = capacity;
    a.mask = mask;
    a.scale_log2 = scale * 1.4426950408889634f;
    a.Hq = ctx->shape.n_q_heads, a.Hkv = ctx->shape.n_kv_heads, a.max_tt = ctx->shape.max_tt;
    a.part_o = reinterpret_cast<uint4*>(w.attn_part_o), a.part_ml = w.attn_part_ml;
    a.max_items = w.attn_max_items;
    a.status = w.status;
    a.piece_count = w.attn_count;
    unsigned char* plan = w.attn_plan;
    a.plan_head = reinterpret_cast<PlanHead*>(plan), plan += sizeof(PlanHead);
    a.plan_cluster = reinterpret_cast<PlanCluster*>(plan), plan += sizeof(PlanCluster) * kMaxGrid;
    a.plan_first = reinterpret_cast<PlanItem*>(plan), plan += sizeof(PlanItem) * kMaxGrid;
    a.plan_item = reinterpret_cast<PlanItem*>(plan), plan += sizeof(PlanItem) * w.attn_max_items * kMaxCluster;
    a.plan_group = reinterpret_cast<PlanGroup*>(plan);
    a.test_drop = w.test_drop;
    const int D = ctx->shape.head_dim;
    const int G = a.Hq / a.Hkv;
    a.q_by_tma = group_by_tma(G) ? 1 : 0;
    a.log2_group = 0;
    while ((2 << a.log2_group) <= G) ++a.log2_group;
    HostState* hs = host_state(ctx);
    std::lock_guard<std::mutex> lock(hs->mu);
    // the most groups of a tree this context builds (attention over larger ones is correct, and slower)
    const int groups = batch * a.Hkv * ceil_div(most_nodes(ctx->shape) * G, kBM);
    a.cluster = choose_cluster(hs->resident, ctx->sm_count, groups, batch, static_cast<int>((capacity + kBN - 1) / kBN));
    if (w.attn_cluster > 0) a.cluster = forced_cluster(hs->resident, std::min(w.attn_cluster, kMaxCluster), groups);
    a.clusters = a.cluster > 1 ? groups : hs->resident[1];
    a.min_tiles = w.attn_min_tiles > 0 ? w.attn_min_tiles : a.cluster > 1 ? 1 : 2;
    const int grid = a.clusters * a.cluster;
    a.chunk_first = 0, a.chunk_step = chunks_most(D, a.cluster) * kSlotBytes;
    for (int c = 0; c <= a.cluster; ++c) a.chunk_first |= static_cast<unsigned long long>(first_chunk(D, a.cluster, c)) << (7 * c);
    // the pieces of cut groups lie where the two-kernel modes have partials (72 bytes a unit against 32)
    a.may_cut = a.cluster > 1 && groups > batch * a.Hkv && (9 * a.clusters + 3) / 4 <= a.max_items &&
                (w.attn_stream > 0 || (w.attn_stream < 0 && (capacity + kBN - 1) / kBN > kPieceTiles * a.cluster)) ? 1 : 0;
    a.piece_acc = reinterpret_cast<float4*>(a.part_o);
    a.piece_ml = reinterpret_cast<float2*>(a.piece_acc + static_cast<int64_t>(a.clusters) * 4 * kBM * (D / 16));
    if (w.attn_rounds > 0 && a.cluster == 1) a.clusters = std::max(1, a.clusters / w.attn_rounds);
    // one resident round of units with room for all of a group's partials, else more CTAs per SM
    a.comb_chunk = groups * (D / 8 / kCombPieces) <= ctx->sm_count ? kCombChunkMost : kCombChunk;
    a.stream_gain = w.attn_stream, a.rounds = w.attn_even_rounds;
    a.most_rounds = D == 128 ? kMaxRounds : 1;
    a.l2_tiles = D == 128 ? static_cast<int>(kL2Bytes / (2 * 2 * kBN * D)) : 1 << 30;
    MapKey kk = {k_cache, stride_tok, stride_head, stride_seq, capacity, a.Hkv, batch, 0};
    MapKey kv = kk;
    kv.base = v_cache;
    CUtensorMap mk, mv, mq;
    if (!cached_map(hs, kk, D, &mk) || !cached_map(hs, kv, D, &mv)) return cudaErrorInvalidValue;
    if (a.q_by_tma) {
        const MapKey kq = {q, G, a.max_tt, 0, 0, a.Hkv, batch, 1};
        if (!cached_map(hs, kq, D, &mq)) return cudaErrorInvalidValue;
    } else {
        mq = mk;  // unused by the kernel
    }
    // The work list: made by the first call after anything that may have changed the step, reused
    // by the calls for the other layers.
    const bool reuse = hs->plan_valid && hs->plan_steps == d_steps && hs->plan_n_nodes == d_n_nodes &&
                       hs->plan_batch == batch && hs->plan_capacity == capacity && hs->plan_stream == st;
    if (!reuse) {
        cudaError_t e = launch_pdl(attention_plan_kernel, dim3(1), dim3(kMaxGrid), 0, st, a);
        if (e != cudaSuccess) return e;
        hs->plan_valid = true, hs->plan_steps = d_steps, hs->plan_n_nodes = d_n_nodes, hs->plan_batch = batch;
        hs->plan_capacity = capacity, hs->plan_stream = st, hs->plan_age = 0;
    }
    a.plan_after_wait = hs->plan_age == 0 ? 1 : 0;
    cudaError_t e = D == 128 ? launch_for_dim<128>(ctx, a, grid, mk, mv, mq, st) : launch_for_dim<64>(ctx, a, grid, mk, mv, mq, st);
    hs->plan_age += a.cluster > 1 ? 1 : 2;
    return e;
}

int attention_max_batch() { return kMaxBatch; }
int attention_place_rows() { return kBM; }
int attention_max_groups(int batch, int n_kv_heads, int max_tt, int group) {
    return batch * n_kv_heads * ((max_tt * group + kBM - 1) / kBM);
}
int attention_counters() { return kMaxGrid * kPieceWarps; }
// Items of the two-kernel modes, also the most partials: a round of splits or a range a CTA (which may begin inside a
// group), and up to kMaxRounds rounds.  Up to kFewGroups groups one round is balanced to within a seventh: such contexts have
// no room for more.  (The sums of cut groups in clusters, 9/4 places a cluster, lie in the same memory; the launch checks that
// they fit.)
constexpr int kFewGroups = 20;
int attention_max_items(int groups, int sm_count) {
    const int grid = std::min(sm_count, kMaxGrid);
    return std::max(groups, groups <= kFewGroups ? grid : (kMaxRounds - 1) * grid) + grid;
}
size_t attention_plan_bytes(int max_items, int max_groups) {
    return sizeof(PlanHead) + sizeof(PlanCluster) * kMaxGrid + sizeof(PlanItem) * (kMaxGrid + static_cast<size_t>(max_items) * kMaxCluster) +
           sizeof(PlanGroup) * static_cast<size_t>(max_groups);
}

}  // namespace resps
