// Draft-tree build from the scanned rows (Section 3.2, "Draft Tree Expansion":
// cumulative score V_i along the root path, the k best of a layer are expanded;
// "Confidence-Based Candidate Reranking": all expanded tokens are reranked and the
// best TT-1 kept; Algorithm 2, tree-building loop).  One CTA per sequence; integer
// and fp64 work on at most k + (d-1)k^2 candidates, all in shared memory.
//
// A level's candidates are k lists (one per frontier member), each already in the method's order
// because a scanned row is sorted.  The next frontier is the k best of them: one warp takes the best
// list head k times.  The rerank is a selection over all candidates by a histogram of the scores.
//
// Bound by latency: one CTA per sequence and a chain of small dependent steps.  What is kept short is
// the chain, and what is avoided is work that grows with k^3: ranking every candidate of a level
// against every other list (k^3 searches a level) took 598 us at TT=128, d=8, k=32 (7200 candidates).
#include <cmath>

#include "common.cuh"

namespace resps {
namespace {

constexpr int kTreeThreads = 512;
constexpr unsigned kFull = 0xFFFFFFFFu;
constexpr int kLevelThreads = 256;  // a launch that ranks one level only (level form)
constexpr int kBins = kTreeThreads;         // steps of score in the rerank's histogram
constexpr int kTieList = 256;       // candidates of one step that are ranked by counting
constexpr double kLowest = -1e30;   // log-probabilities stay finite

struct TreeShared {
    int kept[RESPS_MAX_TT];  // candidates kept by the rerank, in no order
    int hist[kBins];
    int list[kTieList];
    int parent[RESPS_MAX_TT], depth[RESPS_MAX_TT], has_child[RESPS_MAX_TT], row[RESPS_MAX_TT];
    int warp_sum[32];
    int n_kept, n_list, cut, cut_before, cut_count;
    long long low, high;
};

struct TreeArgs {
    const resps_step* steps;
    int n_levels, n_slots;
    int vocab, max_tt, max_k, max_depth, max_rows;
    const float* row_val;
    const int32_t* row_id;
    const double* row_lse;
    const int32_t* root_token;
    int32_t *tokens, *parent, *depth, *position_ids;
    uint64_t* mask;
    int32_t *retrieve, *n_leaves, *n_nodes;
    int32_t* node_row;  // workspace [batch][max_tt]: level * RESPS_MAX_K + slot of the draft row a node's children came from
    int32_t* status;
    int cand_cap;  // candidates the shared-memory arrays hold
    // Level form: emit_level = j >= 0 ranks the levels up to j from the rows scanned so far, hands out
    // the frontier after level j and stops; -1 builds the whole tree.
    int emit_level;
    FrontierOut fr;
    // Frontiers of the levels ranked so far [batch][RESPS_MAX_DEPTH][RESPS_MAX_K] (level form: every call
    // ranks one level and leaves its frontier here; use_state = 1 reads it).
    int32_t* state_frontier;
    double* state_score;
    int use_state;
    int setup_before_wait;  // 1: a scan or merge kernel of the same call runs directly before this kernel
};

// Path scores as integers, for the warp-wide maximum and the shared-memory minimum: the map keeps the
// order of finite doubles (and their equality, zero being stored as +0) and is its own inverse.
__device__ __forceinline__ long long score_key(double s) {
    const long long bits = __double_as_longlong(s + 0.0);
    return bits ^ ((bits >> 63) & 0x7FFFFFFFFFFFFFFFll);
}
__device__ __forceinline__ double key_score(long long key) {
    return __longlong_as_double(key ^ ((key >> 63) & 0x7FFFFFFFFFFFFFFFll));
}

// Exact floor(e / d) for 0 <= e < 2^22 and 1 <= d <= 2^10: the quotient's fraction is at least
// 0.5 / d away from an integer after the half is added, far more than the float rounding.
struct FastDiv {
    float inv;
    __device__ explicit FastDiv(int d) : inv(1.0f / static_cast<float>(d)) {}
    __device__ __forceinline__ int div(int e) const { return __float2int_rd((static_cast<float>(e) + 0.5f) * inv); }
};

__global__ void __launch_bounds__(kTreeThreads, 1) tree_build_kernel(const TreeArgs a) {
    // The step parameters were written at least two kernels ago (a scan or a merge kernel of the same
    // call always sits between their writer and this kernel, and signals its dependents only after its
    // own wait), so they are read, and everything that follows from them is
    // set up, before the wait for the rows: under the tail of the kernel that scans them.  (Where no such
    // kernel precedes this one -- the last call of the level form -- the wait comes first.)
    if (!a.setup_before_wait) pdl_wait();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nthreads = blockDim.x;
    const StepDims sd = clamp_step(a.steps[b], a.n_levels, a.n_slots, a.max_tt, a.max_k, a.vocab);
    const int k = sd.k, kk = k * k;
    const int d = (a.emit_level >= 0) ? min(sd.d, a.emit_level + 1) : sd.d;  // levels ranked by this launch
    const int n_cand = k + (d - 1) * kk;
    const int m = min(sd.tt - 1, n_cand);
    const int n = m + 1;

    double* score = reinterpret_cast<double*>(smem_raw);                  // [cand_cap] own log-prob, then the path score
    double* fscore = score + a.cand_cap;                                  // [max_depth][max_k] frontier scores
    int* node_of = reinterpret_cast<int*>(fscore + RESPS_MAX_DEPTH * RESPS_MAX_K);  // [cand_cap] node index of a kept candidate
    int* frontier = node_of + a.cand_cap;                                 // [max_depth][max_k] candidates
    __shared__ TreeShared sh;

    // Index arithmetic by the run-time k and k^2 goes through an exact float reciprocal (operands stay
    // below 2^22).
    const FastDiv by_k(k), by_kk(kk);
    const int64_t row0 = static_cast<int64_t>(b) * a.max_rows;
    struct Cand {
        int level, list, place;  // level, list inside the level (frontier slot of the parent), place in the list
    };
    auto decode = [&](int c) {
        Cand r;
        if (c < k) {
            r.level = 0, r.list = 0, r.place = c;
        } else {
            const int t = c - k, jm1 = by_kk.div(t), i = t - jm1 * kk;
            r.level = jm1 + 1;
            r.list = by_k.div(i);
            r.place = i - r.list * k;
        }
        return r;
    };
    auto parent_of = [&](int c) {  // the parent's place in the frontier arrays, -1: the root
        if (c < k) return -1;
        const int t = c - k, jm1 = by_kk.div(t);
        return jm1 * RESPS_MAX_K + by_k.div(t - jm1 * kk);
    };
    auto cand_row = [&](const Cand& r) { return (r.level == 0) ? 0 : 1 + (r.level - 1) * k + r.list; };

#pragma unroll 1
    for (int i = tid; i < kBins; i += nthreads) sh.hist[i] = 0;
    if (tid < RESPS_MAX_TT) sh.kept[tid] = 0x7FFFFFFF, sh.has_child[tid] = 0, sh.row[tid] = -1;
    if (tid == 0) sh.n_kept = 0;
    // Level form: a call ranks one level, the last call none; what the calls before left in the workspace
    // is read instead (levels >= 1; level 0 is the first row itself).
    const int first_level = (a.emit_level >= 0) ? a.emit_level : 0;  // the first level this launch needs the rows of
    const int c_first = (first_level == 0) ? 0 : k + (first_level - 1) * kk;
    const int64_t state0 = static_cast<int64_t>(b) * RESPS_MAX_DEPTH * RESPS_MAX_K;
    constexpr int kAhead = 4;  // candidates a thread loads together; the first ones are located before the wait
    int64_t at_row[kAhead], at[kAhead];
    auto locate = [&](int c0) {
#pragma unroll
        for (int u = 0; u < kAhead; ++u) {
            const Cand r = decode(min(c0 + u * nthreads, n_cand - 1));
            at_row[u] = row0 + cand_row(r);
            at[u] = at_row[u] * a.max_k + r.place;
        }
    };
    locate(c_first + tid);
    const int own_parent = parent_of(tid);
    if (a.setup_before_wait) pdl_wait();  // the kernel before this one in the stream has completed: the scanned rows are there
    pdl_launch_dependents();
    if (a.emit_level >= 0 && a.emit_level >= sd.d) {
        // (a sequence whose own d is below j + 1 has nothing at this level: its entries stay untouched)
        if (tid == 0 && sd.clamped) atomicOr(a.status, RESPS_STATUS_STEP_CLAMPED);
        return;
    }
    if (a.use_state) {
        const int known = (a.emit_level >= 0) ? a.emit_level : d;  // levels ranked by earlier calls
#pragma unroll 1
        for (int i = tid; i < known * RESPS_MAX_K; i += nthreads) {
            frontier[i] = a.state_frontier[state0 + i];
            fscore[i] = a.state_score[state0 + i];
        }
    }
    // ---- every candidate's own log-probability, in one round trip to global memory (the rows
    // a level reads do not depend on the levels before it) ------------------------------------------
#pragma unroll 1
    for (int c0 = c_first + tid; c0 < n_cand; c0 += kAhead * nthreads) {
        float val[kAhead];
        double lse[kAhead];
        if (c0 != c_first + tid) locate(c0);
#pragma unroll
        for (int u = 0; u < kAhead; ++u) {
            if (c0 + u * nthreads < n_cand) val[u] = a.row_val[at[u]], lse[u] = a.row_lse[at_row[u]];
        }
#pragma unroll
        for (int u = 0; u < kAhead; ++u) {
            const int c = c0 + u * nthreads;
            if (c < n_cand) score[c] = fmax(fmin(static_cast<double>(val[u]) - lse[u], 0.0), kLowest) + 0.0;
        }
    }
    __syncthreads();

    // ---- frontiers: one warp walks the levels.  A level's candidates are k lists (one per frontier
    // member) already in the method's order, because a scanned row is sorted, and only the k best of the
    // level are needed: lane p holds the head of list p, and k times the best head is taken (ties by the
    // lower lane, which has the lower candidate indices).  No block-wide barrier in the chain, no branch
    // on a lane's own data, and the entry behind a head is made ready in the shadow of the reduction:
    // about 150 cycles an entry (an insertion into the order of the heads took 420, a binary search of
    // every candidate in every other list 4000-25000 a level, against 1900 for k = 10 and 4800 for k = 32).
    if (warp == 0) {
        if (first_level == 0) {
            if (lane < k) frontier[lane] = lane, fscore[lane] = score[lane];
            __syncwarp();
        }
        const int j0 = (a.use_state && a.emit_level < 0) ? d : max(first_level, 1);
#pragma unroll 1
        for (int j = j0; j < d; ++j) {
            constexpr long long kNone = static_cast<long long>(0x8000000000000000ull);
            const bool on = lane < k;
            const int base = k + (j - 1) * kk;
            const double parent = on ? fscore[(j - 1) * RESPS_MAX_K + lane] : 0.0;
            const double* list = score + base + lane * k;
            double head_score = on ? list[0] + parent : 0.0;
            long long head = on ? score_key(head_score) : kNone;
            double next = (on && k > 1) ? list[1] : 0.0;
            int place = 0;
            const unsigned lower_lanes = (1u << lane) - 1u;
#pragma unroll 1
            for (int r = 0; r < k; ++r) {
                const int hi = static_cast<int>(head >> 32);
                const int top_hi = __reduce_max_sync(kFull, hi);
                unsigned best = __ballot_sync(kFull, hi == top_hi);
                const double next_score = next + parent;
                const long long next_key = (on && place + 1 < k) ? score_key(next_score) : kNone;
                if (best & (best - 1)) {  // the same upper half more than once: the lower half decides
                    const bool in = hi == top_hi;
                    const unsigned lo = in ? static_cast<unsigned>(head) : 0u;
                    const unsigned top_lo = __reduce_max_sync(kFull, lo);  // (every lane takes part)
                    best = __ballot_sync(kFull, in && lo == top_lo);
                }
                const bool win = ((best >> lane) & 1u) && !(best & lower_lanes);
                if (win) {
                    frontier[j * RESPS_MAX_K + r] = base + lane * k + place;
                    fscore[j * RESPS_MAX_K + r] = head_score;
                }
                head = win ? next_key : head;
                head_score = win ? next_score : head_score;
                place += win ? 1 : 0;
                if (win) next = list[min(place + 1, k - 1)];
            }
            __syncwarp();
        }
        if (a.emit_level < 0) {
            // a lower bound of the rerank's m-th best, if the frontiers alone hold m candidates: their
            // worst member (the lower half of its key cleared)
            const int mine = (lane < d) ? static_cast<int>(score_key(fscore[lane * RESPS_MAX_K + k - 1]) >> 32) : 0x7FFFFFFF;
            const int least = __reduce_min_sync(kFull, mine);
            if (lane == 0) sh.low = static_cast<long long>(least) << 32;
        }
    }
    __syncthreads();

    if (a.emit_level >= 0) {
        // ---- level form: the frontier after level j, for the draft model's next pass ------------------
        // Member p is draft node 1 + j k + p (the root is draft node 0, the frontier of level i occupies
        // 1 + i k .. i k + k): token, the slot of its parent in the previous frontier, position id, the
        // ancestor-or-self mask over draft nodes (only while they fit 128 bits) and its score.
        const int j = a.emit_level;
        if (tid < k) {
            const int c = frontier[j * RESPS_MAX_K + tid];
            const int64_t of = static_cast<int64_t>(b) * a.max_k + tid;
            const Cand r = decode(c);
            a.fr.tokens[of] = a.row_id[(row0 + cand_row(r)) * a.max_k + r.place];
            a.fr.parent_slot[of] = (j == 0) ? -1 : r.list;
            a.fr.position_ids[of] = sd.L + j + 1;
            a.fr.node_index[of] = 1 + j * k + tid;
            if (a.fr.score) a.fr.score[of] = fscore[j * RESPS_MAX_K + tid];
            a.state_frontier[state0 + j * RESPS_MAX_K + tid] = c;
            a.state_score[state0 + j * RESPS_MAX_K + tid] = fscore[j * RESPS_MAX_K + tid];
            unsigned long long lo = 1ull, hi = 0ull;  // the root
            if (1 + (j + 1) * k <= 128) {
                int cc = c, slot = tid;
#pragma unroll 1
                for (int jj = j; jj >= 0; --jj) {
                    const int node = 1 + jj * k + slot;
                    if (node < 64)
                        lo |= 1ull << node;
                    else
                        hi |= 1ull << (node - 64);
                    if (jj > 0) {
                        slot = by_k.div(cc - (k + (jj - 1) * kk));
                        cc = frontier[(jj - 1) * RESPS_MAX_K + slot];
                    }
                }
            } else {
                lo = 0ull;
            }
            a.fr.mask[of * 2 + 0] = lo;
            a.fr.mask[of * 2 + 1] = hi;
        }
        if (tid == 0 && sd.clamped) atomicOr(a.status, RESPS_STATUS_STEP_CLAMPED);
        return;
    }

    // ---- global rerank: keep the m best of all candidates -------------------------------------------
    // A selection, not a sort: a histogram over equal steps of score between the best score (a first-level
    // candidate: scores only fall along a path) and a lower bound of the m-th best finds the step in which
    // the m-th best lies; the steps above are kept whole, and the few candidates inside it are ranked by
    // counting.  The bound is the worst frontier member when the frontiers alone hold m candidates, else
    // the worst candidate.  A step with many candidates is cut again; one whose candidates all tie is cut
    // by index.  (Subtraction, product and truncation are monotone, so a better score is never in a later
    // step.)
    const bool bounded = d * k >= m;
    double top = fscore[0], low = key_score(sh.low), inv = 0.0;
    auto set_range = [&](double t, double l) {  // (the reciprocal need not be exact, only the same for all)
        top = t, low = l;
        inv = static_cast<double>(__fdividef(static_cast<float>(kBins), static_cast<float>(t - l)));
    };
    auto count = [&](int c, double s) {
        int at = kBins;  // outside
        if (s >= low && s <= top) {
            at = max(min(__double2int_rz((top - s) * inv), kBins - 1), 0);  // (0 * inf counts as 0)
            atomicAdd(&sh.hist[at], 1);
        }
        node_of[c] = at;
    };
    if (bounded) set_range(top, low);
    double least = low;
#pragma unroll 1
    for (int c = tid, u = 0; c < n_cand; c += nthreads, ++u) {
        const int parent = (u == 0) ? own_parent : parent_of(c);
        double s = score[c];
        if (parent >= 0) score[c] = s = s + fscore[parent];
        if (bounded)
            count(c, s);
        else
            least = fmin(least, s);
    }
    if (!bounded) {
        __syncthreads();
        if (least < low) atomicMin(&sh.low, score_key(least));
        __syncthreads();
        set_range(top, key_score(sh.low));
    }
    int need = m;
    constexpr int kMaxRounds = 256;  // (a round narrows the range of scores several hundredfold: never reached)
#pragma unroll 1
    for (int round = 0; need > 0 && round < kMaxRounds; ++round) {
        if (round > 0 || !bounded)
#pragma unroll 1
            for (int c = tid; c < n_cand; c += nthreads) count(c, score[c]);
        __syncthreads();
        {  // the step in which the count reaches `need`; a warp's share of the steps is contiguous
            const int mine = sh.hist[tid];
            int incl = mine;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int t = __shfl_up_sync(kFull, incl, o);
                if (lane >= o) incl += t;
            }
            if (lane == 31) sh.warp_sum[warp] = incl;
            __syncthreads();
            const int before_warp = __reduce_add_sync(kFull, lane < warp ? sh.warp_sum[lane] : 0);
            const int before = before_warp + incl - mine;
            if (before < need && before + mine >= need) sh.cut = tid, sh.cut_before = before, sh.cut_count = mine;
            if (tid == 0) sh.n_list = 0, sh.low = score_key(top), sh.high = score_key(low);
            sh.hist[tid] = 0;
        }
        __syncthreads();
        const int cut = sh.cut, in_cut = sh.cut_count;
        need -= sh.cut_before;
        const bool whole = in_cut == need, again = !whole && in_cut > kTieList;
#pragma unroll 1
        for (int c0 = 0; c0 < n_cand; c0 += kTreeThreads) {
            const int c = c0 + tid;
            const int at = (c < n_cand) ? node_of[c] : kBins;
            const bool keep = at < cut || (at == cut && whole);
            const unsigned bal = __ballot_sync(kFull, keep);
            if (bal) {  // one counter update per warp
                int pos = 0;
                if (lane == 0) pos = atomicAdd(&sh.n_kept, __popc(bal));
                pos = __shfl_sync(kFull, pos, 0) + __popc(bal & ((1u << lane) - 1u));
                if (keep) sh.kept[pos] = c;
            }
            if (c < n_cand) node_of[c] = 0;
            if (at == cut && !whole) {
                if (!again) {
                    sh.list[atomicAdd(&sh.n_list, 1)] = c;
                } else {
                    atomicMin(&sh.low, score_key(score[c]));
                    atomicMax(&sh.high, score_key(score[c]));
                }
            }
        }
        __syncthreads();
        if (whole) break;
        if (!again) {
            if (tid < in_cut) {
                const int c = sh.list[tid];
                const double s = score[c];
                int rank = 0;
#pragma unroll 1
                for (int i = 0; i < in_cut; ++i) {
                    const int o = sh.list[i];
                    rank += (score[o] > s || (score[o] == s && o < c)) ? 1 : 0;
                }
                if (rank < need) sh.kept[atomicAdd(&sh.n_kept, 1)] = c;
            }
            __syncthreads();
            break;
        }
        set_range(key_score(sh.high), key_score(sh.low));
        if (low == top) {  // equal scores: the lower indices
#pragma unroll 1
            for (int c0 = 0; need > 0 && c0 < n_cand; c0 += kTreeThreads) {
                const int c = c0 + tid;
                const bool tie = c < n_cand && score[c] == low;
                const unsigned bal = __ballot_sync(kFull, tie);
                __syncthreads();
                if (lane == 0) sh.warp_sum[warp] = __popc(bal);
                __syncthreads();
                const int before = __reduce_add_sync(kFull, lane < warp ? sh.warp_sum[lane] : 0) + __popc(bal & ((1u << lane) - 1u));
                if (tie && before < need) sh.kept[atomicAdd(&sh.n_kept, 1)] = c;
                need -= __reduce_add_sync(kFull, lane < kTreeThreads / 32 ? sh.warp_sum[lane] : 0);
            }
            __syncthreads();
            break;
        }
    }
    if (tid >= RESPS_MAX_TT) return;  // at most 127 candidates are left: four warps and their own barrier
    auto meet = [] { asm volatile("bar.sync 1, 128;" ::: "memory"); };

    // ---- node index = 1 + kept candidates with a lower index ------------------------------------------
    const int64_t ob = static_cast<int64_t>(b) * a.max_tt;
    int node = 0, token = 0, dep = 0;
    Cand own = {0, 0, 0};
    if (tid < m) {
        const int c = sh.kept[tid];
        own = decode(c);
        token = a.row_id[(row0 + cand_row(own)) * a.max_k + own.place];  // on its way during what follows
        dep = own.level + 1;
        const int4* all = reinterpret_cast<const int4*>(sh.kept);
#pragma unroll 1
        for (int i = 0; i < (m + 3) / 4; ++i) {
            const int4 v = all[i];
            node += (v.x < c) + (v.y < c) + (v.z < c) + (v.w < c);
        }
        ++node;
        node_of[c] = node;
    } else if (tid == m) {
        token = a.root_token[b];
    }
    meet();
    int pn = -1;
    if (tid < m) {
        pn = (own.level == 0) ? 0 : node_of[frontier[(own.level - 1) * RESPS_MAX_K + own.list]];
        sh.parent[node] = pn;
        sh.has_child[pn] = 1;
    } else if (tid == m) {
        sh.parent[0] = -1;
        sh.row[0] = 0;
    }
    // The draft row every node's children were taken from (kept in the workspace for the acceptance
    // under sampling, which needs the draft distribution behind every tried child): the root's is row
    // (0, 0); the p-th member of the frontier after level j < d-1 was given row (j+1, p).
#pragma unroll 1
    for (int e = tid; e < (d - 1) * k; e += RESPS_MAX_TT) {
        const int j = by_k.div(e), p = e - j * k;
        const int i = node_of[frontier[j * RESPS_MAX_K + p]];
        if (i > 0) sh.row[i] = (j + 1) * RESPS_MAX_K + p;
    }
    if (tid <= m) sh.depth[node] = dep;
    meet();

    // ---- ancestor masks, leaves, retrieve rows (thread = node) ------------------------------------------
    const bool leaf = tid < n && !sh.has_child[tid];
    const unsigned bal = __ballot_sync(kFull, leaf);
    if (lane == 0) sh.warp_sum[warp] = __popc(bal);
    meet();
    if (tid < n) {
        const int rs = a.max_depth + 1;
        const int last = sh.depth[tid];
        int row = __popc(bal & ((1u << lane) - 1u));
#pragma unroll 1
        for (int w = 0; w < warp; ++w) row += sh.warp_sum[w];
        int32_t* path = a.retrieve + (ob + row) * rs;
        unsigned long long lo = 0ull, hi = 0ull;
        int cur = tid;
#pragma unroll 1
        for (int t = last; t >= 0; --t) {
            const unsigned long long bit = 1ull << (cur & 63);
            if (cur < 64)
                lo |= bit;
            else
                hi |= bit;
            if (leaf) path[t] = cur;
            cur = sh.parent[cur];
        }
        if (leaf)
#pragma unroll 1
            for (int t = last + 1; t < rs; ++t) path[t] = -1;
        a.mask[(ob + tid) * 2 + 0] = lo;
        a.mask[(ob + tid) * 2 + 1] = hi;
        a.node_row[ob + tid] = sh.row[tid];
        // (these by the candidate's thread: the token id has been on its way since the candidate was known)
        a.tokens[ob + node] = token;
        a.parent[ob + node] = pn;
        a.depth[ob + node] = dep;
        a.position_ids[ob + node] = sd.L + dep;
    }
    if (tid == 0) {
        a.n_leaves[b] = sh.warp_sum[0] + sh.warp_sum[1] + sh.warp_sum[2] + sh.warp_sum[3];
        a.n_nodes[b] = n;
        if (sd.clamped || sh.n_kept != m) atomicOr(a.status, RESPS_STATUS_STEP_CLAMPED);
    }
}
}  // namespace

constexpr int kMaxCandidates = 14944;  // k + (d-1) k^2: what shared memory holds (12 bytes each)

static size_t tree_smem_bytes(int cand_cap) {
    return static_cast<size_t>(cand_cap) * (sizeof(double) + sizeof(int)) +
           RESPS_MAX_DEPTH * RESPS_MAX_K * (sizeof(double) + sizeof(int));
}

cudaError_t launch_tree_build(const resps_ctx* ctx, const resps_step* d_steps, int batch,
                              int n_levels, int n_slots, const int32_t* root_token,
                              int32_t* tokens, int32_t* parent, int32_t* depth, int32_t* position_ids,
                              uint64_t* mask, int32_t* retrieve, int32_t* n_leaves, int32_t* n_nodes,
                              cudaStream_t st, bool after_scan) {
    const resps_shape& s = ctx->shape;
    TreeArgs a;
    a.steps = d_steps;
    a.n_levels = n_levels, a.n_slots = n_slots;
    a.vocab = s.vocab, a.max_tt = s.max_tt, a.max_k = s.max_k, a.max_depth = s.max_depth;
    a.max_rows = ctx->ws.max_rows;
    a.row_val = ctx->ws.row_val, a.row_id = ctx->ws.row_id, a.row_lse = ctx->ws.row_lse;
    a.root_token = root_token;
    a.tokens = tokens, a.parent = parent, a.depth = depth, a.position_ids = position_ids;
    a.mask = mask, a.retrieve = retrieve, a.n_leaves = n_leaves, a.n_nodes = n_nodes;
    a.node_row = ctx->ws.node_row;
    a.status = ctx->ws.status;
    a.cand_cap = s.max_k + (s.max_depth - 1) * s.max_k * s.max_k;
    a.emit_level = -1;
    a.state_frontier = ctx->ws.tree_frontier, a.state_score = ctx->ws.tree_score;
    a.use_state = after_scan ? 0 : 1;
    a.setup_before_wait = after_scan ? 1 : 0;
    a.fr = FrontierOut{};
    const size_t smem = tree_smem_bytes(a.cand_cap);
    return launch_pdl(tree_build_kernel, dim3(batch), dim3(kTreeThreads), smem, st, a);
}

cudaError_t launch_tree_level(const resps_ctx* ctx, const resps_step* d_steps, int batch, int n_levels, int n_slots,
                              int level, const FrontierOut& out, cudaStream_t st) {
    const resps_shape& s = ctx->shape;
    TreeArgs a = {};
    a.steps = d_steps;
    a.n_levels = n_levels, a.n_slots = n_slots;
    a.vocab = s.vocab, a.max_tt = s.max_tt, a.max_k = s.max_k, a.max_depth = s.max_depth;
    a.max_rows = ctx->ws.max_rows;
    a.row_val = ctx->ws.row_val, a.row_id = ctx->ws.row_id, a.row_lse = ctx->ws.row_lse;
    a.node_row = ctx->ws.node_row;
    a.status = ctx->ws.status;
    a.cand_cap = s.max_k + (s.max_depth - 1) * s.max_k * s.max_k;
    a.emit_level = level;
    a.state_frontier = ctx->ws.tree_frontier, a.state_score = ctx->ws.tree_score;
    a.use_state = 1;
    a.setup_before_wait = 1;  // the scan of this level's rows runs directly before
    a.fr = out;
    return launch_pdl(tree_build_kernel, dim3(batch), dim3(kLevelThreads), tree_smem_bytes(a.cand_cap), st, a);
}

// Largest k + (d-1)k^2 the shared-memory arrays can hold.
int tree_candidate_limit() { return kMaxCandidates; }

cudaError_t tree_setup(resps_ctx*) {
    return cudaFuncSetAttribute(tree_build_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                static_cast<int>(tree_smem_bytes(kMaxCandidates)));
}

}  // namespace resps
