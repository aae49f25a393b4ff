// Verification and acceptance under sampling, temperature T > 0 (Section 3.2, "Acceptance
// Criterion": a draft token y is accepted with probability min(1, P_T(y) / P_d(y)); Section 4.1,
// "Lossless Output Fidelity": rejection-based correction keeps the target's distribution).
//
// For a chain of draft tokens this is the paper's rule with the correction step of the
// speculative-sampling papers it cites (on the first rejection the token is drawn from the
// normalised residual max(0, P_T - P_d); after a chain accepted in full, from P_T).  In a tree the
// children of the current node are tried in node order; after a rejected child x the target side
// becomes the normalised residual max(0, p - q), the draft side q without x, renormalised, and the
// next sibling is tried against those; when no child is left the token is drawn from the residual.
//
// All of it is a walk of at most max_depth + 1 nodes, but each step of the walk needs sums over the
// whole vocabulary (normalisers of softmax and of residuals, the cumulative sum the token is drawn
// from).  A thread-block cluster of 16 CTAs serves one sequence: every CTA takes a sixteenth of the
// vocabulary, every CTA writes its partial sums into every peer's shared memory behind the hardware
// cluster barrier (no spinning anywhere), and every thread then takes the same decision from the same
// numbers.  Arithmetic is fp64 throughout: a decision (accept or not, which token) is a comparison of
// sums over 10^5 terms, and only at fp64 is the order of summation immaterial to it.
//
// The exponentials are taken once per visited node.  The target-side value P and the raw draft-side
// exponential Q of every token of the CTA's slice live in shared memory (what does not fit, in an
// L2-resident scratch); token e belongs to thread e % 512, so rows are read once and coalesced and only the
// owner touches a token's values.  The draft side is Q times one scalar (softmax sum and renormalisations
// are the same factor for every token; a removed token's entry is set to zero).
//
// Bound by a chain of small steps: per node two row slices from HBM, 2 x 16 fp64 exponentials a thread and
// one exchange over the cluster (1.3 us), per rejection one pass over shared memory and one exchange.
// What is kept short: the children are found by ballots, their (P, Q) are pushed into every CTA's shared
// memory behind the exchange's barrier, every thread takes the decision for itself, the rows of the child
// that is tried first are asked into L2 while its parent is worked on, and the loops are short (the kernel
// runs once per step: unrolled over the tokens it was 70 KB of code).  The exponentials are relative to the CTA's
// own maximum, so that maxima and sums cross the cluster together.  With clusters of 8 CTAs of 1024 threads,
// the draft side in L2, one thread looking up children and deciding, the calls of TT=60 d=7 k=10 V=128256 took
// 100 us.
#include <cmath>

#include "common.cuh"
#include "exp_le0.cuh"

namespace resps {
namespace {

// CTAs per sequence (more than 8: not portable, sm_100 has it).  Seven clusters of 16 are resident, so a batch of 8
// takes two turns; the clusters of 8 CTAs before were 15.  In us a call, single calls behind an L2 flush, before / now, at
// V = 128256, TT=60 d=7 k=10: 1 sequence 139 / 56, 7 175 / 69, 8 184 / 78, 12 179 / 106, 15 201 / 130, 16 214 / 133,
// 24 266 / 180, 32 352 / 227; at V = 32000: 1 86 / 40, 8 99 / 60, 15 113 / 83, 32 195 / 156.  No batch is slower.
constexpr int kClu = 16;
constexpr int kSampThreads = 512;
constexpr int kWarps = kSampThreads / 32;
constexpr unsigned kFull = 0xFFFFFFFFu;

struct SampledArgs {
    const resps_step* steps;
    const int32_t* n_nodes;
    const float* target;
    int64_t ld_b, ld_row;
    const float* draft;
    int64_t dld_b, dld_level, dld_row;
    const int32_t* node_row;  // [batch][max_tt]: level * RESPS_MAX_K + slot of the row a node's children came from
    double inv_t;             // 1 / temperature
    const int32_t *tokens, *parent;
    const double *u_accept, *u_sample;
    int vocab, max_tt, max_depth, max_k;
    int32_t *accept_path, *accept_len, *out_tokens;
    resps_step* steps_next;
    double* scratch;        // [batch][kClu][2][state] (P, Q) of tokens that do not fit shared memory
    int64_t state;          // doubles of one CTA's P (or Q) array, padding included
    int p_in_smem, q_in_smem;
};

struct Pair {
    double x, y;
};

// What the stored target-side value of a token still lacks: the division by the softmax sum, or one
// rejection round (Section 3.2, "Acceptance Criterion": target side -> normalised max(0, p - q)).  The
// draft side is kept as the raw exponentials times one scalar for the whole row (the softmax sum and
// the renormalisations after every removal are the same factor for every token), with the entry of
// a removed token set to zero.
struct Pending {
    int kind;      // 1 the softmax sum, 2 a rejection round
    double a;      // reciprocal of the target's sum (kind 1) / of the residual's normaliser (kind 2; 0: residual empty, p is kept)
    double sq_old; // kind 2: the draft side's scalar as it was when the round's child was tried
};
// A division by a normaliser is a multiplication by its fp64 reciprocal (one rounding more than the
// quotient; the decisions compare sums of 10^5 such terms and are taken with a margin far above that).
__device__ __forceinline__ double recip_or_zero(double s) { return s > 0.0 ? 1.0 / s : 0.0; }
// `factor` puts a softmax weight on the row's scale (kind 1); q_raw is on it already.
__device__ __forceinline__ double apply(const Pending& pd, double p, double factor, double q_raw) {
    if (pd.kind == 1) return p * (factor * pd.a);
    return pd.a > 0.0 ? fmax(p - q_raw * pd.sq_old, 0.0) * pd.a : p;
}

// What the peers write into this CTA's shared memory in one exchange over the cluster.  There are two sets, used
// in turn by ALL exchanges of the walk, whatever they carry (the start of a node, a rejection, the draw).  Set s of
// exchange i is written before the cluster barrier of exchange i and read between that barrier and this CTA's arrival
// at the barrier of exchange i + 1; exchange i + 2, the next to write it, begins behind that second barrier.  So one
// barrier per exchange orders every write of a peer behind every read of what it replaces.
struct Exchange {
    double sum[kClu][2];             // partial sums
    double top[kClu][2];             // the maxima they are relative to, times 1 / T (start of a node)
    double tab[RESPS_MAX_K][2];      // (P, Q) of the children's tokens, written by their owners
};
struct SampledShared {
    double exp2_64[kExpTable];       // 2^(i/64)
    double red[kWarps][2];
    Exchange ex[2];                  // written by the peers
    double factor[kClu][2];          // e^(a CTA's maximum - the row's)
    double scan[kWarps];
    double u[RESPS_MAX_K];
    unsigned red_max[kWarps][2];
    int tok[RESPS_MAX_TT], par[RESPS_MAX_TT], row[RESPS_MAX_TT], children[RESPS_MAX_TT];
    int child_at[RESPS_MAX_K];       // a child's token in this CTA's slice, -1: not here
    int child_clu[RESPS_MAX_K];      // the CTA that has it
    int count[4];
    int pick;
};

__device__ __forceinline__ void store_pair_to_peer(double* local, unsigned peer, double x, double y) {
    asm volatile("st.shared::cluster.v2.f64 [%0], {%1, %2};" ::"r"(peer_address(local, peer)), "d"(x), "d"(y) : "memory");
}
// The part of [from, from + count) floats that the bulk prefetch can take (16-byte granular).
__device__ __forceinline__ void prefetch_l2(const float* from, int count) {
    const uintptr_t lo = (reinterpret_cast<uintptr_t>(from) + 15) & ~static_cast<uintptr_t>(15);
    const uintptr_t hi = reinterpret_cast<uintptr_t>(from + count) & ~static_cast<uintptr_t>(15);
    if (hi > lo)
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(lo), "r"(static_cast<uint32_t>(hi - lo)) : "memory");
}

__global__ void __launch_bounds__(kSampThreads, 1) accept_sampled_kernel(const SampledArgs a) {
    pdl_wait();  // the kernel before this one in the stream has completed
    pdl_launch_dependents();
    __shared__ SampledShared sh;
    extern __shared__ __align__(16) unsigned char s_dyn[];
    cluster_arrive();  // waited for before the first store to a peer
    const unsigned rank = cluster_rank();
    const int b = blockIdx.x / kClu, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n = min(max(a.n_nodes[b], 1), a.max_tt);
    const int64_t ob = static_cast<int64_t>(b) * a.max_tt;
    const int cap = a.max_depth + 1;
    if (tid < RESPS_MAX_TT) {
        sh.tok[tid] = (tid < n) ? a.tokens[ob + tid] : -1;
        sh.par[tid] = (tid < n) ? a.parent[ob + tid] : -2;
        sh.row[tid] = (tid < n) ? a.node_row[ob + tid] : -1;
    }
    if (rank == 0 && tid < cap) {
        a.accept_path[b * cap + tid] = (tid == 0) ? 0 : -1;
        a.out_tokens[b * cap + tid] = -1;
    }
    if (tid == 0) sh.pick = -1;
    if (tid < kExpTable) sh.exp2_64[tid] = exp2(static_cast<double>(tid) / kExpTable);
    __syncthreads();
    cluster_wait();
    // this CTA's share of the vocabulary; token e of it belongs to thread e % 512, place e / 512
    const int V = a.vocab, per_cta = (V + kClu - 1) / kClu;
    const int c_lo = min(V, static_cast<int>(rank) * per_cta), n_cta = min(V, c_lo + per_cta) - c_lo;
    const int per = (n_cta + kSampThreads - 1) / kSampThreads;  // places
    // (a padded place per 16: the runs of the draw would otherwise meet on the same banks)
    auto at = [](int e) { return e + (e >> 4); };
    double* const own = a.scratch + (static_cast<int64_t>(b) * kClu + rank) * 2 * a.state;
    double* const P = a.p_in_smem ? reinterpret_cast<double*>(s_dyn) : own;
    double* const Q = a.q_in_smem ? reinterpret_cast<double*>(s_dyn) + a.state : own + a.state;
    int set = 0;  // the set of the next exchange
    int cur = 0, acc = 0, n_child = 0;
    // Two sums over the cluster, the same bits in every thread of every CTA.  Meanwhile (P, Q) of the children's
    // tokens from `from` on, as the pass before left them, go into the table of every CTA (after the call: that of
    // set ^ 1).  At the start of a node the maxima travel along, and the sums are put on the row's common scale.
    auto cluster_sum = [&](double x, double y, int from, bool at_start, double max_t, double max_d) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(kFull, x, o), y += __shfl_xor_sync(kFull, y, o);
        if (lane == 0) sh.red[warp][0] = x, sh.red[warp][1] = y;
        __syncthreads();
        if (warp == 0) {
            x = (lane < kWarps) ? sh.red[lane][0] : 0.0, y = (lane < kWarps) ? sh.red[lane][1] : 0.0;
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) x += __shfl_xor_sync(kFull, x, o), y += __shfl_xor_sync(kFull, y, o);
            if (lane < kClu) {
                store_pair_to_peer(sh.ex[set].sum[rank], lane, x, y);
                if (at_start) store_pair_to_peer(sh.ex[set].top[rank], lane, max_t, max_d);
            }
        } else if (warp == 1 && lane >= from && lane < n_child) {
            const int e = sh.child_at[lane];
            if (e >= 0) {
                const double p = P[at(e)], q = Q[at(e)];
#pragma unroll 1
                for (int c = 0; c < kClu; ++c) store_pair_to_peer(sh.ex[set].tab[lane], c, p, q);
            }
        }
        __syncwarp();
        cluster_barrier();  // (the other set may be written from here on: its readers have arrived)
        const Exchange& ex = sh.ex[set];
        Pair r = {0.0, 0.0};
        if (at_start) {
            if (tid < 2 * kClu) {
                const int side = tid & 1;
                double top = -INFINITY;
#pragma unroll 4
                for (int c = 0; c < kClu; ++c) top = fmax(top, ex.top[c][side]);
                // (a CTA without tokens, or no draft row: nothing to scale)
                const double m = ex.top[tid >> 1][side];
                sh.factor[tid >> 1][side] = m > -INFINITY ? exp_le0(m - top, sh.exp2_64) : 0.0;
            }
            __syncthreads();
#pragma unroll 4
            for (int c = 0; c < kClu; ++c) r.x += ex.sum[c][0] * sh.factor[c][0], r.y += ex.sum[c][1] * sh.factor[c][1];
        } else {
#pragma unroll 4
            for (int c = 0; c < kClu; ++c) r.x += ex.sum[c][0], r.y += ex.sum[c][1];
        }
        set ^= 1;
        return r;
    };
    auto drow_of = [&](int node) {
        const int row = sh.row[node];
        return a.draft + b * a.dld_b + (row / RESPS_MAX_K) * a.dld_level + (row % RESPS_MAX_K) * a.dld_row;
    };

    for (;;) {
        // ---- the rows of the current node: loads in flight while its children are looked up --------------
        const float* trow = a.target + b * a.ld_b + cur * a.ld_row + c_lo;
        const bool maybe_d = sh.row[cur] >= 0;  // a node with children was expanded
        const float* drow = drow_of(maybe_d ? cur : 0) + c_lo;
        float ft = -INFINITY, fd = -INFINITY;
        constexpr int kGroup = 16;  // of each row, in flight together
#pragma unroll 1
        for (int e0 = tid; e0 < n_cta; e0 += kGroup * kSampThreads) {
            float xt[kGroup], xd[kGroup];
#pragma unroll
            for (int u = 0; u < kGroup; ++u) {
                const int e = e0 + u * kSampThreads;
                xt[u] = (e < n_cta) ? __ldg(trow + e) : -INFINITY;
                xd[u] = (e < n_cta && maybe_d) ? __ldg(drow + e) : -INFINITY;
            }
#pragma unroll
            for (int u = 0; u < kGroup; ++u) {
                const int e = e0 + u * kSampThreads;
                ft = fmaxf(ft, xt[u]), fd = fmaxf(fd, xd[u]);
                if (e < n_cta) P[at(e)] = static_cast<double>(xt[u]), Q[at(e)] = static_cast<double>(xd[u]);
            }
        }
        // ---- the children of the current node, in node order ----------------------------------------------
        // (the path array holds max_depth + 1 nodes; a tree is never deeper)
        const bool is_child = tid > 0 && tid < n && sh.par[tid & (RESPS_MAX_TT - 1)] == cur && acc < a.max_depth;
        const unsigned bal = __ballot_sync(kFull, is_child);
        if (warp < 4 && lane == 0) sh.count[warp] = __popc(bal);
        __syncthreads();  // (everyone is done with the previous node's children)
        n_child = 0;
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            if (is_child && w == warp) sh.children[n_child + __popc(bal & ((1u << lane) - 1u))] = tid;
            n_child += sh.count[w];
        }
        if (tid < n_child && tid < a.max_k && tid < RESPS_MAX_K)
            sh.u[tid] = a.u_accept[(static_cast<int64_t>(b) * cap + acc) * a.max_k + tid];
        const bool with_q = n_child > 0;
        // ---- P_T(. | cur) = softmax(row / T) and the draft's P_d: the CTA's maxima, exponentials, sums ----------
        const unsigned mt = __reduce_max_sync(kFull, float_to_ordered(ft)), md = __reduce_max_sync(kFull, float_to_ordered(fd));
        if (lane == 0) sh.red_max[warp][0] = mt, sh.red_max[warp][1] = md;
        __syncthreads();  // (also: the children)
        unsigned top_t = 0u, top_d = 0u;
#pragma unroll 4
        for (int w = 0; w < kWarps; ++w) top_t = max(top_t, sh.red_max[w][0]), top_d = max(top_d, sh.red_max[w][1]);
        const double mx_t = static_cast<double>(ordered_to_float(top_t)) * a.inv_t;
        const double mx_d = static_cast<double>(ordered_to_float(top_d)) * a.inv_t;
        if (tid < n_child && tid < RESPS_MAX_K) {
            const int x = sh.tok[sh.children[tid]], owner = static_cast<int>(static_cast<unsigned>(x) / static_cast<unsigned>(per_cta));
            sh.child_clu[tid] = min(owner, kClu - 1), sh.child_at[tid] = (owner == static_cast<int>(rank)) ? x - c_lo : -1;
        }
        // the rows of the child that is tried first
        if (tid == kSampThreads - 1 && with_q) {
            const int child = sh.children[0];
            prefetch_l2(a.target + b * a.ld_b + child * a.ld_row + c_lo, n_cta);
            if (sh.row[child] >= 0) prefetch_l2(drow_of(child) + c_lo, n_cta);
        }
        double sum_t = 0.0, sum_d = 0.0;
#pragma unroll 4
        for (int e = tid; e < n_cta; e += kSampThreads) {
            const double w = exp_le0(fma(P[at(e)], a.inv_t, -mx_t), sh.exp2_64);
            P[at(e)] = w;
            sum_t += w;
        }
        if (with_q) {
#pragma unroll 4
            for (int e = tid; e < n_cta; e += kSampThreads) {
                const double w = exp_le0(fma(Q[at(e)], a.inv_t, -mx_d), sh.exp2_64);
                Q[at(e)] = w;
                sum_d += w;
            }
        }
        const Pair sum = cluster_sum(sum_t, sum_d, 0, true, n_cta > 0 ? mx_t : -INFINITY, n_cta > 0 && with_q ? mx_d : -INFINITY);
        // What P (and the table's entries) still lack; a pass brings P up to date.
        Pending pend = {1, recip_or_zero(sum.x), 0.0};
        double sq = with_q ? recip_or_zero(sum.y) : 0.0;  // draft side: q = Q * factor * sq
        const double own_t = sh.factor[rank][0], own_d = sh.factor[rank][1];
        // ---- try the children -----------------------------------------------------------------------------
        int next = -1;
#pragma unroll 1
        for (int j = 0; j < n_child && j < a.max_k; ++j) {
            const int child = sh.children[j];
            {
                const double* const entry = sh.ex[set ^ 1].tab[j];  // of the exchange just behind
                const double q_raw = entry[1] * sh.factor[sh.child_clu[j]][1];
                const double p = apply(pend, entry[0], sh.factor[sh.child_clu[j]][0], q_raw);
                const double q = q_raw * sq;
                // u < min(1, p / q), without the quotient
                if (q > 0.0 ? sh.u[j] * q < p : p > 0.0) next = child;
            }
            if (next >= 0) break;
            // rejected: the residual's normaliser and the draft mass that is left without x
            const int x_at = sh.child_at[j];
            double zx = 0.0, zy = 0.0;
            const double scale = own_d * sq;
            if (pend.kind == 1) {
                const double mul = own_t * pend.a;
#pragma unroll 4
                for (int e = tid; e < n_cta; e += kSampThreads) {
                    const double p = P[at(e)] * mul, q = Q[at(e)] * scale;
                    P[at(e)] = p;
                    zx += fmax(p - q, 0.0);
                    zy += (e != x_at) ? q : 0.0;
                }
            } else {
                const double scale_old = own_d * pend.sq_old;
                const bool keep = !(pend.a > 0.0);  // the residual was empty: p stays
#pragma unroll 4
                for (int e = tid; e < n_cta; e += kSampThreads) {
                    const double q_raw = Q[at(e)], q = q_raw * scale, old = P[at(e)];
                    const double p = keep ? old : fmax(old - q_raw * scale_old, 0.0) * pend.a;
                    P[at(e)] = p;
                    zx += fmax(p - q, 0.0);
                    zy += (e != x_at) ? q : 0.0;
                }
            }
            const Pair zr = cluster_sum(zx, zy, j + 1, false, 0.0, 0.0);
            pend = Pending{2, recip_or_zero(zr.x), sq};
            if (x_at >= 0 && x_at % kSampThreads == tid) {  // x leaves the draft side; its own round is applied here
                if (pend.a > 0.0) P[at(x_at)] -= Q[at(x_at)] * scale;
                Q[at(x_at)] = 0.0;
            }
            if (zr.y > 0.0) sq = sq * (1.0 / zr.y);
        }
        if (next >= 0) {
            cur = next;
            ++acc;
            if (rank == 0 && tid == 0) {
                a.accept_path[b * cap + acc] = cur;
                a.out_tokens[b * cap + acc - 1] = sh.tok[cur];
            }
            continue;
        }
        // ---- nobody accepted (or a leaf): draw from the current target-side distribution by inverse CDF in
        // token order: the tokens change hands so that a thread holds a contiguous run --------------------------
#pragma unroll 4
        for (int e = tid; e < n_cta; e += kSampThreads)
            P[at(e)] = apply(pend, P[at(e)], own_t, with_q ? Q[at(e)] * own_d : 0.0);
        __syncthreads();
        const int t_lo = min(n_cta, tid * per), t_hi = min(n_cta, t_lo + per);
        double run = 0.0;
#pragma unroll 4
        for (int e = t_lo; e < t_hi; ++e) run += P[at(e)];
        double inc = run;  // exclusive prefix of the runs over the CTA's threads
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const double w = __shfl_up_sync(kFull, inc, o);
            if (lane >= o) inc += w;
        }
        if (lane == 31) sh.scan[warp] = inc;
        __syncthreads();
        double before = 0.0, cta_total = 0.0;
#pragma unroll 4
        for (int w = 0; w < kWarps; ++w) {
            if (w < warp) before += sh.scan[w];
            cta_total += sh.scan[w];
        }
        const double excl = before + inc - run;
        if (tid < kClu) store_pair_to_peer(sh.ex[set].sum[rank], tid, cta_total, 0.0);
        cluster_barrier();
        double offset = 0.0, total = 0.0;
#pragma unroll 4
        for (int c = 0; c < kClu; ++c) {
            const double t = sh.ex[set].sum[c][0];
            if (c < static_cast<int>(rank)) offset += t;
            total += t;
        }
        const double target = a.u_sample[static_cast<int64_t>(b) * cap + acc] * total;
        // the owner of the target: the last non-empty run that starts at or before it
        const double start = offset + excl;
        const bool last_run = t_lo < t_hi && c_lo + t_hi == V;
        if (t_lo < t_hi && start <= target && (start + run > target || last_run)) {
            double cum = start;
            int pick = t_hi - 1;
#pragma unroll 1
            for (int e = t_lo; e < t_hi; ++e) {
                cum += P[at(e)];
                if (cum > target) {
                    pick = e;
                    break;
                }
            }
            asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(peer_address(&sh.pick, 0u)), "r"(c_lo + pick) : "memory");
        }
        cluster_barrier();
        if (rank == 0 && tid == 0) {
            int tok = sh.pick;
            if (tok < 0) tok = V - 1;  // rounding left the target past every run: the last token
            a.out_tokens[b * cap + acc] = tok;
            a.accept_len[b] = acc;
            if (a.steps_next) {
                resps_step s = a.steps[b];
                s.prefix_len += acc + 1;
                a.steps_next[b] = s;
            }
        }
        break;
    }
    // (the barrier before is the last access to a peer's shared memory)
}

}  // namespace

constexpr size_t kDynSmemCap = 216 * 1024;

static int64_t sampled_state(int vocab) {  // padded doubles of one CTA's slice
    const int per_cta = (vocab + kClu - 1) / kClu;
    return per_cta + per_cta / 16 + 2;
}

size_t sampled_scratch_doubles(int max_batch, int vocab) {
    return static_cast<size_t>(max_batch) * kClu * 2 * sampled_state(vocab);
}

cudaError_t sampled_setup(resps_ctx*) {
    cudaError_t e = cudaFuncSetAttribute(accept_sampled_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(accept_sampled_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kDynSmemCap));
}

cudaError_t launch_accept_sampled(const resps_ctx* ctx, const resps_step* d_steps, const int32_t* d_n_nodes, int batch,
                                  const float* target, int64_t ld_b, int64_t ld_row, const float* draft, int64_t dld_b,
                                  int64_t dld_level, int64_t dld_row, double temperature, const int32_t* tokens,
                                  const int32_t* parent, const double* u_accept, const double* u_sample,
                                  int32_t* accept_path, int32_t* accept_len, int32_t* out_tokens, resps_step* steps_next,
                                  cudaStream_t st) {
    SampledArgs a;
    a.steps = d_steps, a.n_nodes = d_n_nodes;
    a.target = target, a.ld_b = ld_b, a.ld_row = ld_row;
    a.draft = draft, a.dld_b = dld_b, a.dld_level = dld_level, a.dld_row = dld_row;
    a.node_row = ctx->ws.node_row;
    a.inv_t = 1.0 / temperature;
    a.tokens = tokens, a.parent = parent, a.u_accept = u_accept, a.u_sample = u_sample;
    a.vocab = ctx->shape.vocab, a.max_tt = ctx->shape.max_tt, a.max_depth = ctx->shape.max_depth;
    a.max_k = ctx->shape.max_k;
    a.accept_path = accept_path, a.accept_len = accept_len, a.out_tokens = out_tokens, a.steps_next = steps_next;
    a.scratch = ctx->ws.samp_scratch;
    a.state = sampled_state(ctx->shape.vocab);
    const size_t side = sizeof(double) * static_cast<size_t>(a.state);  // both sides fit up to a vocabulary of 208 000
    a.p_in_smem = side <= kDynSmemCap ? 1 : 0;
    a.q_in_smem = 2 * side <= kDynSmemCap ? 1 : 0;
    const size_t dyn_bytes = a.q_in_smem ? 2 * side : a.p_in_smem ? side : 0;
    return launch_pdl_cluster(accept_sampled_kernel, kClu, dim3(batch * kClu), dim3(kSampThreads), dyn_bytes, st, a);
}

}  // namespace resps
