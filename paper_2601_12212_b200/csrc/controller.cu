// Controller glue (Algorithm 1: action caching over a cache interval of N steps; Eq. 3 / Eq. 5: the
// reward, tokens per second, averaged over the interval; Eq. 4: the state is the concatenation of three
// hidden layers of the target model, read in place; Appendix A: the policy is a [128, 128] network over
// the filtered action grid).  One kernel per decoding step: it books the reward of the step that has
// just finished and, when the interval is over, asks the policy and writes the new (TT, d, k) into the
// device-resident step parameters, where the kernels of the step read them.
//
// A cluster of 16 CTAs serves one sequence, every CTA a sixteenth of each layer's outputs.  The first layer
// is a matrix-vector product over the 3 x 4096 state (6 MB of fp32 weights): a CTA stages the state in shared
// memory once for all of its hidden units, a few warps share a unit, and a thread keeps eight 16-byte loads in
// flight.  The weights of the two small layers are asked into L2 before that and then wait in registers, a row to a
// warp; the layers' outputs travel to the peers' shared memory behind the cluster's barrier, so that nothing goes
// through global memory.  The choice is made by one CTA:
// maximum, exponentials and running sums by all of its threads.
//
// Bound by the first layer's weights through L2 into 16 SMs per sequence (0.4 MB each, about 3 us), around it
// a chain of three exchanges; a step whose cached action is still valid is bound by its launch.  With a CTA
// per hidden unit and the last one to arrive running both small layers and, by one thread, the softmax, a step
// that asks took 40 us at 8 sequences of the 3 x 4096 state and 180 actions (now 18.4, and 28.6 with the weights in
// HBM, as between the questions of a decode loop); one that does not takes 1.8.
#include <cmath>

#include "common.cuh"

namespace resps {
namespace {

constexpr int kCtlThreads = 512;
constexpr int kWarps = kCtlThreads / 32;
constexpr int kClu = 16;            // CTAs per sequence (more than 8: not portable, sm_100 has it)
constexpr int kMaxHidden = 256;
constexpr int kMaxActions = 1024;
constexpr int kStage = 16384;       // features staged at once
constexpr int kPiece = 2048;        // features of a W1 row asked into L2 by one instruction
constexpr int kAhead = 8;           // 16-byte loads of a thread in flight
constexpr unsigned kFull = 0xFFFFFFFFu;
static_assert(kMaxHidden <= kClu * kWarps, "a warp per hidden unit in the second layer");
static_assert(kMaxActions <= 2 * kCtlThreads, "two actions per thread in the choice");

struct ControllerArgs {
    resps_policy pol;
    const __nv_bfloat16* hidden[3];  // three layers' hidden states, [batch][features / 3] each
    int64_t ld_hidden;
    int batch, interval;
    float temperature;
    const double* uniform;       // [batch] or null (temperature 0)
    const int32_t* accept_len;   // [batch] of the finished step, or null
    const float* elapsed_s;      // [batch] seconds of the finished step, or null
    resps_controller_state* state;
    resps_step* steps;
    float* reward_avg;           // [batch]: written when an interval closes (else left alone)
    float* logits_out;           // [batch][n_actions] or null
    int32_t* action_out;         // [batch] or null
};

struct ControllerShared {
    alignas(16) __nv_bfloat16 state[kStage];
    float h1[kMaxHidden], h2[kMaxHidden];  // written by the peers
    float logit[kMaxActions];              // of the first CTA: written by the peers
    float part[kWarps];
    unsigned long long key[kWarps];
    double sum[kWarps];
    int action;
};

__device__ __forceinline__ bool aligned_to(const void* p, unsigned bytes) {
    return (reinterpret_cast<unsigned long long>(p) & (bytes - 1u)) == 0ull;
}
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    return v;
}
// one float to the same place in the shared memory of peer `lane` (of all peers: by 16 lanes)
__device__ __forceinline__ void store_to_peer(float* local, unsigned peer, float v) {
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(peer_address(local, peer)), "f"(v) : "memory");
}
// row . s_x over n inputs by a warp, the row's elements already in registers (n <= kMaxHidden)
struct Row {
    float w[kMaxHidden / 32];
    __device__ __forceinline__ void load(const float* row, int n, int lane, bool valid) {
#pragma unroll
        for (int j = 0; j < kMaxHidden / 32; ++j) w[j] = (valid && lane + 32 * j < n) ? __ldg(row + lane + 32 * j) : 0.f;
    }
    __device__ __forceinline__ float dot(const float* s_x, int n, int lane) const {
        float acc = 0.f;
#pragma unroll
        for (int j = 0; j < kMaxHidden / 32; ++j)
            if (lane + 32 * j < n) acc = fmaf(w[j], s_x[lane + 32 * j], acc);
        return warp_sum(acc);
    }
};

__global__ void __launch_bounds__(kCtlThreads, 2) controller_kernel(const ControllerArgs a) {
    pdl_wait();  // the kernel before this one in the stream has completed
    pdl_launch_dependents();
    __shared__ ControllerShared sh;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned rank = cluster_rank();
    const int b = blockIdx.x / kClu;
    // (The neighbour's cluster may be writing `beside` at the same time.  Whichever words are seen, old or new, decide one
    // thing only: which sequence asks W1 into L2 below.  No result depends on it, so the read is left unordered: as
    // relaxed loads of device scope the two words cost 1.2 to 2 us of the 6 us of a call at 8 sequences.)
    const resps_controller_state st = a.state[b], beside = a.state[max(b - 1, 0)];
    const bool ask = (st.cache_step == 0) || (st.action < 0);
    const bool writer = rank == 0 && tid == 0;
    cluster_arrive();  // waited for before the state, or a peer's shared memory, is written
    resps_controller_state n = st;
    if (writer && a.accept_len) {  // the finished step's reward
        n.reward_sum += static_cast<float>(a.accept_len[b] + 1) / a.elapsed_s[b];
        n.reward_steps += 1;
    }
    if (!ask) {
        // ---- the cached action stays: advance the cache step (once every CTA has read the state) ------------
        cluster_wait();
        if (writer) {
            n.cache_step += 1;
            if (n.cache_step >= a.interval) n.cache_step = 0;
            a.state[b] = n;
            if (a.action_out) a.action_out[b] = n.action;
        }
        return;
    }
    const int H = a.pol.hidden, F = a.pol.n_features, A = a.pol.n_actions;
    const int units = (H + kClu - 1) / kClu, u_lo = static_cast<int>(rank) * units, n_units = max(0, min(H - u_lo, units));
    const int rows = (A + kClu - 1) / kClu, r_lo = static_cast<int>(rank) * rows, n_rows = max(0, min(A - r_lo, rows));
    const float* row2 = a.pol.w2 + static_cast<int64_t>(u_lo + warp) * H;
    const float* row3 = a.pol.w3 + static_cast<int64_t>(r_lo + warp) * H;
    if (lane * 32 < H) {
        if (warp < n_units) asm volatile("prefetch.global.L2 [%0];" ::"l"(row2 + lane * 32));
        if (warp < n_rows) asm volatile("prefetch.global.L2 [%0];" ::"l"(row3 + lane * 32));
    }

    // ---- first layer: `per_unit` warps share a hidden unit ----------------------------------------------
    const int per_unit = kWarps / units, mine = warp / per_unit, share = warp - mine * per_unit;
    float acc = 0.f;
    {
        const int per_layer = F / 3;
        const bool vec_h = (per_layer & 7) == 0 && (a.ld_hidden & 7) == 0 && aligned_to(a.hidden[0], 16) &&
                           aligned_to(a.hidden[1], 16) && aligned_to(a.hidden[2], 16);
        const bool vec_w = (F & 3) == 0 && aligned_to(a.pol.w1, 16);
#pragma unroll 1
        for (int f0 = 0; f0 < F; f0 += kStage) {
            const int nf = min(kStage, F - f0);
            if (f0 > 0) __syncthreads();  // the last part has been read
            const float* w = a.pol.w1 + static_cast<int64_t>(u_lo + mine) * F + f0;
            const float4* w4 = reinterpret_cast<const float4*>(w);
            const int quads = (vec_w && mine < n_units) ? nf >> 2 : 0, step = per_unit * 32;
            float4 x[kAhead];
            int i = share * 32 + lane;
#pragma unroll
            for (int q = 0; q < kAhead; ++q)
                if (i + q * step < quads) x[q] = __ldg(w4 + i + q * step);
            // W1 is likely to have left L2 since it was last read, and a thread's eight loads would take a round trip to
            // HBM each: the rows are asked into L2 at once.  (By one of the sequences next to one another that ask.)
            if (f0 == 0 && vec_w && !(b > 0 && (beside.cache_step == 0 || beside.action < 0))) {
                const int u = tid >> 5, at = lane * kPiece;
                if (u < n_units) {
#pragma unroll 1
                    for (int f = at; f < F; f += 32 * kPiece)
                        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(a.pol.w1 + static_cast<int64_t>(u_lo + u) * F + f),
                                     "r"(min(kPiece, F - f) * 4));
                }
            }
            if (vec_h) {
#pragma unroll 4
                for (int e = tid * 8; e < nf; e += kCtlThreads * 8) {
                    const int f = f0 + e, layer = (f >= per_layer) + (f >= 2 * per_layer);
                    *reinterpret_cast<uint4*>(sh.state + e) =
                        __ldg(reinterpret_cast<const uint4*>(a.hidden[layer] + b * a.ld_hidden + f - layer * per_layer));
                }
            } else {
#pragma unroll 1
                for (int e = tid; e < nf; e += kCtlThreads) {
                    const int f = f0 + e, layer = (f >= per_layer) + (f >= 2 * per_layer);
                    sh.state[e] = a.hidden[layer][b * a.ld_hidden + f - layer * per_layer];
                }
            }
            __syncthreads();
#pragma unroll 1
            for (; i < quads; i += kAhead * step) {
#pragma unroll
                for (int q = 0; q < kAhead; ++q)
                    if (i + q * step < quads) {
                        const uint2 h = *reinterpret_cast<const uint2*>(sh.state + 4 * (i + q * step));
                        acc = fmaf(x[q].x, __uint_as_float(h.x << 16), acc);
                        acc = fmaf(x[q].y, __uint_as_float(h.x & 0xFFFF0000u), acc);
                        acc = fmaf(x[q].z, __uint_as_float(h.y << 16), acc);
                        acc = fmaf(x[q].w, __uint_as_float(h.y & 0xFFFF0000u), acc);
                        if (i + (q + kAhead) * step < quads) x[q] = __ldg(w4 + i + (q + kAhead) * step);
                    }
            }
            if (!vec_w && mine < n_units) {
#pragma unroll 4
                for (int e = share * 32 + lane; e < nf; e += step) acc = fmaf(__ldg(w + e), __bfloat162float(sh.state[e]), acc);
            }
        }
    }
    Row w2, w3;
    w2.load(row2, H, lane, warp < n_units);
    w3.load(row3, H, lane, warp < n_rows);
    acc = warp_sum(acc);
    if (lane == 0) sh.part[warp] = acc;
    __syncthreads();
    cluster_wait();
    if (warp < n_units) {  // unit `warp`: its warps' shares
        float v = a.pol.b1[u_lo + warp];
#pragma unroll 1
        for (int q = 0; q < per_unit; ++q) v += sh.part[warp * per_unit + q];
        v = tanhf(v);
        if (lane < kClu) store_to_peer(&sh.h1[u_lo + warp], lane, v);
    }
    cluster_barrier();
    // ---- second layer: a unit per warp ------------------------------------------------------------------
    if (warp < n_units) {
        const float v = tanhf(w2.dot(sh.h1, H, lane) + a.pol.b2[u_lo + warp]);
        if (lane < kClu) store_to_peer(&sh.h2[u_lo + warp], lane, v);
    }
    cluster_barrier();
    // ---- action logits, to the first CTA ------------------------------------------------------------------
#pragma unroll 1
    for (int r = warp; r < n_rows; r += kWarps) {
        if (r != warp) w3.load(a.pol.w3 + static_cast<int64_t>(r_lo + r) * H, H, lane, true);
        const float v = w3.dot(sh.h2, H, lane) + a.pol.b3[r_lo + r];
        if (lane == 0) {
            store_to_peer(&sh.logit[r_lo + r], 0u, v);
            if (a.logits_out) a.logits_out[static_cast<int64_t>(b) * A + r_lo + r] = v;
        }
    }
    cluster_barrier();
    if (rank != 0) return;

    // ---- the choice.  Actions [per * tid, per * tid + per) belong to a thread -----------------------------
    const int per = A > kCtlThreads ? 2 : 1;
    // largest logit, ties -> lowest index: (ordered value, ~index) keys
    unsigned long long best = 0ull;
#pragma unroll 1
    for (int o = per * tid; o < min(A, per * tid + per); ++o) {
        const unsigned long long key = pack_val_id(sh.logit[o], o);
        best = key > best ? key : best;
    }
#pragma unroll 1
    for (int off = 16; off > 0; off >>= 1) {
        const unsigned long long other = __shfl_xor_sync(kFull, best, off);
        best = other > best ? other : best;
    }
    if (lane == 0) sh.key[warp] = best;
    if (tid == 0) sh.action = A - 1;
    __syncthreads();
    best = sh.key[lane & (kWarps - 1)];
#pragma unroll 1
    for (int off = kWarps / 2; off > 0; off >>= 1) {
        const unsigned long long other = __shfl_xor_sync(kFull, best, off);
        best = other > best ? other : best;
    }
    int action = key_id(best);
    if (a.temperature > 0.f) {
        // softmax(logits / T) in fp64 (a quotient grows with its numerator: the maximum is the best logit's), the
        // inverse of its running sum in action order
        const double T = static_cast<double>(a.temperature), mx = static_cast<double>(key_val(best)) / T;
        double e[2] = {0.0, 0.0}, run;
#pragma unroll 1
        for (int i = 0; i < per; ++i)
            if (per * tid + i < A) {
                const double v = exp(static_cast<double>(sh.logit[per * tid + i]) / T - mx);
                if (i == 0) e[0] = v; else e[1] = v;
            }
        double incl = e[0] + e[1];
#pragma unroll 1
        for (int off = 1; off < 32; off <<= 1) {
            const double before = __shfl_up_sync(kFull, incl, off);
            if (lane >= off) incl += before;
        }
        if (lane == 31) sh.sum[warp] = incl;
        __syncthreads();
        double upto = sh.sum[lane & (kWarps - 1)];
#pragma unroll 1
        for (int off = 1; off < kWarps; off <<= 1) {
            const double before = __shfl_up_sync(kFull, upto, off, kWarps);
            if ((lane & (kWarps - 1)) >= off) upto += before;
        }
        const double target = a.uniform[b] * __shfl_sync(kFull, upto, kWarps - 1);
        const double before = __shfl_sync(kFull, upto, (warp + kWarps - 1) & (kWarps - 1));
        run = (warp > 0 ? before : 0.0) + incl - e[1];  // up to and with the thread's first action
        if (per * tid < A && run > target) atomicMin(&sh.action, per * tid);
        else if (per == 2 && per * tid + 1 < A && run + e[1] > target) atomicMin(&sh.action, per * tid + 1);
        __syncthreads();
        action = sh.action;
    }
    if (writer) {
        if (n.reward_steps > 0) a.reward_avg[b] = n.reward_sum / static_cast<float>(n.reward_steps);  // Eq. 5
        n.reward_sum = 0.f, n.reward_steps = 0;
        n.action = action;
        n.cache_step = 1;
        if (n.cache_step >= a.interval) n.cache_step = 0;
        a.state[b] = n;
        resps_step s = a.steps[b];
        s.tt = a.pol.actions[3 * action + 0], s.d = a.pol.actions[3 * action + 1], s.k = a.pol.actions[3 * action + 2];
        a.steps[b] = s;
        if (a.action_out) a.action_out[b] = action;
    }
}

}  // namespace

int controller_max_hidden() { return kMaxHidden; }
int controller_max_actions() { return kMaxActions; }

cudaError_t controller_setup(resps_ctx*) {
    return cudaFuncSetAttribute(controller_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
}

cudaError_t launch_controller(const resps_ctx*, const resps_policy* pol, const void* h, const void* m, const void* l,
                              int64_t ld_hidden, int batch, int interval, float temperature, const double* uniform,
                              const int32_t* accept_len, const float* elapsed_s, resps_controller_state* state,
                              resps_step* steps, float* reward_avg, float* logits_out, int32_t* action_out,
                              cudaStream_t st) {
    ControllerArgs a;
    a.pol = *pol;
    a.hidden[0] = static_cast<const __nv_bfloat16*>(h);
    a.hidden[1] = static_cast<const __nv_bfloat16*>(m);
    a.hidden[2] = static_cast<const __nv_bfloat16*>(l);
    a.ld_hidden = ld_hidden, a.batch = batch, a.interval = interval, a.temperature = temperature;
    a.uniform = uniform, a.accept_len = accept_len, a.elapsed_s = elapsed_s;
    a.state = state, a.steps = steps, a.reward_avg = reward_avg, a.logits_out = logits_out, a.action_out = action_out;
    return launch_pdl_cluster(controller_kernel, kClu, dim3(batch * kClu), dim3(kCtlThreads), 0, st, a);
}

}  // namespace resps
