// Adaptive block length (Section 3.1 "Adaptive Block Length"; Section 4: tau = 0.8): after every draft a small router
// decides, per sequence, whether the small model goes on drafting or the drafts made so far are verified.
//
// Features of one draft, from the small model's distribution q = softmax(logits) for it: the entropy of q (nats), the
// k largest probabilities in descending order (lowest id first on ties), and the small model's embedding rows of those
// k tokens.  Router: hidden = relu(W1 x + b1), s = sigmoid(w2 . hidden + b2) = predicted probability that the large
// model disagrees; drafting continues while 1 - s >= tau and fewer than gamma_max drafts exist.
//
// A sequence's row of logits and the hidden units are dealt to the CTAs of one cluster (a lone CTA took 43 us for 32000
// logits and 64 x 2053 weights: one multiprocessor's reads, and every pass over the row follows the one before): each CTA finds the maximum, the exponential sums and the k best of its slice and sends them to the others;
// all of them merge the eight records, gather the feature vector and compute every eighth hidden unit; CTA 0 adds the
// eight shares of w2 . hidden and decides.  A warp's first weights are fetched before the wait on the preceding kernel.
// All sums run in a fixed order, fp32.  What is left (16 us for a launch alone, 8.7 of them in the kernel) is two cluster barriers
// and the code's way into the instruction cache: each step runs once (27 us with unrolled per-thread lists of the k best).
// Dynamic shared memory: (1 + k + k * d) floats for the feature vector.
#pragma once
#include <math.h>
#include <limits.h>
#include "common.cuh"
#include "misc_kernels.cuh"
#include "tc_common.cuh"

namespace tandem {

constexpr int RT_THREADS = 256;
constexpr int RT_WARPS = RT_THREADS / 32;
constexpr int RT_CLUSTER = 8;
constexpr int RT_REGS = 16;
static_assert(RT_WARPS == 8 && RT_CLUSTER == 8, "one lane per warp's, and per CTA's, record");
constexpr int RT_MAX_K = 8;

struct RouterArgs {
    const float* w1;    // [hidden][1 + k + k * d]
    const float* b1;    // [hidden]
    const float* w2;    // [hidden]
    float b2, tau;
    int k, hidden;
};

// What is known of a part of the row: maximum, sum of e = exp(l - max), sum of e (l - max), the k best entries.
struct RouterPart { float m, z, s1, val[RT_MAX_K]; int idx[RT_MAX_K]; };
constexpr int RT_PART_WORDS = sizeof(RouterPart) / 4;

// The best entry (value descending, lower id first on ties) over the warp's lanes; every lane gets it.
__device__ __forceinline__ void rt_warp_best(float& v, int& i) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float ov = __shfl_xor_sync(0xffffffffu, v, o);
        const int oi = __shfl_xor_sync(0xffffffffu, i, o);
        if (ov > v || (ov == v && oi < i)) { v = ov; i = oi; }
    }
}
// One part out of eight: lane c < 8 holds part c's sums and walks its list.  Warp-wide.  (Not inlined: a launch runs its code once,
// and what it costs is fetching the instructions.)
__device__ __noinline__ void rt_merge(const RouterPart* parts, int k, RouterPart& out, int lane) {
    const RouterPart& mine = parts[lane & 7];
    const float m = warp_max(mine.m);
    float z = 0.f, s1 = 0.f;
    if (lane < 8 && mine.m > -INFINITY) {   // sums moved to the common maximum
        const float dm = mine.m - m, f = expf(dm);
        z = mine.z * f;
        s1 = f * fmaf(dm, mine.z, mine.s1);
    }
    z = warp_sum(z);
    s1 = warp_sum(s1);
    if (lane == 0) { out.m = m; out.z = z; out.s1 = s1; }
    int at = 0;
    for (int j = 0; j < k; ++j) {
        float bv = lane < 8 && at < k ? mine.val[at] : -INFINITY;
        int bi = lane < 8 && at < k ? mine.idx[at] : INT_MAX;
        const int own = bi;
        rt_warp_best(bv, bi);
        if (own == bi && bi != INT_MAX) ++at;
        if (lane == 0) { out.val[j] = bv; out.idx[j] = bi; }
    }
}

// Start of an adaptive iteration: every live sequence drafts, nobody has a draft yet.  grid: 1; block: 256.
__global__ void __launch_bounds__(256) adaptive_begin_kernel(LoopState st, int batch) {
    pdl_wait();
    pdl_launch_dependents();
    __shared__ int s_live;
    if (threadIdx.x == 0) s_live = 0;
    __syncthreads();
    for (int b = threadIdx.x; b < batch; b += 256) {
        const int live = st.done[b] ? 0 : 1;
        st.drafting[b] = live;
        st.block_len[b] = 0;
        if (live) atomicAdd(&s_live, 1);
    }
    __syncthreads();
    if (threadIdx.x == 0) { st.counters[7] = s_live; st.counters[9] = 0; }
}

// After draft step s (0-based): the router's decision for every sequence that is still drafting.  The last cluster to
// finish publishes (router ticket, sequences still drafting) to the host.
// logits: [batch][V] of this step; emb: the small model's embedding table [V][d].
// grid: (RT_CLUSTER, batch), a cluster per sequence; block: RT_THREADS.
template <typename T>
__global__ void __launch_bounds__(RT_THREADS) router_kernel(LoopState st, int batch, const float* __restrict__ logits, int V, int s,
                                                            int gamma_max, const T* __restrict__ emb, int d, RouterArgs r) {
    extern __shared__ float s_x[];                       // the feature vector, 1 + k + k * d floats
    __shared__ RouterPart s_slice[RT_CLUSTER];           // by rank, written by every CTA of the cluster
    __shared__ RouterPart s_warp[RT_WARPS], s_own, s_row;
    __shared__ float s_share[RT_CLUSTER];                // CTA 0: the CTAs' shares of w2 . hidden
    __shared__ float s_acc[RT_WARPS];
    cluster_arrive_relaxed();   // opening handshake: waited for before the first remote store
    const int rank = blockIdx.x, b = blockIdx.y, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int F = 1 + r.k + r.k * d;
    constexpr int PF = 64;                               // weights per lane of this warp's first hidden unit, fetched ahead (parameters)
    const int u0 = rank + RT_CLUSTER * warp;
    float wpre[PF];
#pragma unroll
    for (int i = 0; i < PF; ++i) wpre[i] = u0 < r.hidden && lane + 32 * i < F ? __ldg(r.w1 + (size_t)u0 * F + lane + 32 * i) : 0.f;
    pdl_wait();
    pdl_launch_dependents();
    const int slice = (((V + RT_CLUSTER - 1) / RT_CLUSTER) + 3) & ~3;
    const int v0 = min(V, rank * slice), v1 = min(V, v0 + slice);
    cluster_wait();
    if (st.drafting[b]) {   // (uniform over the cluster)
        const float* row = logits + (size_t)b * V;
        // Up to RT_REGS of the slice's logits per thread stay in registers (32768 in the row); longer rows are read again for
        // each step (a launch 18.8 us at 32768 logits, 34.9 at 32776, 49.7 at 65536, 82 at 131072).  `each` visits this thread's logits.
        const bool in_regs = slice <= RT_THREADS * RT_REGS;
        float x[RT_REGS];
        if (in_regs) {
#pragma unroll
            for (int i = 0; i < RT_REGS; ++i) x[i] = v0 + tid + i * RT_THREADS < v1 ? __ldcg(row + v0 + tid + i * RT_THREADS) : -INFINITY;
        }
        auto each = [&](auto visit) {
            if (in_regs) {
#pragma unroll
                for (int i = 0; i < RT_REGS; ++i) visit(x[i], v0 + tid + i * RT_THREADS);
            } else {
#pragma unroll 1
                for (int i = v0 + tid; i < v1; i += RT_THREADS) visit(__ldcg(row + i), i);
            }
        };
        // the warp's k best entries, one after the other: the best of those that come after the last one found
        float pv = INFINITY, wm = -INFINITY;
        int pi = -1;
#pragma unroll 1
        for (int j = 0; j < r.k; ++j) {
            float bv = -INFINITY;
            int bi = INT_MAX;
            each([&](float v, int i) {   // (indices rise: on equal values the first one stays)
                if (v > bv && (v < pv || (v == pv && i > pi))) { bv = v; bi = i; }
            });
            rt_warp_best(bv, bi);
            pv = bv; pi = bi;
            if (j == 0) wm = bv;
            if (lane == 0) { s_warp[warp].val[j] = bv; s_warp[warp].idx[j] = bi; }
        }
        // exponential sums relative to the warp's maximum (an empty share: -inf, zeros)
        float z = 0.f, s1 = 0.f;
        if (wm > -INFINITY)
            each([&](float v, int) {
                const float t = fmaxf(v - wm, -200.f), e = expf(t);   // (past the row's end: -inf, whose exponential is zero as that of -200 is)
                z += e;
                s1 = fmaf(e, t, s1);
            });
        z = warp_sum(z);
        s1 = warp_sum(s1);
        if (lane == 0) { s_warp[warp].m = wm; s_warp[warp].z = z; s_warp[warp].s1 = s1; }
        __syncthreads();
        if (warp == 0) rt_merge(s_warp, r.k, s_own, lane);
        __syncthreads();
        for (int i = tid; i < RT_CLUSTER * RT_PART_WORDS; i += RT_THREADS) {   // to every CTA of the cluster, itself included
            const int to = i / RT_PART_WORDS, w = i - to * RT_PART_WORDS;
            st_dsmem_f32(smem_u32(reinterpret_cast<float*>(&s_slice[rank]) + w), to, reinterpret_cast<const float*>(&s_own)[w]);
        }
        cluster_sync_all();
        if (warp == 0) rt_merge(s_slice, r.k, s_row, lane);
        __syncthreads();
        // the feature vector into shared memory, then this CTA's hidden units: warp w takes units rank + 8 w, rank + 8 (w + 8), ..
        if (tid == 0) s_x[0] = logf(s_row.z) - s_row.s1 / s_row.z;          // entropy: -sum q log q with q = e / z
        if (tid < r.k) s_x[1 + tid] = expf(s_row.val[tid] - s_row.m) / s_row.z;
        constexpr int VN = VecN<T>::N;                    // (d is a multiple of 8)
        for (int v = tid; v < r.k * (d / VN); v += RT_THREADS) {
            const int j = v / (d / VN), e = (v - j * (d / VN)) * VN;
            const int id = s_row.idx[j] == INT_MAX ? 0 : s_row.idx[j];
            float f[VN];
            load_vec(emb + (size_t)id * d + e, f);
#pragma unroll
            for (int i = 0; i < VN; ++i) s_x[1 + r.k + j * d + e + i] = f[i];
        }
        __syncthreads();
        float acc = 0.f;                                  // this warp's share of w2 . relu(hidden)
#pragma unroll 1
        for (int u = u0; u < r.hidden; u += RT_CLUSTER * RT_WARPS) {
            const float* wr = r.w1 + (size_t)u * F;
            float dot = 0.f;
            int f0 = lane;
            if (u == u0) {
#pragma unroll
                for (int i = 0; i < PF; ++i) if (lane + 32 * i < F) dot = fmaf(wpre[i], s_x[lane + 32 * i], dot);
                f0 = lane + 32 * PF;
            }
#pragma unroll 8
            for (int f = f0; f < F; f += 32) dot = fmaf(__ldg(wr + f), s_x[f], dot);
            dot = warp_sum(dot) + __ldg(r.b1 + u);
            acc = fmaf(__ldg(r.w2 + u), fmaxf(dot, 0.f), acc);
        }
        if (lane == 0) s_acc[warp] = acc;
        __syncthreads();
        if (tid == 0) {
            float share = 0.f;
            for (int w = 0; w < RT_WARPS; ++w) share += s_acc[w];
            st_dsmem_f32(smem_u32(&s_share[rank]), 0, share);
        }
        cluster_sync_all();
        if (rank == 0 && tid == 0) {
            float pre = r.b2;
            for (int c = 0; c < RT_CLUSTER; ++c) pre += s_share[c];
            const float disagree = 1.0f / (1.0f + expf(-pre));
            const float conf = 1.0f - disagree;
            st.block_len[b] = s + 1;
            st.confidence[b * st.gamma_limit + s] = conf;
            if (!(conf >= r.tau) || s + 1 >= gamma_max) {
                st.drafting[b] = 0;
                atomicSub(st.counters + 7, 1);
            }
        }
    }
    // the last cluster of the launch publishes to the host: data first, then the ticket it polls on
    if (rank == 0 && tid == 0) {
        __threadfence();
        const int t = atomicAdd(st.counters + 9, 1);
        if (t == batch - 1) {
            st.counters[9] = 0;
            __threadfence();
            const int ticket = st.counters[8] + 1;
            st.counters[8] = ticket;
            st.host_flags[6] = atomicAdd(st.counters + 7, 0);
            __threadfence_system();
            st.host_flags[5] = ticket;
        }
    }
}

}  // namespace tandem
