// Sampled Tandem + SPEED (Section 3.1 builds on the SPEED / speculative-decoding framework): drafts are drawn from
// the small model's distribution q = softmax(logits_S / T_S); draft r is kept with probability min(1, p(d_r) / q(d_r)),
// p = softmax(logits_L / T_L); at the first rejection the token is redrawn from the positive part of p - q; if every
// draft is kept, one more token is drawn from the large model's next distribution.
//
// Every draw uses one uniform variate from a counter-based generator keyed by (seed, sequence, iteration, slot):
// slots 0..gamma-1 draw the drafts, 16 + r tests draft r, 48 redraws.  A draw from weights w with variate u returns
// the first index whose running sum exceeds u * sum(w).  The running sums are fp32: each warp owns a contiguous range of
// the row, the ranges' sums are scanned in range order, and the warp whose range contains the target finds the index by
// its 32-weight pieces' sums, then inside the piece.
//
// A row of logits is dealt to the eight CTAs of a cluster and stays in registers between the maximum, the sums and the
// search (up to 32768 logits; longer rows are read again for each step: a launch, on average over draws, sums and decisions, 11.3 us
// at 32768 logits, 14.3 at 32776, 17.3 at 65536, 25.4 at 131072, a microsecond or two of it event overhead).  One CTA per row was bound by the
// passes over the row following one another: 32000 logits, four sequences, three drafts, a draw 12.1 us and the decisions
// 45.2 us.  The maxima and sums that the accept tests need come from the draws (small model) and from a launch over all rows
// of the block (large model) instead of four passes per draft in the deciding CTA.
#pragma once
#include <math.h>
#include "common.cuh"
#include "gemm_simt.cuh"
#include "misc_kernels.cuh"
#include "tc_common.cuh"

namespace tandem {

constexpr int SMP_SLOT_ACCEPT = 16;
constexpr int SMP_SLOT_REDRAW = 48;

__device__ __forceinline__ float uniform_variate(unsigned long long seed, int seq, int iteration, int slot) {
    const unsigned long long x = splitmix64(splitmix64(splitmix64(splitmix64(seed) ^ (unsigned long long)seq) ^ (unsigned long long)iteration) ^
                                            (unsigned long long)slot);
    return (float)(x >> 40) * (1.0f / 16777216.0f);   // 24 bits: exact in fp32
}

constexpr int SMC_THREADS = 256, SMC_WARPS = SMC_THREADS / 32, SMC_CLUSTER = 8;
constexpr int SMC_RANGES = SMC_CLUSTER * SMC_WARPS;          // contiguous ranges of a row, one per warp of the cluster
constexpr int SMC_REGS = 16;                                 // weights per lane, one of each 32-weight piece of the range

// One draw by a cluster from the weights weight(load(i), m), i in [0, V).  RELMAX: the weights are relative to the maximum m of
// load(i), exp((x - m) * inv_t), and every warp takes its own range's maximum until the ranges' records meet; otherwise they
// are absolute (m = 0).  Every CTA gets every range's (m, sum); the one warp whose range contains u * total finds the index and
// returns it in all of its lanes (all other warps return -1).  *m_out, *total_out (nullable): the row's maximum and the total
// relative to it.  box: SMC_RANGES float2 of shared memory, written by all CTAs of the cluster, whose opening handshake must
// be closed.  All threads of the cluster take part.
template <bool RELMAX, typename L, typename W>
__device__ __forceinline__ int smc_draw(L load, W weight, int V, int rank, float inv_t, float u, float2* box, float* m_out, float* total_out) {
    const int lane = threadIdx.x & 31, id = rank * SMC_WARPS + (threadIdx.x >> 5);
    const int chunk = (((V + SMC_RANGES - 1) / SMC_RANGES) + 31) & ~31;
    const int i0 = min(V, id * chunk), i1 = min(V, i0 + chunk);
    const bool in_regs = chunk <= 32 * SMC_REGS;             // (uniform) else the range is read again for each step
    float m = RELMAX ? -INFINITY : 0.f, local = 0.f;
    float p[SMC_REGS];
    if (in_regs) {
        decltype(load(0)) x[SMC_REGS];
#pragma unroll
        for (int j = 0; j < SMC_REGS; ++j) x[j] = load(min(i0 + 32 * j + lane, V - 1));
        if constexpr (RELMAX) {
#pragma unroll
            for (int j = 0; j < SMC_REGS; ++j) m = fmaxf(m, i0 + 32 * j + lane < i1 ? x[j] : -INFINITY);
            m = warp_max(m);
        }
#pragma unroll
        for (int j = 0; j < SMC_REGS; ++j) {
            p[j] = i0 + 32 * j + lane < i1 ? weight(x[j], m) : 0.f;
            local += p[j];
        }
    } else {
        if constexpr (RELMAX) {
#pragma unroll 8
            for (int i = i0 + lane; i < i1; i += 32) m = fmaxf(m, load(i));
            m = warp_max(m);
        }
#pragma unroll 8
        for (int i = i0 + lane; i < i1; i += 32) local += weight(load(i), m);
    }
    local = warp_sum(local);
    if (lane < SMC_CLUSTER) {
        st_dsmem_f32(smem_u32(&box[id].x), lane, m);
        st_dsmem_f32(smem_u32(&box[id].y), lane, local);
    }
    cluster_sync_all();
    // ranges 2 L and 2 L + 1 in lane L: common maximum, sums relative to it, inclusive running sums
    const float2 a = box[2 * lane], b = box[2 * lane + 1];
    const float M = warp_max(fmaxf(a.x, b.x));
    const float sa = a.x > -INFINITY ? a.y * expf((a.x - M) * inv_t) : 0.f, sb = b.x > -INFINITY ? b.y * expf((b.x - M) * inv_t) : 0.f;
    float incl = sa + sb;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const float q = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += q;
    }
    const float total = __shfl_sync(0xffffffffu, incl, 31);
    const float prev = __shfl_up_sync(0xffffffffu, incl, 1);
    const float before = lane > 0 ? prev : 0.f;                   // running sum ahead of this lane's pair
    const float target = u * total;
    if (m_out) *m_out = M;
    if (total_out) *total_out = total;
    // the first range whose running sum exceeds the target; rounding may leave none: then the last range with any weight
    const bool in_a = before + sa > target;
    const unsigned hit = __ballot_sync(0xffffffffu, in_a || incl > target), some = __ballot_sync(0xffffffffu, sa > 0.f || sb > 0.f);
    const int from = hit ? __ffs(hit) - 1 : (some ? 31 - __clz(some) : 0);
    const bool second = hit ? !in_a : sb > 0.f;
    const bool own_second = __shfl_sync(0xffffffffu, (int)second, from) != 0;
    const float excl = __shfl_sync(0xffffffffu, second ? before + sa : before, from);
    if (2 * from + (own_second ? 1 : 0) != id) return -1;
    const float f = m > -INFINITY ? expf((m - M) * inv_t) : 0.f;
    int pick = -1, last = -1;                                     // last: the range's last positive weight, where rounding fell short of the target
    if (in_regs) {
        // sums of the 32-weight pieces (lanes 2 j and 2 j + 1 get piece j), then the piece that contains the target
        float q[SMC_REGS];
#pragma unroll
        for (int j = 0; j < SMC_REGS; ++j) q[j] = p[j];
        const float two = warp_sum_many<SMC_REGS>(q, lane) * f;
        const float piece = __shfl_sync(0xffffffffu, two, (2 * lane) & 31);
        float run = lane < SMC_REGS ? piece : 0.f;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const float t = __shfl_up_sync(0xffffffffu, run, o);
            if (lane >= o) run += t;
        }
        const unsigned ph = __ballot_sync(0xffffffffu, lane < SMC_REGS && excl + run > target);
        if (hit && ph) {
            const int j = __ffs(ph) - 1;
            const float upto = __shfl_sync(0xffffffffu, run, max(j - 1, 0));
            const float ahead = excl + (j > 0 ? upto : 0.f);
            float x = 0.f;
#pragma unroll
            for (int jj = 0; jj < SMC_REGS; ++jj) if (jj == j) x = p[jj];
            x *= f;
            float s = x;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const float t = __shfl_up_sync(0xffffffffu, s, o);
                if (lane >= o) s += t;
            }
            const unsigned eh = __ballot_sync(0xffffffffu, ahead + s > target), pos = __ballot_sync(0xffffffffu, x > 0.f);
            if (eh) pick = i0 + 32 * j + __ffs(eh) - 1;
            else if (pos) pick = i0 + 32 * j + 31 - __clz(pos);
        }
#pragma unroll
        for (int j = 0; j < SMC_REGS; ++j) if (p[j] > 0.f) last = i0 + 32 * j + lane;
    } else {
        float run = excl;
        for (int base = i0; base < i1 && pick < 0; base += 32) {
            const int i = base + lane;
            const float x = i < i1 ? weight(load(i), m) * f : 0.f;
            if (x > 0.f) last = i;
            float s = x;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const float t = __shfl_up_sync(0xffffffffu, s, o);
                if (lane >= o) s += t;
            }
            const unsigned eh = __ballot_sync(0xffffffffu, run + s > target);
            if (hit && eh) pick = base + __ffs(eh) - 1;
            run += __shfl_sync(0xffffffffu, s, 31);
        }
    }
    if (pick < 0) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) last = max(last, __shfl_xor_sync(0xffffffffu, last, o));
        pick = max(last, 0);   // (all weights zero: index 0)
    }
    return pick;
}

// Draft s of every live sequence, drawn from softmax(logits / temp).  logits: [batch][V] of draft step s; stats[b] receives
// the row's maximum and the sum of its weights.  grid: (SMC_CLUSTER, batch), a cluster per sequence; block: SMC_THREADS.
__global__ void __launch_bounds__(SMC_THREADS) sample_draft_kernel(LoopState st, const float* __restrict__ logits, int V, int s,
                                                                   float temp, unsigned long long seed, float2* __restrict__ stats) {
    __shared__ float2 box[SMC_RANGES];
    cluster_arrive_relaxed();   // opening handshake
    pdl_wait();
    pdl_launch_dependents();
    cluster_wait();
    const int b = blockIdx.y;
    const float* row = logits + (size_t)b * V;
    const float inv_t = 1.0f / temp;
    const float u = uniform_variate(seed, b, st.counters[0], s);
    float m, z;
    const int tok = smc_draw<true>([&](int i) { return __ldcg(row + i); }, [&](float x, float mx) { return expf((x - mx) * inv_t); }, V, blockIdx.x,
                                   inv_t, u, box, &m, &z);
    if (tok >= 0 && (threadIdx.x & 31) == 0) { st.drafts[b * st.gamma_limit + s] = tok; stats[b] = make_float2(m, z); }
}

// Maximum and sum of weights of every row of the large model's block.  logits: [rows][V].
// grid: (SMC_CLUSTER, rows); block: SMC_THREADS.
__global__ void __launch_bounds__(SMC_THREADS) sample_stats_kernel(const float* __restrict__ logits, int V, float temp, float2* __restrict__ stats) {
    __shared__ float2 box[SMC_RANGES];
    cluster_arrive_relaxed();   // opening handshake
    pdl_wait();
    pdl_launch_dependents();
    cluster_wait();
    const float* row = logits + (size_t)blockIdx.y * V;
    const float inv_t = 1.0f / temp;
    float m, z;
    smc_draw<true>([&](int i) { return __ldcg(row + i); }, [&](float x, float mx) { return expf((x - mx) * inv_t); }, V, blockIdx.x, inv_t, 0.f, box,
                   &m, &z);
    if (blockIdx.x == 0 && threadIdx.x == 0) stats[blockIdx.y] = make_float2(m, z);
}

// Accept / redraw decisions of one iteration, one cluster per sequence: writes accept_len[b] and, at index accept_len of
// the sequence's target array, the token that follows the kept drafts.  The bookkeeping (emit, advance n, publish)
// is done by verify_kernel in mode 4, which takes these decisions as given.
// logits_large: [batch][gamma+1][V] with stats_large per row; logits_small: [gamma][batch][V] with stats_small per row.
// grid: (SMC_CLUSTER, batch); block: SMC_THREADS.
__global__ void __launch_bounds__(SMC_THREADS) sample_verify_kernel(LoopState st, int batch, int gamma, const float* __restrict__ logits_large,
                                                                    const float* __restrict__ logits_small, int V, float temp_large,
                                                                    float temp_small, unsigned long long seed,
                                                                    const float2* __restrict__ stats_large, const float2* __restrict__ stats_small) {
    __shared__ float2 box[SMC_RANGES];
    cluster_arrive_relaxed();   // opening handshake
    pdl_wait();
    pdl_launch_dependents();
    cluster_wait();
    const int b = blockIdx.y, lane = threadIdx.x & 31;
    if (st.done[b]) return;     // (uniform over the cluster)
    const int iteration = st.counters[0];
    const float inv_tl = 1.0f / temp_large, inv_ts = 1.0f / temp_small;
    // lane a tests draft a (every warp for itself); the first rejection is the accept length
    bool rejected = false;
    if (lane < gamma) {
        const float* lrow = logits_large + ((size_t)b * (gamma + 1) + lane) * V;
        const float* srow = logits_small + ((size_t)lane * batch + b) * V;
        const int tok = st.drafts[b * st.gamma_limit + lane];
        const float2 sl = __ldcg(stats_large + b * (gamma + 1) + lane), ss = __ldcg(stats_small + lane * batch + b);
        const float pL = expf((__ldcg(lrow + tok) - sl.x) * inv_tl) / sl.y;
        const float pS = expf((__ldcg(srow + tok) - ss.x) * inv_ts) / ss.y;
        const float ratio = pS > 0.f ? fminf(1.0f, pL / pS) : 1.0f;
        rejected = !(uniform_variate(seed, b, iteration, SMP_SLOT_ACCEPT + lane) < ratio);
    }
    const unsigned mask = __ballot_sync(0xffffffffu, rejected);
    const int a = mask ? __ffs(mask) - 1 : gamma;
    const float u = uniform_variate(seed, b, iteration, SMP_SLOT_REDRAW);
    // the positive part of p - q at the first rejection, or the large model's next distribution
    const float* lr = logits_large + ((size_t)b * (gamma + 1) + a) * V;
    const float* sr = logits_small + ((size_t)(a < gamma ? a : 0) * batch + b) * V;
    const float2 sl = __ldcg(stats_large + b * (gamma + 1) + a);
    const float2 ss = a < gamma ? __ldcg(stats_small + a * batch + b) : make_float2(0.f, 1.f);
    const float cl = 1.0f / sl.y, cs = 1.0f / ss.y;
    int tok = smc_draw<false>([&](int i) { return make_float2(__ldcg(lr + i), a < gamma ? __ldcg(sr + i) : 0.f); },
                              [&](float2 x, float) {
                                  const float l = expf((x.x - sl.x) * inv_tl);
                                  return a < gamma ? fmaxf(l * cl - expf((x.y - ss.x) * inv_ts) * cs, 0.f) : l;
                              }, V, blockIdx.x, inv_tl, u, box, nullptr, nullptr);
    if (lane != 0) tok = -1;
    if (tok >= 0) {
        st.accept_len[b] = a;
        st.targets[b * (st.gamma_limit + 1) + a] = tok;
    }
}

}  // namespace tandem
