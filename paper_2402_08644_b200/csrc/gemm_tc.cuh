// bf16 GEMMs  y[m][n] = sum_k x[m][k] * W[n][k]  on the tcgen05 tensor cores, fp32 accumulation in TMEM.
//
//  gemm_tc_decode_kernel   few rows (<= 64): the weight matrix is the MMA's A operand (128 output features
//                          per tile on the TMEM lanes), the token rows are the B operand (16..64 columns).
//                          The job is streaming W once from HBM: every CTA owns one (tile, K-slice) unit so
//                          that all SMs pull weights, tiles arrive by TMA through a ring of stages, and the
//                          K-slices of a tile sit in one thread-block cluster: each CTA sends its partial
//                          sums to the CTA that finishes those token rows (remote shared-memory stores), which
//                          adds them in slice order.
//                          LayerNorm ahead of a map is applied behind it:
//                          LN(x) W^T = r ((x - c).g) W^T - r (m - c) (g W^T) + b W^T
//                          with the row's mean m and reciprocal deviation r.  The producer of x leaves (x - c).g in two bf16
//                          planes, with c near m (see NextLn: a bit of the planes is lost for every doubling of |m - c| beyond the
//                          deviation), g and b ride along as four more rows of the B operand (each as value + remainder), and
//                          the row's statistics are merged while the products run, so nothing but TMA stands between
//                          the producer and the MMAs (PRO_LNT).  Activations enter the product as the sum of two bf16 numbers (the rounded value and the rounded
//                          remainder, about 16 significant bits): the B tile holds, for every 16 token rows, their values followed
//                          by their remainders, one MMA of N = 2 NB covers both (the weight tile is read
//                          from shared memory once), and the epilogue adds the two accumulator columns of a
//                          token row.  The kernel streams weights, so the wider B operand costs no bandwidth.
//                          The weight loads are issued before the kernel waits for its predecessor in the
//                          stream (programmatic dependent launch), so they overlap its run; a kernel lets its
//                          own successor start once the predecessor is done, which keeps one kernel's worth of
//                          prefetch in flight (deeper chains of waiting kernels cost more than they hide).
//  gemm_tc_pair_kernel     many rows (prompt pass): 256 x 256 output tiles, one per pair of multiprocessors, both operands by
//                          TMA; persistent, with two accumulators in TMEM, so that a tile's epilogue runs under the next
//                          tile's MMAs.
//  gemm_tc_split_kernel    prompt passes whose 256 x 256 tiles would leave multiprocessors idle: 128 x 128 tiles, one per
//                          cluster of one, two or four CTAs that share the tile's K range.
//
// Decode kernel: an output element's reduction order depends on (N, K) only, never on the number of rows, so a block
// pass and a one-row pass give identical bits.  Prompt kernels: the kernel and the K-slices are chosen from the pass's rows too, so
// the last bits of a prompt's keys and values can depend on what it is batched with.
#pragma once
#include <limits.h>
#include "common.cuh"
#include "gemm_simt.cuh"
#include "tc_common.cuh"

namespace tandem {

// How the token rows become the B operand: PRO_BF16: bf16 rows as they are (remainder rows zero); PRO_LN: fp32 rows
// of at most 1024 elements, LayerNorm, then value + remainder; PRO_F32: fp32 rows as value + remainder; PRO_TMA: the producer of the rows has
// already written them as two bf16 planes (values, remainders), and TMA brings them into the B stages beside the
// weights (no registers, no rounds, nothing for warps 0-3 to do before the epilogue).
// PRO_LNT: LayerNorm rows, (x - c).g by TMA like PRO_TMA and the rest in the epilogue (see above); the small pair's maps behind a
// LayerNorm took 4.4 us of the stream's time with the rows normalised in the prologue of every CTA (batch 1, 2), and
// 4.4 + 1.9 us with a LayerNorm kernel of their own (more sequences).
enum { PRO_BF16 = 0, PRO_LN = 1, PRO_F32 = 2, PRO_TMA = 3, PRO_LNT = 4 };
constexpr int EPI_SCORE = 7;                        // many rows: no store, per row and SCORE_TILE features (max, index, sum of exp(y - max)), and y at a given feature
constexpr int SCORE_TILE = 64;
enum { TC_ERR_SLOT = 1, TC_ERR_OPERANDS = 2, TC_ERR_ACCUM = 3, TC_ERR_EXCHANGE = 4 };   // which bounded wait gave up

struct TcDecodeArgs {
    const void* x;          // PRO_BF16: bf16 [rows][ldx];  PRO_LN / PRO_F32: float [rows][ldx];  PRO_TMA: unused (tensor map)
    int ldx;
    int x_row0;                 // PRO_TMA: first token row of this launch
    int release_early;          // PRO_TMA: the successor is released right after the wait on the predecessor (a small matrix:
                                // a chain of dependent steps, nothing to protect) instead of after the last token-row loads
    const float* ln_g;      // PRO_LN: LayerNorm gain / bias [K]
    const float* ln_b;
    int ln_row;             // PRO_LNT: first of the four rows of this LayerNorm in its tensor map
    const float2* ln_stats; // PRO_LNT: [rows][ln_groups], see NextLn
    int ln_groups;
    const float* ln_ref;    // PRO_LNT: [rows] c of the planes, see NextLn
    float* ln_mean;         // PRO_LNT: [rows] the rows' means, which the first CTA leaves for the producer of the next LayerNorm's planes
    int rows, K, N;         // N = output features over all segments
    int seg_rows0, tiles0;  // output features and tiles of the first weight segment (one tensor map per segment)
    int seg_rows;           // output features of every further segment
    int tiles_per_seg;      // ceil(seg_rows / 128)
    int splits;             // K-slices per tile: 1, 2, 4 or 8 = the cluster size; grid = tiles * splits
    int stream_weights;     // 1: weights are read once per pass and should not stay in L2
    int wait_first;         // 1: nothing is read before the wait on the preceding kernel (a stand-alone call: whatever precedes
                            // it may be writing the weights)
    int* err_flag;          // nullable
    unsigned poll_limit;    // polls before a wait on an mbarrier gives up; 0 = MBAR_POLL_LIMIT
    int rows_early;         // EPI_QKV / EPI_KV: the row arrays are older than the preceding kernel, and fetched ahead of the wait on it
    int withhold_weights;   // test hook for the give-up path: the TMA thread issues no loads, so the wait for
                            // operands must run out (nothing is in flight when the kernel leaves)
    float* amax_val;        // EPI_ARGMAX: [rows][amax_stride] best value per tile
    int* amax_idx;          //             and its output feature
    int amax_stride;
    EpiArgs e;
};

// The same pass from its row r0 on (nr rows): everything that is indexed by token row moves along.
template <int PRO, int EPI>
inline void tcd_shift_rows(TcDecodeArgs& a, int r0, int nr) {
    a.rows = nr;
    a.x_row0 += r0;
    if (a.x) a.x = static_cast<const unsigned char*>(a.x) + (size_t)r0 * a.ldx * (PRO == PRO_BF16 ? 2 : 4);
    if (PRO == PRO_LNT) { a.ln_stats += (size_t)r0 * a.ln_groups; a.ln_ref += r0; a.ln_mean += r0; }
    if (EPI == EPI_ARGMAX) { a.amax_val += (size_t)r0 * a.amax_stride; a.amax_idx += (size_t)r0 * a.amax_stride; }
    EpiArgs& e = a.e;
    if (e.out) e.out = static_cast<unsigned char*>(e.out) + (size_t)r0 * e.ldo * ((EPI == EPI_QKV || EPI == EPI_STORE || e.out_lo) ? 2 : 4);
    if (e.out_lo) e.out_lo = static_cast<unsigned char*>(e.out_lo) + (size_t)r0 * e.ldo * 2;   // (value / remainder planes are bf16)
    if (e.row_seq) { e.row_seq += r0; e.row_pos += r0; }
    if (e.snap) e.snap = static_cast<float*>(e.snap) + (size_t)r0 * e.snap_ld;
    if (e.ln.gain) { e.ln.hi += (size_t)r0 * e.ldo; e.ln.lo += (size_t)r0 * e.ldo; e.ln.stats += (size_t)r0 * e.ln.groups; e.ln.ref += r0; }
}

constexpr int TCD_THREADS = 192;   // warps 0-3: B operand + epilogue; warp 4: TMA; warp 5: TMEM + MMA issue
template <int NB, bool LNT> struct TcdCfg {
    static constexpr int NB2 = 2 * NB;              // B-operand rows = accumulator columns: for every 16 token rows their values, then their remainders
    static constexpr int N = NB2 + (LNT ? 16 : 0);  // ... and the LayerNorm's g, g's remainder, b, b's remainder (of 16 columns four are used)
    static constexpr int STAGES = NB <= 16 ? (LNT ? 4 : 5) : 3;   // two CTAs fit on an SM up to NB = 48 (at most 113 KB each with the static part)
    static constexpr int A_BYTES = 128 * 128;       // 128 weight rows x 64 bf16
    static constexpr int B_BYTES = NB2 * 128;       // 2 NB rows x 64 bf16
    static constexpr int LN_BYTES = LNT ? 4 * 128 : 0;
    static constexpr int STAGE_BYTES = A_BYTES + B_BYTES + (LNT ? 1024 : 0);   // (the MMA's last twelve B rows are whatever follows: unread columns)
    static constexpr int INBOX_BYTES = NB * 128 * 4;   // the K-slices' partial sums for the token rows this CTA finishes
    static constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + INBOX_BYTES + 1024;   // + slack to align the ring to 1024
    static constexpr int TMEM_COLS = N <= 32 ? 32 : (N <= 64 ? 64 : (N <= 128 ? 128 : 256));
};
static_assert(TcdCfg<16, true>::SMEM_BYTES + 1024 <= 113 * 1024 && TcdCfg<16, false>::SMEM_BYTES + 1024 <= 113 * 1024 &&
              TcdCfg<32, true>::SMEM_BYTES + 1024 <= 113 * 1024 && TcdCfg<48, true>::SMEM_BYTES + 1024 <= 113 * 1024,
              "two CTAs per SM: a kernel and its prefetching successor (static shared memory below 1 KB)");

// x = hi + lo with hi = bf16(x), lo = bf16(x - hi): the pair carries x to about 16 significant bits.
__device__ __forceinline__ void split_bf16x2(float x0, float x1, uint32_t& hi, uint32_t& lo) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(x0, x1);
    const __nv_bfloat162 l = __floats2bfloat162_rn(x0 - __low2float(h), x1 - __high2float(h));
    hi = *reinterpret_cast<const uint32_t*>(&h);
    lo = *reinterpret_cast<const uint32_t*>(&l);
}

__device__ __forceinline__ void tc_report(int* err_flag, int code) {
    if (err_flag) atomicExch(err_flag, code);
}
__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
    const __nv_bfloat162 p = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&p);
}
__device__ __forceinline__ float4 ln_apply(float4 x, float mu, float rs, float4 g, float4 b) {
    return make_float4((x.x - mu) * rs * g.x + b.x, (x.y - mu) * rs * g.y + b.y, (x.z - mu) * rs * g.z + b.z, (x.w - mu) * rs * g.w + b.w);
}

// Where column c of weight segment `seg` goes for EPI_QKV / EPI_KV: the query buffer (row stride ldo) or a cache.
// The address of (row j, column c) is base + row term + col, with the row term j * ldo or the cache row offset.
struct ScatterCol { bf16* base; long long col; bool is_q; };
template <int EPI>
__device__ __forceinline__ ScatterCol scatter_col(const EpiArgs& e, int seg, int c) {
    ScatterCol sc;
    int s = seg;
    if (EPI == EPI_QKV && s == 0) { sc.base = static_cast<bf16*>(e.out); sc.col = c; sc.is_q = true; return sc; }
    if (EPI == EPI_QKV) s -= 1;
    const int h = c / e.d_head, el = c - h * e.d_head;
    sc.base = static_cast<bf16*>(s == 0 ? e.kcache : e.vcache);
    sc.col = (long long)h * e.t_max * e.d_head + el;
    sc.is_q = false;
    return sc;
}

// grid: tiles * splits CTAs in clusters of `splits` (the K-slices of one tile); dynamic smem TcdCfg::SMEM_BYTES.
template <int NB, int PRO, int EPI>
__global__ void __launch_bounds__(TCD_THREADS)
gemm_tc_decode_kernel(const TcDecodeArgs a, const __grid_constant__ CUtensorMap tm0, const __grid_constant__ CUtensorMap tm1,
                      const __grid_constant__ CUtensorMap tm2, const __grid_constant__ CUtensorMap tmx,
                      const __grid_constant__ CUtensorMap tml) {
    constexpr bool LNT = PRO == PRO_LNT, BY_TMA = PRO == PRO_TMA || LNT;   // BY_TMA: the token rows are loaded beside the weights
    using C = TcdCfg<NB, LNT>;
    extern __shared__ __align__(1024) unsigned char smem_dyn[];
    __shared__ __align__(8) uint64_t s_full[C::STAGES];
    __shared__ __align__(8) uint64_t s_empty[C::STAGES];
    __shared__ __align__(8) uint64_t s_accum;
    __shared__ __align__(8) uint64_t s_inbox;   // counts the bytes of the K-slices' partial sums sent to this CTA
    __shared__ uint32_t s_tmem;
    __shared__ float s_mu[NB], s_rstd[NB];   // LayerNorm prologues: the rows' means (PRO_LNT: less c) and reciprocal deviations;  EPI_RESID: s_mu[s] = c of row j_first + s
    __shared__ long long s_rowoff[NB];   // EPI_QKV / EPI_KV: the row-dependent part of an output's cache index

    const int tid = threadIdx.x, warp = warp_uniform(tid >> 5), lane = tid & 31;
    const uint32_t ring0 = (smem_u32(smem_dyn) + 1023u) & ~1023u;          // shared-space address of stage 0
    unsigned char* ring = smem_dyn + (ring0 - smem_u32(smem_dyn));         // the same place as a generic pointer

    const int S = a.splits;
    const uint32_t poll_limit = a.poll_limit ? a.poll_limit : MBAR_POLL_LIMIT;
    const int unit = blockIdx.x;
    const int tile = unit / S, sp = unit - tile * S;                       // sp = this CTA's rank in its cluster
    const int seg = tile < a.tiles0 ? 0 : 1 + (tile - a.tiles0) / a.tiles_per_seg;
    const int n_local0 = (seg == 0 ? tile : tile - a.tiles0 - (seg - 1) * a.tiles_per_seg) * 128;
    const int seg_rows = seg == 0 ? a.seg_rows0 : a.seg_rows;               // output features of this tile's segment
    const int seg_base = seg == 0 ? 0 : a.seg_rows0 + (seg - 1) * a.seg_rows;   // and its first output feature
    const int KB = (a.K + 63) >> 6;
    const int kb_base = KB / S, kb_rem = KB - kb_base * S;
    const int kb0 = sp * kb_base + min(sp, kb_rem);
    const int nkb = kb_base + (sp < kb_rem ? 1 : 0);
    const int K4 = a.K >> 2;
    // LayerNorm rows (they sit in registers, 8 float4 per lane) and a K-slice that fits the ring without reuse: the B
    // operand is then written straight from the registers that gave the statistics.
    const bool ln_regs = PRO == PRO_LN && nkb <= C::STAGES;
    // Token rows whose outputs this CTA finishes: all of them without split-K, else a contiguous share of ceil(rows / S).
    const int rpc = S == 1 ? a.rows : (a.rows + S - 1) / S;
    const int j_first = S == 1 ? 0 : sp * rpc;
    const int j_count = max(0, min(rpc, a.rows - j_first));
    float hres[EPI == EPI_RESID ? NB : 1];   // EPI_RESID: the residual values this thread's outputs are added to
    float next_gain = 0.f;                   // EPI_RESID: gain of the LayerNorm that follows, at this thread's feature (a parameter)
    const float inv_k = LNT ? 1.0f / (float)a.K : 0.f;
    int my_seq = 0, my_pos = 0;              // EPI_QKV / EPI_KV, threads below a.rows: this token row's sequence and position

    if (warp == 5) {
        if (lane == 0) {
            for (int s = 0; s < C::STAGES; ++s) {
                mbar_init(smem_u32(&s_full[s]), BY_TMA ? 2 : 5);   // the TMA thread's arrive + one per B-operand warp (BY_TMA: its second arrive)
                mbar_init(smem_u32(&s_empty[s]), 1);   // the MMA thread's commit
            }
            mbar_init(smem_u32(&s_accum), 1);
            mbar_init(smem_u32(&s_inbox), 1);
            mbar_init_fence();
        }
        __syncwarp();
        tmem_alloc(smem_u32(&s_tmem), C::TMEM_COLS);
        tmem_relinquish();
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = warp_uniform(s_tmem);
    if (S > 1) cluster_arrive_relaxed();   // opening handshake: waited for just before the first remote store

    if (warp == 4) {
        // ---- weight tiles: independent of every earlier kernel of a context, so no wait on the predecessor here ----
        if (a.wait_first) pdl_wait();
        const CUtensorMap* tm = seg == 0 ? &tm0 : (seg == 1 ? &tm1 : &tm2);
        const uint64_t pol = l2_policy_evict_first();
        auto load_a = [&](int i, int st) {
            const uint32_t bar = smem_u32(&s_full[st]);
            mbar_arrive_expect_tx(bar, C::A_BYTES + C::LN_BYTES);
            if (LNT) tma_load_2d_nohint(ring0 + st * C::STAGE_BYTES + C::A_BYTES + C::B_BYTES, &tml, (kb0 + i) * 64, a.ln_row, bar);   // parameters too
            if (a.stream_weights) tma_load_2d(ring0 + st * C::STAGE_BYTES, tm, (kb0 + i) * 64, n_local0, bar, pol);
            else tma_load_2d_nohint(ring0 + st * C::STAGE_BYTES, tm, (kb0 + i) * 64, n_local0, bar);
        };
        if (a.withhold_weights) {
            // (test hook: nothing is loaded)
        } else if (BY_TMA) {
            // Weights of the first ring-ful before the wait on the predecessor, then the wait, then their token rows
            // (boxes of 16 rows in both planes; a copy for each plane instead: the small model's output head 5.41 us, 4.80 like this), then weights and rows together as stages come free.
            auto load_b = [&](int i, int st) {
                const uint32_t bar = smem_u32(&s_full[st]);
                const uint32_t dst = ring0 + st * C::STAGE_BYTES + C::A_BYTES;
                mbar_arrive_expect_tx(bar, C::B_BYTES);
#pragma unroll
                for (int r16 = 0; r16 < NB; r16 += 16) tma_load_3d_nohint(dst + r16 * 256, &tmx, (kb0 + i) * 64, a.x_row0 + r16, 0, bar);   // values, remainders
            };
            const int n_pre = min(nkb, C::STAGES);
            if (elect_one()) {
                tma_prefetch_desc(tm);
                tma_prefetch_desc(&tmx);
                if (LNT) tma_prefetch_desc(&tml);
                for (int i = 0; i < n_pre; ++i) load_a(i, i);
            }
            pdl_wait();
            if (elect_one())
                for (int i = 0; i < n_pre; ++i) load_b(i, i);
            for (int i = n_pre; i < nkb; ++i) {
                const int st = i % C::STAGES;
                if (!mbar_wait_warp(smem_u32(&s_empty[st]), ((i / C::STAGES) - 1) & 1, poll_limit)) {
                    tc_report(a.err_flag, TC_ERR_SLOT);
                    break;
                }
                if (elect_one()) {
                    load_a(i, st);
                    load_b(i, st);
                }
            }
            pdl_launch_dependents();   // the last token rows are on their way: the successor may start (see the note at the epilogue)
        } else {
            if (elect_one()) tma_prefetch_desc(tm);
            for (int i = 0; i < nkb; ++i) {
                const int st = i % C::STAGES;
                if (i >= C::STAGES && !mbar_wait_warp(smem_u32(&s_empty[st]), ((i / C::STAGES) - 1) & 1, poll_limit)) {
                    tc_report(a.err_flag, TC_ERR_SLOT);
                    break;
                }
                if (elect_one()) load_a(i, st);
            }
        }
        __syncwarp();
    } else if (warp == 5) {
        // ---- MMA issue: one elected thread of a converged warp ----
        constexpr uint32_t idesc = umma_idesc_bf16(128, C::N);
        constexpr uint64_t NEXT = C::STAGE_BYTES / 16;   // a stage further on, in a descriptor's units
        uint64_t da = umma_desc_k_sw128(ring0), db = umma_desc_k_sw128(ring0 + C::A_BYTES);
        uint32_t phase = 0, ok = mbar_test(smem_u32(&s_full[0]), 0);
        for (int i = 0, st = 0; i < nkb; ++i) {
            if (!mbar_wait_tested(ok, smem_u32(&s_full[st]), phase, poll_limit)) {
                tc_report(a.err_flag, TC_ERR_OPERANDS);
                break;
            }
            tc_fence_after_sync();
            const int done = st;
            const uint64_t ka = da, kb = db;
            if (++st == C::STAGES) { st = 0; phase ^= 1; da -= (C::STAGES - 1) * NEXT; db -= (C::STAGES - 1) * NEXT; }
            else { da += NEXT; db += NEXT; }
            if (i + 1 < nkb) ok = mbar_test(smem_u32(&s_full[st]), phase);
            umma_bf16_k64(tmem, ka, kb, idesc, i != 0 ? 1u : 0u);
            umma_commit_one(smem_u32(&s_empty[done]));
        }
        umma_commit_one(smem_u32(&s_accum));
        // TMEM goes back as soon as the epilogue warps have read the accumulator (they arrive on barrier 2 right after
        // their loads), not at the end of the kernel: nothing is left to do for this warp after that.
        asm volatile("bar.sync 2, 160;" ::: "memory");
        tc_fence_after_sync();
        tmem_dealloc(tmem, C::TMEM_COLS);
    } else {
    // ---- warps 0-3: token rows into the B stages (then the epilogue) ----
    float4 gq[C::STAGES], bq[C::STAGES];   // register path: gain / bias of this lane's slot in each of the CTA's K-blocks
    if (a.wait_first) pdl_wait();
    if ((EPI == EPI_QKV || EPI == EPI_KV) && a.rows_early && tid < a.rows) { my_seq = __ldcg(a.e.row_seq + tid); my_pos = __ldcg(a.e.row_pos + tid); }
    if (EPI == EPI_RESID && a.e.ln.gain && n_local0 + tid < seg_rows) next_gain = __ldg(a.e.ln.gain + seg_base + n_local0 + tid);
    if (ln_regs) {
#pragma unroll
        for (int i = 0; i < C::STAGES; ++i) {
            const int k4 = ((kb0 + i) >> 1) * 32 + lane;
            const bool mine = i < nkb && ((kb0 + i) & 1) == (lane >> 4) && k4 < K4;
            gq[i] = mine ? __ldg(reinterpret_cast<const float4*>(a.ln_g) + k4) : make_float4(0.f, 0.f, 0.f, 0.f);
            bq[i] = mine ? __ldg(reinterpret_cast<const float4*>(a.ln_b) + k4) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
    }
    pdl_wait();   // x, and everything the epilogue touches, comes from earlier kernels; gains and biases are parameters
    if (EPI == EPI_QKV || EPI == EPI_KV) {
        // cache index of (row j, head h, element el) = ((seq_j * H + h) * t_max + pos_j) * d_head + el: the row part once
        // per row.  Only the epilogue needs it: the two loads are in flight while the B operand is produced, and the
        // barrier that publishes the offsets sits after that.
        if (tid < a.rows && !a.rows_early) {                                          // first used ahead of the epilogue
            if (a.e.row_seq) { my_seq = a.e.row_seq[tid]; my_pos = a.e.row_pos[tid]; }
            else my_seq = a.x_row0 + tid;                                             // stand-alone: row j is sequence j at position 0
        }
    }
    if (EPI == EPI_RESID) {
        // the residual-stream values this thread will add to: fetched now, off the critical path
        const float* hp = static_cast<const float*>(a.e.out);
        const int nl = n_local0 + tid;
#pragma unroll
        for (int s = 0; s < NB; ++s) {
            if (s >= j_count) break;   // (every loop over rows leaves at the last row: the unrolled rest is never fetched)
            hres[s] = nl < seg_rows ? __ldcg(hp + (size_t)(j_first + s) * a.e.ldo + seg_base + nl) : 0.f;
        }
        if (a.e.ln.gain && tid < j_count) s_mu[tid] = __ldcg(a.e.ln.ref + j_first + tid);   // (published by the barrier ahead of the epilogue)
    }
    if (ln_regs) {
        // short LayerNorm rows: one pass over x.  Lane L holds the row's float4 number L + 32u in
        // t[u], i.e. K-block 2u + (L >= 16), 16-byte chunk (L & 15) / 2, half L & 1.
        // A warp's rows are fetched one row ahead, so the loads of its rows overlap.
        float4 tn[8];
        if (warp < a.rows) {
            const float4* xr = reinterpret_cast<const float4*>(static_cast<const float*>(a.x) + (size_t)warp * a.ldx);
#pragma unroll
            for (int u = 0; u < 8; ++u) tn[u] = (lane + 32 * u < K4) ? __ldcg(xr + lane + 32 * u) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        pdl_launch_dependents();   // (a K-slice that fits the ring: see the note at the epilogue)
        for (int r = warp; r < a.rows; r += 4) {
            float4 t[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) t[u] = tn[u];
            if (r + 4 < a.rows) {
                const float4* xr = reinterpret_cast<const float4*>(static_cast<const float*>(a.x) + (size_t)(r + 4) * a.ldx);
#pragma unroll
                for (int u = 0; u < 8; ++u) tn[u] = (lane + 32 * u < K4) ? __ldcg(xr + lane + 32 * u) : make_float4(0.f, 0.f, 0.f, 0.f);
            }
            float s = 0.f;
#pragma unroll
            for (int u = 0; u < 8; ++u) s += (t[u].x + t[u].y) + (t[u].z + t[u].w);
            const float mu = warp_sum(s) / (float)a.K;
            float q = 0.f;
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                if (lane + 32 * u < K4) {
                    const float d0 = t[u].x - mu, d1 = t[u].y - mu, d2 = t[u].z - mu, d3 = t[u].w - mu;
                    q = fmaf(d0, d0, q); q = fmaf(d1, d1, q); q = fmaf(d2, d2, q); q = fmaf(d3, d3, q);
                }
            }
            const float rs = 1.0f / sqrtf(warp_sum(q) / (float)a.K + 1e-5f);
#pragma unroll
            for (int i = 0; i < C::STAGES; ++i) {
                const int kb = kb0 + i;
                if (i >= nkb) break;
                if ((kb & 1) == (lane >> 4)) {
                    const int u = kb >> 1;
                    float4 xv = t[0];
#pragma unroll
                    for (int uu = 1; uu < 8; ++uu) if (u == uu) xv = t[uu];
                    uint2 val = make_uint2(0u, 0u), rem = make_uint2(0u, 0u);   // beyond K the weights are zero-filled; so is x
                    if (u * 32 + lane < K4) {
                        const float4 y = ln_apply(xv, mu, rs, gq[i], bq[i]);
                        split_bf16x2(y.x, y.y, val.x, rem.x);
                        split_bf16x2(y.z, y.w, val.y, rem.y);
                    }
                    const int c = (lane & 15) >> 1;
                    unsigned char* bt = ring + i * C::STAGE_BYTES + C::A_BYTES + (NB > 16 ? (r & ~15) + r : r) * 128 + ((c ^ (r & 7)) << 4) + ((lane & 1) << 3);
                    *reinterpret_cast<uint2*>(bt) = val;
                    *reinterpret_cast<uint2*>(bt + 16 * 128) = rem;   // (the same swizzle phase)
                }
            }
        }
        // rows >= a.rows of the B tiles stay as they are: a column of the product depends on its own row only
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0)
            for (int i = 0; i < nkb; ++i) mbar_arrive(smem_u32(&s_full[i]));
    } else if (LNT) {
        // The rows' statistics from the groups' (mean, sum of squared deviations): eight lanes per row, four of a lane's groups
        // fetched at once, sums relative to the first group's mean.  For each row the order of the sums depends on K only.
        // (Fetched one after the other where a row has fewer than 32 groups, and with divisions behind the sums, they held the
        // products up: a one-row pass through a 512-wide map 2.79 us of the chain, 2.31 us like this, a layer of that width 13.1 -> 12.2 us.)
        if (nkb <= C::STAGES || a.release_early) pdl_launch_dependents();   // (see the note at the epilogue)
        for (int r0 = warp * 4; r0 < a.rows; r0 += 16) {
            const int r = r0 + (lane >> 3), gl = lane & 7;
            const float2* sp = a.ln_stats + (size_t)min(r, a.rows - 1) * a.ln_groups;
            const float ref = __ldcg(sp).x, c = __ldcg(a.ln_ref + min(r, a.rows - 1));
            float s = 0.f, q = 0.f;
#pragma unroll 1
            for (int g0 = gl; g0 < a.ln_groups; g0 += 32) {
                float2 p[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) p[u] = g0 + 8 * u < a.ln_groups ? __ldcg(sp + g0 + 8 * u) : make_float2(0.f, 0.f);
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const float n = (float)max(0, min(32, a.K - 32 * (g0 + 8 * u))), dm = p[u].x - ref;   // (0 past the last group)
                    s = fmaf(n, dm, s);
                    q += fmaf(n * dm, dm, p[u].y);
                }
            }
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) { s += __shfl_xor_sync(0xffffffffu, s, o); q += __shfl_xor_sync(0xffffffffu, q, o); }
            const float dmu = s * inv_k;
            if (gl == 0 && r < a.rows) {
                s_mu[r] = (ref - c) + dmu;
                if (unit == 0) a.ln_mean[r] = ref + dmu;
                s_rstd[r] = __frsqrt_rn(fmaf(fmaxf(q - s * dmu, 0.f), inv_k, 1e-5f));
            }
        }
        bar_sync(1, 128);
    } else if (!BY_TMA) {
        // general case: statistics (LayerNorm), then the K-blocks a ring's worth at a time
        if (PRO == PRO_LN) {
            for (int r = warp; r < a.rows; r += 4) {   // one warp per row, fixed lane-strided order
                const float4* xr = reinterpret_cast<const float4*>(static_cast<const float*>(a.x) + (size_t)r * a.ldx);
                float4 t[8];           // the same arithmetic as the register path above
#pragma unroll
                for (int u = 0; u < 8; ++u) t[u] = (lane + 32 * u < K4) ? __ldcg(xr + lane + 32 * u) : make_float4(0.f, 0.f, 0.f, 0.f);
                float s = 0.f;
#pragma unroll
                for (int u = 0; u < 8; ++u) s += (t[u].x + t[u].y) + (t[u].z + t[u].w);
                const float mu = warp_sum(s) / (float)a.K;
                float q = 0.f;
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    if (lane + 32 * u < K4) {
                        const float d0 = t[u].x - mu, d1 = t[u].y - mu, d2 = t[u].z - mu, d3 = t[u].w - mu;
                        q = fmaf(d0, d0, q); q = fmaf(d1, d1, q); q = fmaf(d2, d2, q); q = fmaf(d3, d3, q);
                    }
                }
                const float var = warp_sum(q) / (float)a.K;
                if (lane == 0) { s_mu[r] = mu; s_rstd[r] = 1.0f / sqrtf(var + 1e-5f); }
            }
            bar_sync(1, 128);
        }
        constexpr int CPT = NB * 8 / 128;   // 8-element chunks of the NB token rows of one K-block per thread
        for (int i0 = 0; i0 < nkb; i0 += C::STAGES) {
            // a ring's worth of K-blocks at a time: all loads first, so their latencies overlap
            uint4 raw[PRO == PRO_BF16 ? C::STAGES : 1][CPT];
            float4 raw32[PRO == PRO_BF16 ? 1 : C::STAGES][CPT][2];
#pragma unroll
            for (int g = 0; g < C::STAGES; ++g)
#pragma unroll
                for (int ch = 0; ch < CPT; ++ch) {
                    const int idx = tid + ch * 128, r = idx >> 3, c = idx & 7;
                    const int k = (kb0 + i0 + g) * 64 + c * 8;
                    const bool live = i0 + g < nkb && r < a.rows && k < a.K;
                    if (PRO == PRO_BF16) {
                        raw[g][ch] = live ? __ldcg(reinterpret_cast<const uint4*>(static_cast<const bf16*>(a.x) + (size_t)r * a.ldx + k))
                                          : make_uint4(0u, 0u, 0u, 0u);
                    } else {
                        const float4* xp = reinterpret_cast<const float4*>(static_cast<const float*>(a.x) + (size_t)r * a.ldx + k);
                        raw32[g][ch][0] = live ? __ldcg(xp) : make_float4(0.f, 0.f, 0.f, 0.f);
                        raw32[g][ch][1] = live ? __ldcg(xp + 1) : make_float4(0.f, 0.f, 0.f, 0.f);
                    }
                }
            if (nkb <= C::STAGES) pdl_launch_dependents();   // (a K-slice that fits the ring: see the note at the epilogue)
            bool dead = false;
#pragma unroll
            for (int g = 0; g < C::STAGES; ++g) {
                const int i = i0 + g;
                if (i >= nkb || dead) break;
                const int st = g;   // i0 is a multiple of STAGES
                if (i >= C::STAGES && !mbar_wait(smem_u32(&s_empty[st]), ((i / C::STAGES) - 1) & 1, poll_limit)) {
                    tc_report(a.err_flag, TC_ERR_SLOT);
                    dead = true;
                    break;
                }
                unsigned char* bt = ring + st * C::STAGE_BYTES + C::A_BYTES;
#pragma unroll
                for (int ch = 0; ch < CPT; ++ch) {
                    const int idx = tid + ch * 128, r = idx >> 3, c = idx & 7;
                    uint4 val = make_uint4(0u, 0u, 0u, 0u), rem = make_uint4(0u, 0u, 0u, 0u);
                    if (PRO == PRO_BF16) {
                        val = raw[g][ch];
                    } else {
                        const int k = (kb0 + i) * 64 + c * 8;
                        if (r < a.rows && k < a.K) {
                            float4 u0 = raw32[g][ch][0], u1 = raw32[g][ch][1];
                            if (PRO == PRO_LN) {
                                const float mu = s_mu[r], rs = s_rstd[r];
                                u0 = ln_apply(u0, mu, rs, __ldg(reinterpret_cast<const float4*>(a.ln_g + k)), __ldg(reinterpret_cast<const float4*>(a.ln_b + k)));
                                u1 = ln_apply(u1, mu, rs, __ldg(reinterpret_cast<const float4*>(a.ln_g + k) + 1), __ldg(reinterpret_cast<const float4*>(a.ln_b + k) + 1));
                            }
                            split_bf16x2(u0.x, u0.y, val.x, rem.x); split_bf16x2(u0.z, u0.w, val.y, rem.y);
                            split_bf16x2(u1.x, u1.y, val.z, rem.z); split_bf16x2(u1.z, u1.w, val.w, rem.w);
                        }
                    }
                    // 128-byte swizzle: the 16-byte chunk index is XORed with the row index modulo 8
                    unsigned char* dst = bt + (NB > 16 ? (r & ~15) + r : r) * 128 + ((c ^ (r & 7)) << 4);
                    *reinterpret_cast<uint4*>(dst) = val;
                    *reinterpret_cast<uint4*>(dst + 16 * 128) = rem;   // the remainder row of token row r (same swizzle phase)
                }
                fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&s_full[st]));
            }
        }
    }
    }

    // ---- epilogue: warps 0-3 own TMEM lanes 32 * warp .. +31 = output features of the tile ----
    float v[NB];
    const int tl = warp * 32 + lane;
    ScatterCol sc;
    if (warp < 4) {
        // The successor may start (set up, fetch its first weight tiles) once this kernel's token-row loads are out of
        // its way: right after they have been issued when the K-slice fits the ring (one round of loads; see above),
        // else here, after the last round has been written.  Letting it start right after the wait measured 2-3 %
        // slower per iteration (its CTAs' set-up and loads compete with the row loads); later than here (after the
        // accumulator is ready, or after the exchange) slower again (the successor's head start shrinks).
        // (BY_TMA with a K-slice longer than the ring and a matrix large enough to be a stream: the TMA thread does it, after
        // its last loads; otherwise there is nothing of this kernel's in the successor's way, and it is released at once)
        if (!BY_TMA || (!LNT && (nkb <= C::STAGES || a.release_early))) pdl_launch_dependents();
        if (EPI == EPI_QKV || EPI == EPI_KV) {
            if (tid < a.rows) s_rowoff[tid] = ((long long)my_seq * a.e.n_heads * a.e.t_max + my_pos) * a.e.d_head;
            bar_sync(1, 128);
        }
        if (EPI == EPI_RESID && a.e.ln.gain) bar_sync(1, 128);
        if (EPI == EPI_QKV || EPI == EPI_KV) sc = scatter_col<EPI>(a.e, seg, n_local0 + tl);   // (a division: ahead of the wait)
        if (!mbar_wait(smem_u32(&s_accum), 0, poll_limit)) tc_report(a.err_flag, TC_ERR_ACCUM);
        tc_fence_after_sync();
        float c1 = 0.f, c2 = 0.f;                     // PRO_LNT: this feature's (slice of) g W^T and b W^T
        const uint32_t acc = tmem + (static_cast<uint32_t>(warp * 32) << 16);
        uint32_t w[4] = {0u, 0u, 0u, 0u};
        if (LNT) tmem_issue4(acc + C::NB2, w);
#pragma unroll
        for (int c0 = 0; c0 < NB; c0 += 16) {
            if (c0 >= a.rows) break;                  // columns of absent token rows are never read
            uint32_t t[16], u[16];
            tmem_issue16(acc + 2 * c0, t);            // x's values times W
            tmem_issue16(acc + 2 * c0 + 16, u);       // x's remainders times W
            tmem_wait_ld(t, u, w);
            if (LNT && c0 == 0) {
                c1 = __uint_as_float(w[0]) + __uint_as_float(w[1]);
                c2 = __uint_as_float(w[2]) + __uint_as_float(w[3]);
            }
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                v[c0 + i] = __uint_as_float(t[i]) + __uint_as_float(u[i]);
                if (LNT) v[c0 + i] = fmaf(s_rstd[c0 + i], fmaf(-s_mu[c0 + i], c1, v[c0 + i]), c2);   // (rows past the last: never used)
            }
        }
        tc_fence_before_sync();
        asm volatile("bar.arrive 2, 160;" ::: "memory");   // the accumulator has been read: warp 5 may free the TMEM columns
    }
    const int n_local = n_local0 + tl;                 // warps 0-3: this thread's output feature
    const bool valid = n_local < seg_rows;
    const int n = seg_base + n_local;
    if (EPI == EPI_ARGMAX) {                            // whole tiles only (S == 1)
        if (warp < 4) {
            float* out = static_cast<float*>(a.e.out);
            float* s_av = reinterpret_cast<float*>(ring + C::STAGES * C::STAGE_BYTES);   // [4 warps][NB], where the inbox would be
            int* s_ai = reinterpret_cast<int*>(s_av + 4 * NB);
#pragma unroll
            for (int j = 0; j < NB; ++j) {
                if (j >= a.rows) break;
                {
                    float bv = valid ? v[j] : -INFINITY;
                    int bi = valid ? n : INT_MAX;
                    if (valid) out[(size_t)j * a.e.ldo + n] = v[j];
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) {
                        const float ov = __shfl_xor_sync(0xffffffffu, bv, o);
                        const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
                        if (ov > bv || (ov == bv && oi < bi)) { bv = ov; bi = oi; }
                    }
                    if (lane == 0) { s_av[warp * NB + j] = bv; s_ai[warp * NB + j] = bi; }
                }
            }
            bar_sync(1, 128);
            if (tid < a.rows) {
                float bv = s_av[tid];
                int bi = s_ai[tid];
                for (int w = 1; w < 4; ++w)
                    if (s_av[w * NB + tid] > bv || (s_av[w * NB + tid] == bv && s_ai[w * NB + tid] < bi)) { bv = s_av[w * NB + tid]; bi = s_ai[w * NB + tid]; }
                a.amax_val[(size_t)tid * a.amax_stride + tile] = bv;
                a.amax_idx[(size_t)tid * a.amax_stride + tile] = bi;
            }
        }
    } else {
        if (S > 1) {
            // The cluster's CTAs hold the K-slices of one tile, and CTA r finishes token rows [r * rpc, (r + 1) * rpc).
            // Every CTA sends each row's partial sums to the inbox of the CTA that finishes it, with stores that count
            // their bytes on the receiver's inbox barrier; a CTA that finishes rows waits until S x rows x 128 floats
            // have arrived and sums its inbox in slice order.  No cluster-wide barrier: a CTA without rows of its own
            // leaves right after sending, the others once everything addressed to them has arrived (nothing is
            // written into a CTA's shared memory after that).
            const uint32_t inbox0 = ring0 + C::STAGES * C::STAGE_BYTES;           // [S][rpc][128] fp32
            cluster_wait();   // closes the opening handshake: every CTA of the cluster is running
            if (warp < 4) {
                const uint32_t ibar = smem_u32(&s_inbox);
                if (tid == 0 && j_count > 0) mbar_arrive_expect_tx(ibar, (uint32_t)(S * j_count * 128 * 4));
                int dst = 0, jj = 0;
#pragma unroll
                for (int j = 0; j < NB; ++j) {
                    if (j >= a.rows) break;
                    st_async_dsmem_f32(inbox0 + ((sp * rpc + jj) * 128 + tl) * 4, ibar, dst, v[j]);
                    if (++jj == rpc) { jj = 0; ++dst; }
                }
                if (j_count > 0 && !mbar_wait(ibar, 0, poll_limit)) tc_report(a.err_flag, TC_ERR_EXCHANGE);
            }
            if (warp < 4) {
                const float* inbox = reinterpret_cast<const float*>(ring + C::STAGES * C::STAGE_BYTES);
#pragma unroll
                for (int s = 0; s < NB / 2; ++s) {
                    if (s >= j_count) break;
                    float acc = 0.f;
#pragma unroll
                    for (int ss = 0; ss < 8; ++ss) if (ss < S) acc += inbox[((ss * rpc + s) * 128) + tl];   // slice order
                    v[s] = acc;
                }
            }
        }
        // v[s] is now the finished product of token row j_first + s and this thread's feature
        if (warp < 4) {
            const int n_group = max(0, min(32, seg_rows - (n_local0 + warp * 32)));   // features of this warp's group of 32
#pragma unroll
            for (int s = 0; s < NB; ++s) {
                if (s >= j_count) break;
                {
                    const int j = j_first + s;
                    float hv = v[s];
                    if (EPI == EPI_RESID) hv += hres[s];
                    if (valid) {
                        if (EPI == EPI_RESID || EPI == EPI_STORE_F32) {
                            static_cast<float*>(a.e.out)[(size_t)j * a.e.ldo + n] = hv;
                            if (EPI == EPI_RESID && a.e.snap) static_cast<float*>(a.e.snap)[(size_t)j * a.e.snap_ld + n] = hv;
                            if (EPI == EPI_RESID && a.e.ln.gain) {
                                const float x = (hv - s_mu[s]) * next_gain;
                                const bf16 hi = __float2bfloat16_rn(x);
                                a.e.ln.hi[(size_t)j * a.e.ldo + n] = hi;
                                a.e.ln.lo[(size_t)j * a.e.ldo + n] = __float2bfloat16_rn(x - __bfloat162float(hi));
                            }
                        } else if (EPI == EPI_GELU) {   // activations between the decode kernels stay fp32, or value + remainder planes
                            const float gv = gelu_bf16_out(hv);
                            if (a.e.out_lo) {
                                const bf16 hi = __float2bfloat16_rn(gv);
                                static_cast<bf16*>(a.e.out)[(size_t)j * a.e.ldo + n] = hi;
                                static_cast<bf16*>(a.e.out_lo)[(size_t)j * a.e.ldo + n] = __float2bfloat16_rn(gv - __bfloat162float(hi));
                            } else {
                                static_cast<float*>(a.e.out)[(size_t)j * a.e.ldo + n] = gv;
                            }
                        } else if (EPI == EPI_QKV || EPI == EPI_KV) {
                            sc.base[(sc.is_q ? (long long)j * a.e.ldo : s_rowoff[j]) + sc.col] = __float2bfloat16_rn(hv);
                        } else {
                            epilogue<bf16, EPI>(a.e, j, n, hv);
                        }
                    }
                    if (EPI == EPI_RESID) v[s] = hv;   // (for the statistics below)
                }
            }
            if (EPI == EPI_RESID && a.e.ln.gain && n_group > 0) {   // (warp-uniform)
                // Mean and squared deviations of this warp's 32 features, four rows at a time in one transposing reduction (row by
                // row, with two five-step sums each, they cost 1.3 us of a 7.4 us launch with four rows per CTA).  Sums are
                // relative to the group's first feature.
                const float inv = 1.0f / (float)n_group;
                float2* stats = a.e.ln.stats + (size_t)j_first * a.e.ln.groups + ((seg_base + n_local0 + warp * 32) >> 5);
                if (j_count == 1) {   // one row (a step's, or a row of a block dealt to its own CTA): five shuffles instead of nine, the same tree
                    const float ref = __shfl_sync(0xffffffffu, v[0], 0), dv = valid ? v[0] - ref : 0.f;
                    float sums[2] = {dv, dv * dv};
                    const float mine = warp_sum_many<2>(sums, lane);                     // lanes 0-15: the sum, 16-31: the sum of squares
                    const float sd = mine, sq = __shfl_sync(0xffffffffu, mine, 16);
                    if (lane == 0) *stats = make_float2(fmaf(sd, inv, ref), fmaxf(fmaf(-sd * inv, sd, sq), 0.f));
                } else
#pragma unroll
                for (int s0 = 0; s0 < NB; s0 += 4) {
                    if (s0 >= j_count) break;
                    float sums[8], ref[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const float hv = s0 + u < j_count ? v[s0 + u] : 0.f;
                        ref[u] = __shfl_sync(0xffffffffu, hv, 0);
                        const float dv = valid ? hv - ref[u] : 0.f;
                        sums[2 * u] = dv;
                        sums[2 * u + 1] = dv * dv;
                    }
                    const float mine = warp_sum_many<8>(sums, lane);                     // lane L: sum number L / 4
                    const float sd = __shfl_sync(0xffffffffu, mine, lane & ~7), sq = __shfl_sync(0xffffffffu, mine, (lane & ~7) + 4);
                    const int u = lane >> 3;
                    if ((lane & 7) == 0 && s0 + u < j_count) {
                        const float rf = u == 0 ? ref[0] : (u == 1 ? ref[1] : (u == 2 ? ref[2] : ref[3]));
                        stats[(size_t)(s0 + u) * a.e.ln.groups] = make_float2(fmaf(sd, inv, rf), fmaxf(fmaf(-sd * inv, sd, sq), 0.f));
                    }
                }
            }
        }
    }
}

// ---------------------------------------------------------------------------------------------------
// Many rows: A = token rows, B = weight rows, both by TMA.
// ---------------------------------------------------------------------------------------------------

struct TcTiledArgs {
    int M, K, N;
    int seg_rows0, tiles0;   // first segment: output features, feature tiles
    int seg_rows, tiles_per_seg;
    int tiles_n, tiles_m;    // feature tiles over all segments, row tiles (of 256 in the pair kernel, else 128)
    int splits;              // gemm_tc_split_kernel: CTAs that share a tile's K range
    int whole, parts;        // gemm_tc_pair_kernel: tiles done whole; parts that each of the remaining ones is cut into (1, 2, 4)
    int lo_row;              // PL: row of the remainder plane's first row in the token rows' tensor map
    int* err_flag;
    float* tile_max; int* tile_idx; float* tile_sum;   // EPI_SCORE: [M][tile_stride]
    int tile_stride;
    const int* truth; float* truth_val;                // EPI_SCORE: [M] the feature whose value goes to truth_val
    const int* keep; float* kept;                      // EPI_SCORE: [M] the row of kept [][N] that takes all of the row's values (-1: none)
    EpiArgs e;
};

constexpr int TCT_TILE_BYTES = 128 * 128;          // 128 rows x 64 bf16
constexpr int TCP_THREADS = 320;   // warps 0-7: epilogue, two per 32 rows; warp 8: TMA; warp 9: TMEM + MMA issue
constexpr int TCP_BN = 256;                           // output features per tile
// PL: the token rows are two bf16 planes (values, remainders; fp32 rows to about 16 bits), both multiplied with the same weight tile into
// the same accumulator: a K-block brings 48 KB for twice the products.
template <bool PL> struct TcpCfg {
    static constexpr int STAGES = PL ? 4 : 6;
    static constexpr int W_AT = (PL ? 2 : 1) * TCT_TILE_BYTES;          // this CTA's token rows, then its half of the weight rows
    static constexpr int STAGE_BYTES = W_AT + TCT_TILE_BYTES;
    static constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + 1024;
};
constexpr int TCP_GROUP_M = 8;                        // row tiles that share a sweep over the weights, see tcp_item

// EPI_SCORE: SCORE_TILE features of one row from its TMEM lane; n0: the first of them, valid: how many exist.  Warp-wide loads.
__device__ __forceinline__ void score_tile(const TcTiledArgs& a, uint32_t acc, int m, int n0, int valid) {
    const bool mine = m < a.M && valid > 0;
    const int keep = mine ? a.keep[m] : -1;
    {
        float v[SCORE_TILE];
#pragma unroll
        for (int i = 0; i < SCORE_TILE; i += 16) {
            float t[16];
            tmem_ld16(acc + i, t);
#pragma unroll
            for (int u = 0; u < 16; ++u) v[i + u] = i + u < valid ? t[u] : -INFINITY;
        }
        if (mine) {
            float best = -INFINITY, z = 0.f, true_v = 0.f;
            int bi = -1;
            const int truth = a.truth[m] - n0;
#pragma unroll
            for (int i = 0; i < SCORE_TILE; ++i) {
                if (v[i] > best) { best = v[i]; bi = i; }
                if (i == truth) true_v = v[i];
            }
#pragma unroll
            for (int i = 0; i < SCORE_TILE; ++i) z += expf(v[i] - best);
            const size_t o = (size_t)m * a.tile_stride + n0 / SCORE_TILE;
            a.tile_max[o] = best;
            a.tile_idx[o] = bi < 0 ? INT_MAX : n0 + bi;
            a.tile_sum[o] = z;
            if (truth >= 0 && truth < valid && truth < SCORE_TILE) a.truth_val[m] = true_v;
        }
    }
    if (!__any_sync(0xffffffffu, keep >= 0)) return;   // (all but the sequences' last blocks)
#pragma unroll 1
    for (int i = 0; i < SCORE_TILE; i += 16) {
        float t[16];
        tmem_ld16(acc + i, t);
        if (keep < 0) continue;
        float* row = a.kept + (size_t)keep * a.N + n0 + i;
        if ((a.N & 3) == 0 && i + 16 <= valid) {
#pragma unroll
            for (int u = 0; u < 16; u += 4) *reinterpret_cast<float4*>(row + u) = make_float4(t[u], t[u + 1], t[u + 2], t[u + 3]);
        } else {
#pragma unroll
            for (int u = 0; u < 16; ++u) if (i + u < valid) row[u] = t[u];
        }
    }
}

// Sixteen consecutive output features of one row.  n_local0 is a multiple of 16.  PL with EPI_GELU: to two planes.
template <int EPI, bool PL>
__device__ __forceinline__ void epilogue16(const EpiArgs& e, int m, int seg, int seg_base, int seg_rows, int n_local0, size_t row_off, const float (&v)[16]) {
    const int n0 = seg_base + n_local0;
    if (n_local0 + 16 > seg_rows || (e.ldo & 7) || (seg_rows & 7)) {
        for (int i = 0; i < 16; ++i)
            if (n_local0 + i < seg_rows) {
                epilogue<bf16, EPI>(e, m, n0 + i, v[i]);
                if (EPI == EPI_GELU && PL) {
                    const float g = gelu_bf16_out(v[i]);
                    static_cast<bf16*>(e.out_lo)[(size_t)m * e.ldo + n0 + i] = __float2bfloat16_rn(g - __bfloat162float(__float2bfloat16_rn(g)));
                }
            }
        return;
    }
    if (EPI == EPI_STORE_F32 || EPI == EPI_RESID) {
        float4* p = reinterpret_cast<float4*>(static_cast<float*>(e.out) + (size_t)m * e.ldo + n0);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            float4 t = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
            if (EPI == EPI_RESID) { const float4 o = p[i]; t.x += o.x; t.y += o.y; t.z += o.z; t.w += o.w; }
            p[i] = t;
        }
        return;
    }
    uint4 lo, hi;
    if (EPI == EPI_GELU && PL) {
        uint4 rlo, rhi;
        split_bf16x2(gelu_bf16_out(v[0]), gelu_bf16_out(v[1]), lo.x, rlo.x); split_bf16x2(gelu_bf16_out(v[2]), gelu_bf16_out(v[3]), lo.y, rlo.y);
        split_bf16x2(gelu_bf16_out(v[4]), gelu_bf16_out(v[5]), lo.z, rlo.z); split_bf16x2(gelu_bf16_out(v[6]), gelu_bf16_out(v[7]), lo.w, rlo.w);
        split_bf16x2(gelu_bf16_out(v[8]), gelu_bf16_out(v[9]), hi.x, rhi.x); split_bf16x2(gelu_bf16_out(v[10]), gelu_bf16_out(v[11]), hi.y, rhi.y);
        split_bf16x2(gelu_bf16_out(v[12]), gelu_bf16_out(v[13]), hi.z, rhi.z); split_bf16x2(gelu_bf16_out(v[14]), gelu_bf16_out(v[15]), hi.w, rhi.w);
        uint4* r = reinterpret_cast<uint4*>(static_cast<bf16*>(e.out_lo) + (size_t)m * e.ldo + n0);
        r[0] = rlo;
        r[1] = rhi;
    } else if (EPI == EPI_GELU) {
        lo.x = pack_bf16x2(gelu_bf16_out(v[0]), gelu_bf16_out(v[1])); lo.y = pack_bf16x2(gelu_bf16_out(v[2]), gelu_bf16_out(v[3]));
        lo.z = pack_bf16x2(gelu_bf16_out(v[4]), gelu_bf16_out(v[5])); lo.w = pack_bf16x2(gelu_bf16_out(v[6]), gelu_bf16_out(v[7]));
        hi.x = pack_bf16x2(gelu_bf16_out(v[8]), gelu_bf16_out(v[9])); hi.y = pack_bf16x2(gelu_bf16_out(v[10]), gelu_bf16_out(v[11]));
        hi.z = pack_bf16x2(gelu_bf16_out(v[12]), gelu_bf16_out(v[13])); hi.w = pack_bf16x2(gelu_bf16_out(v[14]), gelu_bf16_out(v[15]));
    } else {
        lo.x = pack_bf16x2(v[0], v[1]); lo.y = pack_bf16x2(v[2], v[3]); lo.z = pack_bf16x2(v[4], v[5]); lo.w = pack_bf16x2(v[6], v[7]);
        hi.x = pack_bf16x2(v[8], v[9]); hi.y = pack_bf16x2(v[10], v[11]); hi.z = pack_bf16x2(v[12], v[13]); hi.w = pack_bf16x2(v[14], v[15]);
    }
    bf16* dst;
    if (EPI == EPI_STORE || EPI == EPI_GELU) {
        dst = static_cast<bf16*>(e.out) + (size_t)m * e.ldo + n0;
    } else {   // EPI_QKV / EPI_KV: the query goes to its buffer, keys and values straight into the cache
        int s = seg;
        if (EPI == EPI_QKV && s == 0) {
            dst = static_cast<bf16*>(e.out) + (size_t)m * e.ldo + n_local0;
        } else {
            if (EPI == EPI_QKV) s -= 1;
            const int h = n_local0 / e.d_head, el = n_local0 - h * e.d_head;
            dst = static_cast<bf16*>(s == 0 ? e.kcache : e.vcache) + row_off + (size_t)h * e.t_max * e.d_head + el;
        }
    }
    if ((reinterpret_cast<uintptr_t>(dst) & 31) == 0) {   // (rows of an odd multiple of eight elements alternate)
        st_global_u32x8(dst, lo, hi);
    } else {
        reinterpret_cast<uint4*>(dst)[0] = lo;
        reinterpret_cast<uint4*>(dst)[1] = hi;
    }
}

// The row's part of an index into the caches, EPI_QKV / EPI_KV: two dependent loads, made before the accumulator is awaited.
template <int EPI>
__device__ __forceinline__ size_t cache_row_offset(const EpiArgs& e, int m, int M) {
    if ((EPI != EPI_QKV && EPI != EPI_KV) || m >= M) return 0;
    if (!e.row_seq) return (size_t)m * e.d_head;
    return ((size_t)e.row_seq[m] * e.n_heads * e.t_max + e.row_pos[m]) * e.d_head;
}

// Feature tile -> (segment, first feature within it).
__device__ __forceinline__ int tct_segment(const TcTiledArgs& a, int tile_n, int width, int& n_local0) {
    const int seg = tile_n < a.tiles0 ? 0 : 1 + (tile_n - a.tiles0) / a.tiles_per_seg;
    n_local0 = (seg == 0 ? tile_n : tile_n - a.tiles0 - (seg - 1) * a.tiles_per_seg) * width;
    return seg;
}
// Work item -> (row tile, feature tile, first feature within the tile, width).  Row tiles go in groups of TCP_GROUP_M, inside
// a group row tiles fastest: the pairs that run at the same time share eight row tiles and about nine feature tiles, so
// the weights pass through L2 once per group of row tiles.  (With feature tiles fastest over all of them, few row tiles met
// the whole matrix at a time: 12288 x 4096 weights are 100 MB, about the size of L2.)  Tiles that do not fill a last
// round of all pairs are cut into two or four parts along the features, so that round costs a half or a quarter (12280 x
// 2048: 384 tiles on 74 pairs are 5.2 rounds, 6 without).
__device__ __forceinline__ void tcp_item(const TcTiledArgs& a, int item, int& tile_m, int& tile_n, int& c0, int& width) {
    int t = item;
    c0 = 0;
    width = TCP_BN;
    if (item >= a.whole) {
        const int u = item - a.whole;
        t = a.whole + u / a.parts;
        width = TCP_BN / a.parts;
        c0 = (u - (t - a.whole) * a.parts) * width;
    }
    const int per_group = TCP_GROUP_M * a.tiles_n;
    const int g = t / per_group, r = t - g * per_group;
    const int gm = min(TCP_GROUP_M, a.tiles_m - g * TCP_GROUP_M);
    tile_n = r / gm;
    tile_m = g * TCP_GROUP_M + r - tile_n * gm;
}

// CW columns of an output row (= TMEM lane), TMEM -> registers -> global; acc: the first of them in this warp's lanes; n_local0:
// its feature within the segment.  A thread moves whole 32-byte sectors of its row (with 16-byte accesses the residual
// add fetched every sector of the stream twice).  The residual add has its first 64 old values in flight before the accumulator
// is awaited, which `wait` does.
template <int EPI, bool PL, typename Wait>
__device__ __forceinline__ void tcp_epilogue(const TcTiledArgs& a, uint32_t acc, int m, int seg, int seg_base, int seg_rows, int n_local0, int CW, Wait wait) {
    if (EPI == EPI_RESID && n_local0 + CW <= seg_rows && (a.e.ldo & 7) == 0 && (seg_base & 7) == 0) {
        float* prow = static_cast<float*>(a.e.out) + (size_t)min(m, a.M - 1) * a.e.ldo + seg_base + n_local0;
        f32x8 cur[4], nxt[4];
        auto load = [&](f32x8 (&o)[4], int c) {
#pragma unroll
            for (int j = 0; j < 4; ++j) o[j] = ld_global_f32x8(prow + c + 8 * j);
        };
        load(cur, 0);
        if (CW > 32) load(nxt, 32);
        if (!wait()) return;
#pragma unroll 2
        for (int c = 0; c < CW; c += 32) {
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                float v[16];
                tmem_ld16(acc + c + 16 * q, v);   // warp-wide: every lane takes part
#pragma unroll
                for (int i = 0; i < 8; ++i) { cur[2 * q].v[i] += v[i]; cur[2 * q + 1].v[i] += v[8 + i]; }
                if (m < a.M) {
                    st_global_f32x8(prow + c + 16 * q, cur[2 * q]);
                    st_global_f32x8(prow + c + 16 * q + 8, cur[2 * q + 1]);
                }
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) cur[j] = nxt[j];
            if (c + 64 < CW) load(nxt, c + 64);
        }
        return;
    }
    const size_t row_off = cache_row_offset<EPI>(a.e, m, a.M);
    if (!wait()) return;
    if constexpr (EPI == EPI_SCORE) {   // (one segment, whole tiles)
#pragma unroll 1
        for (int c = 0; c < CW; c += SCORE_TILE) score_tile(a, acc + c, m, n_local0 + c, seg_rows - (n_local0 + c));
        return;
    }
#pragma unroll 1
    for (int c = 0; c < CW; c += 16) {
        float v[16];
        tmem_ld16(acc + c, v);   // warp-wide: every lane takes part
        if (m < a.M && n_local0 + c < seg_rows) epilogue16<EPI, PL>(a.e, m, seg, seg_base, seg_rows, n_local0 + c, row_off, v);
    }
}

// Persistent, on pairs of multiprocessors: a cluster of two CTAs computes a 256 x 256 tile with MMAs that span both (each CTA
// brings its 128 token rows and one half of the 256 weight rows, and keeps its 128 rows of the accumulator), so a
// multiprocessor reads a third less from L2 and shared memory per product than with a 128 x 256 tile of its own, and the ring
// holds six K-blocks instead of four.  The first CTA's warp 9 issues the MMAs; both CTAs' loads count on its barriers; the
// commits arrive on both CTAs' barriers.  The ring runs on across tile boundaries, and two accumulators in TMEM alternate.
// Seconds-long loops under the power cap, against 128 x 256 tiles with four epilogue warps: 8191 x 12288 x 4096 656 -> 594 us
// (1387 TFLOP/s), 8191 x 11008 x 4096 with GELU 585 -> 555 us, 8191 x 4096 x 11008 with the residual add 628 -> 579 us,
// 12280 x 2048 x 2048 with the residual add 156 -> 108 us.
// tmh*: the weights in boxes of 32 rows, for the parts of tiles.
// grid: 2 * min(items, SMs / 2) in clusters of two; dynamic smem TcpCfg::SMEM_BYTES.
template <int EPI, bool PL>
__global__ void __launch_bounds__(TCP_THREADS)
gemm_tc_pair_kernel(const TcTiledArgs a, const __grid_constant__ CUtensorMap tmx, const __grid_constant__ CUtensorMap tm0,
                    const __grid_constant__ CUtensorMap tm1, const __grid_constant__ CUtensorMap tm2,
                    const __grid_constant__ CUtensorMap tmh0, const __grid_constant__ CUtensorMap tmh1, const __grid_constant__ CUtensorMap tmh2) {
    using C = TcpCfg<PL>;
    constexpr int BN = TCP_BN;
    extern __shared__ __align__(1024) unsigned char smem_dyn[];
    __shared__ __align__(8) uint64_t s_full[C::STAGES];    // first CTA: both CTAs' loads of a stage
    __shared__ __align__(8) uint64_t s_empty[C::STAGES];
    __shared__ __align__(8) uint64_t s_acc_full[2], s_acc_free[2];
    __shared__ uint32_t s_tmem;

    const int tid = threadIdx.x, warp = warp_uniform(tid >> 5), lane = tid & 31;
    const int rank = blockIdx.x & 1, pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;
    const uint32_t ring0 = (smem_u32(smem_dyn) + 1023u) & ~1023u;
    const int KB = (a.K + 63) >> 6;
    const int total = a.whole + (a.tiles_n * a.tiles_m - a.whole) * a.parts;

    if (warp == 9) {
        if (lane == 0) {
            for (int s = 0; s < C::STAGES; ++s) { mbar_init(smem_u32(&s_full[s]), 1); mbar_init(smem_u32(&s_empty[s]), 1); }
            for (int s = 0; s < 2; ++s) { mbar_init(smem_u32(&s_acc_full[s]), 1); mbar_init(smem_u32(&s_acc_free[s]), 16); }   // free: one arrive per epilogue warp of the pair
            mbar_init_fence();
        }
        __syncwarp();
        tmem_alloc_pair(smem_u32(&s_tmem), 2 * BN);
        tmem_relinquish_pair();
    }
    tc_fence_before_sync();
    cluster_sync_all();          // both CTAs' barriers are initialised
    tc_fence_after_sync();
    const uint32_t tmem = warp_uniform(s_tmem);

    if (warp == 8) {
        if (elect_one()) { tma_prefetch_desc(&tmx); tma_prefetch_desc(&tm0); }
        pdl_wait();              // the token rows come from the kernel before this one
        int st = 0, round = 0;   // ring position, and how often the ring has gone round
        bool ok = true;
        for (int t = pair; t < total && ok; t += n_pairs) {
            int tile_m, tile_n, c0, width, n_local0;
            tcp_item(a, t, tile_m, tile_n, c0, width);
            const int seg = tct_segment(a, tile_n, BN, n_local0);
            const int m0 = tile_m * 256 + rank * 128, n0 = n_local0 + c0 + rank * (width / 2);
            const CUtensorMap* tw = seg == 0 ? &tm0 : (seg == 1 ? &tm1 : &tm2);
            const CUtensorMap* th = seg == 0 ? &tmh0 : (seg == 1 ? &tmh1 : &tmh2);
            for (int i = 0; i < KB; ++i) {
                if (round > 0 && !mbar_wait_warp(smem_u32(&s_empty[st]), (uint32_t)(round - 1) & 1)) {
                    tc_report(a.err_flag, TC_ERR_SLOT);
                    ok = false;
                    break;
                }
                if (elect_one()) {
                    const uint32_t bar = cluster_map(smem_u32(&s_full[st]), 0), dst = ring0 + st * C::STAGE_BYTES;
                    if (rank == 0) mbar_arrive_expect_tx(smem_u32(&s_full[st]), 2 * C::W_AT + width * 128);
                    tma_load_2d_pair(dst, &tmx, i * 64, m0, bar);                     // rows past the end arrive as zeros (PL: or as another plane's, and are not used)
                    if (PL) tma_load_2d_pair(dst + TCT_TILE_BYTES, &tmx, i * 64, a.lo_row + m0, bar);
                    if (width == BN) tma_load_2d_pair(dst + C::W_AT, tw, i * 64, n0, bar);
                    else
                        for (int q = 0; q < width / 2; q += 32) tma_load_2d_pair(dst + C::W_AT + q * 128, th, i * 64, n0 + q, bar);
                }
                if (++st == C::STAGES) { st = 0; ++round; }
            }
        }
        pdl_launch_dependents();
        __syncwarp();
    } else if (warp == 9) {
        if (rank == 0) {
            int st = 0, round = 0;
            bool ok = true;
            int it = 0;
            for (int t = pair; t < total && ok; t += n_pairs, ++it) {
                const int buf = it & 1;
                const uint32_t idesc = t < a.whole ? umma_idesc_bf16(256, BN) : umma_idesc_bf16(256, BN / a.parts);
                // the accumulator's previous tile (two tiles back) must have been read out by both CTAs
                if (it >= 2 && !mbar_wait_warp(smem_u32(&s_acc_free[buf]), (uint32_t)((it >> 1) - 1) & 1)) {
                    tc_report(a.err_flag, TC_ERR_ACCUM);
                    break;
                }
                tc_fence_after_sync();
                for (int i = 0; i < KB; ++i) {
                    if (!mbar_wait_warp(smem_u32(&s_full[st]), (uint32_t)round & 1)) {
                        tc_report(a.err_flag, TC_ERR_OPERANDS);
                        ok = false;
                        break;
                    }
                    tc_fence_after_sync();
                    if (elect_one()) {
                        const uint64_t da = umma_desc_k_sw128(ring0 + st * C::STAGE_BYTES);
                        const uint64_t db = umma_desc_k_sw128(ring0 + st * C::STAGE_BYTES + C::W_AT);
#pragma unroll
                        for (int k = 0; k < 4; ++k) umma_bf16_pair(tmem + buf * BN, da + 2 * k, db + 2 * k, idesc, (i | k) != 0 ? 1u : 0u);
                        if (PL) {
#pragma unroll
                            for (int k = 0; k < 4; ++k) umma_bf16_pair(tmem + buf * BN, da + TCT_TILE_BYTES / 16 + 2 * k, db + 2 * k, idesc, 1u);
                        }
                        umma_commit_pair(smem_u32(&s_empty[st]));
                    }
                    if (++st == C::STAGES) { st = 0; ++round; }
                }
                if (elect_one()) umma_commit_pair(smem_u32(&s_acc_full[buf]));   // (also after a failed wait: the epilogue warps must not be left waiting)
            }
        }
        __syncwarp();
    } else {
        pdl_wait();
        int it = 0;
        for (int t = pair; t < total; t += n_pairs, ++it) {
            const int buf = it & 1;
            int tile_m, tile_n, c0, width, n_local0;
            tcp_item(a, t, tile_m, tile_n, c0, width);
            const int seg = tct_segment(a, tile_n, BN, n_local0);
            const int col = (warp >> 2) * (width / 2);                    // this warp's half of the columns
            const int seg_rows = seg == 0 ? a.seg_rows0 : a.seg_rows;
            const int seg_base = seg == 0 ? 0 : a.seg_rows0 + (seg - 1) * a.seg_rows;
            bool ok = true;
            auto wait = [&]() {
                ok = mbar_wait(smem_u32(&s_acc_full[buf]), (uint32_t)(it >> 1) & 1);
                if (!ok) tc_report(a.err_flag, TC_ERR_ACCUM);
                tc_fence_after_sync();
                return ok;
            };
            const int m = tile_m * 256 + rank * 128 + (warp & 3) * 32 + lane;   // output row = TMEM lane
            const uint32_t acc = tmem + (static_cast<uint32_t>((warp & 3) * 32) << 16) + buf * BN + col;
            tcp_epilogue<EPI, PL>(a, acc, m, seg, seg_base, seg_rows, n_local0 + c0 + col, width / 2, wait);
            if (!ok) break;
            tc_fence_before_sync();   // this warp's TMEM reads are done: the accumulator may be overwritten
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(cluster_map(smem_u32(&s_acc_free[buf]), 0));
        }
    }
    tc_fence_before_sync();
    cluster_sync_all();           // nobody leaves while the other CTA's operands or accumulators are in use
    tc_fence_after_sync();
    if (warp == 9) tmem_dealloc_pair(tmem, 2 * BN);
}

// Prompt passes of few tiles (the small pair's 511 rows: 32 tiles of 128 x 128 for N = 1024): a tile's time is its
// operands' way from L2 into one multiprocessor (32 KB per 64 of K; the tensor pipe is 7-26 % busy under ncu), so the
// tile's K range is dealt to the S = 1, 2 or 4 CTAs of a cluster.  Each sends its partial sums of the columns that another
// one finishes into that CTA's inbox (16-byte stores that count their bytes on the receiver's barrier, a lane per row, 512
// contiguous bytes per warp and store), and CTA r finishes columns r * 128 / S ..: sums in slice order, then the
// epilogue, which is S times shorter per CTA.  Eight epilogue warps, two per 32 rows.  The inbox lies where the ring was: a
// cluster barrier after the last product says that every ring is free.  That keeps a CTA at 97 KB, so that the next kernel's
// CTAs sit beside it with their first weights loaded (with an inbox of its own a CTA of four took 176 KB, and every kernel
// began with a cold start after the one before).  One tile per cluster.
// grid: tiles * S; dynamic smem TcsCfg::SMEM_BYTES.
constexpr int TCS_THREADS = 320;   // warps 0-7: epilogue; warp 8: TMA; warp 9: TMEM + MMA issue
constexpr int TCS_BN = 128;
template <bool PL> struct TcsCfg {
    static constexpr int STAGES = PL ? 2 : 3;
    static constexpr int W_AT = (PL ? 2 : 1) * TCT_TILE_BYTES;
    static constexpr int STAGE_BYTES = W_AT + TCT_TILE_BYTES;
    static constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + 1024;
    static_assert(2 * (SMEM_BYTES + 1024 + 1024) <= 227 * 1024, "two CTAs per SM");
    static_assert(3 * (128 * TCS_BN * 4 / 4) <= STAGES * STAGE_BYTES && 128 * TCS_BN * 4 / 2 <= STAGES * STAGE_BYTES, "the inbox fits where the ring was");
};

template <int EPI, bool PL>
__global__ void __launch_bounds__(TCS_THREADS)
gemm_tc_split_kernel(const TcTiledArgs a, const __grid_constant__ CUtensorMap tmx, const __grid_constant__ CUtensorMap tm0,
                     const __grid_constant__ CUtensorMap tm1, const __grid_constant__ CUtensorMap tm2) {
    using C = TcsCfg<PL>;
    extern __shared__ __align__(1024) unsigned char smem_dyn[];
    __shared__ __align__(8) uint64_t s_full[C::STAGES];
    __shared__ __align__(8) uint64_t s_empty[C::STAGES];
    __shared__ __align__(8) uint64_t s_accum, s_inbox;
    __shared__ uint32_t s_tmem;

    const int tid = threadIdx.x, warp = warp_uniform(tid >> 5), lane = tid & 31;
    const uint32_t ring0 = (smem_u32(smem_dyn) + 1023u) & ~1023u;
    const int S = a.splits;
    constexpr int stages = C::STAGES;
    const int tile = blockIdx.x / S, sp = blockIdx.x - tile * S;           // sp = this CTA's rank in its cluster
    int n_local0;
    const int seg = tct_segment(a, tile % a.tiles_n, TCS_BN, n_local0);
    const int m0 = (tile / a.tiles_n) * 128;
    const int seg_rows = seg == 0 ? a.seg_rows0 : a.seg_rows;
    const int seg_base = seg == 0 ? 0 : a.seg_rows0 + (seg - 1) * a.seg_rows;
    const int KB = (a.K + 63) >> 6;
    const int kb0 = KB * sp / S, nkb = KB * (sp + 1) / S - kb0;

    if (warp == 9) {
        if (lane == 0) {
            for (int s = 0; s < C::STAGES; ++s) { mbar_init(smem_u32(&s_full[s]), 1); mbar_init(smem_u32(&s_empty[s]), 1); }
            mbar_init(smem_u32(&s_accum), 1);
            mbar_init(smem_u32(&s_inbox), 1);
            mbar_init_fence();
        }
        __syncwarp();
        tmem_alloc(smem_u32(&s_tmem), TCS_BN);
        tmem_relinquish();
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = warp_uniform(s_tmem);
    if (warp == 8) {
        const CUtensorMap* tw = seg == 0 ? &tm0 : (seg == 1 ? &tm1 : &tm2);
        const int n_pre = min(nkb, stages);
        if (elect_one()) {   // weights are parameters: the first ring-ful of them before the wait on the predecessor
            tma_prefetch_desc(&tmx);
            tma_prefetch_desc(tw);
            for (int i = 0; i < n_pre; ++i) {
                const uint32_t bar = smem_u32(&s_full[i]);
                mbar_arrive_expect_tx(bar, C::STAGE_BYTES);
                tma_load_2d_nohint(ring0 + i * C::STAGE_BYTES + C::W_AT, tw, (kb0 + i) * 64, n_local0, bar);
            }
        }
        pdl_wait();
        if (elect_one())
            for (int i = 0; i < n_pre; ++i) {
                tma_load_2d_nohint(ring0 + i * C::STAGE_BYTES, &tmx, (kb0 + i) * 64, m0, smem_u32(&s_full[i]));
                if (PL) tma_load_2d_nohint(ring0 + i * C::STAGE_BYTES + TCT_TILE_BYTES, &tmx, (kb0 + i) * 64, a.lo_row + m0, smem_u32(&s_full[i]));
            }
        int st = 0, round = 0;
        for (int i = n_pre; i < nkb; ++i) {
            if (!mbar_wait_warp(smem_u32(&s_empty[st]), (uint32_t)round & 1)) { tc_report(a.err_flag, TC_ERR_SLOT); break; }
            if (elect_one()) {
                const uint32_t bar = smem_u32(&s_full[st]), dst = ring0 + st * C::STAGE_BYTES;
                mbar_arrive_expect_tx(bar, C::STAGE_BYTES);
                tma_load_2d_nohint(dst, &tmx, (kb0 + i) * 64, m0, bar);
                if (PL) tma_load_2d_nohint(dst + TCT_TILE_BYTES, &tmx, (kb0 + i) * 64, a.lo_row + m0, bar);
                tma_load_2d_nohint(dst + C::W_AT, tw, (kb0 + i) * 64, n_local0, bar);
            }
            if (++st == stages) { st = 0; ++round; }
        }
        pdl_launch_dependents();
        __syncwarp();
        if (S > 1) cluster_sync_all();
    } else if (warp == 9) {
        constexpr uint32_t idesc = umma_idesc_bf16(128, TCS_BN);
        uint32_t phase = 0, ok = mbar_test(smem_u32(&s_full[0]), 0);
        for (int i = 0, st = 0; i < nkb; ++i) {
            if (!mbar_wait_tested(ok, smem_u32(&s_full[st]), phase)) { tc_report(a.err_flag, TC_ERR_OPERANDS); break; }
            tc_fence_after_sync();
            const int done = st;
            if (++st == stages) { st = 0; phase ^= 1; }
            if (i + 1 < nkb) ok = mbar_test(smem_u32(&s_full[st]), phase);
            const uint64_t dx = umma_desc_k_sw128(ring0 + done * C::STAGE_BYTES), dw = umma_desc_k_sw128(ring0 + done * C::STAGE_BYTES + C::W_AT);
            umma_bf16_k64(tmem, dx, dw, idesc, i != 0 ? 1u : 0u);
            if (PL) umma_bf16_k64(tmem, dx + TCT_TILE_BYTES / 16, dw, idesc, 1u);
            umma_commit_one(smem_u32(&s_empty[done]));
        }
        umma_commit_one(smem_u32(&s_accum));
        if (S > 1) cluster_sync_all();
    } else {
        pdl_wait();
        const int quarter = warp & 3, half = warp >> 2;
        const int row = quarter * 32 + lane, m = m0 + row;   // output row = TMEM lane
        const uint32_t acc = tmem + (static_cast<uint32_t>(quarter * 32) << 16);
        const int CS = TCS_BN / S;                           // columns that a CTA finishes
        const uint32_t inbox0 = ring0;                       // [S - 1 senders][CS / 4][128 rows] of four floats
        const uint32_t ibar = smem_u32(&s_inbox);
        // What the epilogue reads is in flight before the accumulator is awaited: the row's place in the caches, and the old values
        // of the residual add, 16 columns ahead from there on (small pair's prompt of 511 rows: 787 -> 772 us).
        const size_t row_off = cache_row_offset<EPI>(a.e, m, a.M);
        const int c_first = half * (CS / 2), c_end = c_first + CS / 2;
        float4 old[EPI == EPI_RESID ? 4 : 1];
        auto old_at = [&](int c0) {   // null where the columns are not added 16 at a time
            const int n_local = n_local0 + sp * CS + c0;
            const bool whole = c0 < c_end && m < a.M && n_local + 16 <= seg_rows && !(a.e.ldo & 7) && !(seg_rows & 7);
            return whole ? reinterpret_cast<float4*>(static_cast<float*>(a.e.out) + (size_t)m * a.e.ldo + seg_base + n_local) : nullptr;
        };
        if (EPI == EPI_RESID)
            if (const float4* p = old_at(c_first)) {
#pragma unroll
                for (int i = 0; i < 4; ++i) old[i] = p[i];
            }
        if (!mbar_wait(smem_u32(&s_accum), 0)) tc_report(a.err_flag, TC_ERR_ACCUM);
        tc_fence_after_sync();
        if (S > 1) {
            // This CTA's products have read its ring, and so have the others'.  With release: the reads, known to be done by
            // the wait above, come before the peers' stores to the same bytes.
            cluster_sync_all();
            if (tid == 0) mbar_arrive_expect_tx(ibar, (uint32_t)((S - 1) * 128 * CS * 4));
            for (int q = 0; q < S; ++q) {
                if (q == sp) continue;
                const uint32_t slot = inbox0 + (uint32_t)(sp < q ? sp : sp - 1) * (128 * CS * 4);   // the receiver leaves itself out
#pragma unroll 1
                for (int c0 = half * (CS / 2); c0 < (half + 1) * (CS / 2); c0 += 16) {
                    float v[16];
                    tmem_ld16(acc + q * CS + c0, v);
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        st_async_dsmem_f32x4(slot + (uint32_t)(((c0 >> 2) + i) * 128 + row) * 16, ibar, q, v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
                }
            }
            if (!mbar_wait(ibar, 0)) tc_report(a.err_flag, TC_ERR_EXCHANGE);
        }
        const float4* inbox = reinterpret_cast<const float4*>(smem_dyn + (inbox0 - smem_u32(smem_dyn)));
        if constexpr (EPI == EPI_SCORE) {   // (one segment, S == 1)
            score_tile(a, acc + c_first, m, n_local0 + c_first, seg_rows - (n_local0 + c_first));
        } else
#pragma unroll 1
        for (int c0 = c_first; c0 < c_end; c0 += 16) {
            float v[16];
            tmem_ld16(acc + sp * CS + c0, v);   // warp-wide: every lane takes part
            if (S > 1) {
                float t[16];
#pragma unroll
                for (int i = 0; i < 16; ++i) t[i] = 0.f;
                for (int q = 0; q < S; ++q) {   // slice order
                    const float4* from = inbox + (size_t)(q < sp ? q : q - 1) * (128 * CS / 4) + (c0 >> 2) * 128 + row;
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const float4 p = q == sp ? make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]) : from[i * 128];
                        t[4 * i] += p.x; t[4 * i + 1] += p.y; t[4 * i + 2] += p.z; t[4 * i + 3] += p.w;
                    }
                }
#pragma unroll
                for (int i = 0; i < 16; ++i) v[i] = t[i];
            }
            const int n_local = n_local0 + sp * CS + c0;
            if (EPI == EPI_RESID) {
                if (float4* p = old_at(c0)) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) old[i] = make_float4(old[i].x + v[4 * i], old[i].y + v[4 * i + 1], old[i].z + v[4 * i + 2], old[i].w + v[4 * i + 3]);
                    const float4* q = old_at(c0 + 16);
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        p[i] = old[i];
                        if (q) old[i] = q[i];
                    }
                    continue;
                }
            }
            if (m < a.M && n_local < seg_rows) epilogue16<EPI, PL>(a.e, m, seg, seg_base, seg_rows, n_local, row_off, v);
        }
        tc_fence_before_sync();
    }
    __syncthreads();
    if (warp == 9) { tc_fence_after_sync(); tmem_dealloc(tmem, TCS_BN); }
}

}  // namespace tandem
