// Row set-up, embedding, LayerNorm, casts, arg-max, and the verify / accept / rollback kernel.
#pragma once
#include <math.h>
#include <limits.h>
#include "common.cuh"
#include "tc_common.cuh"

namespace tandem {

// Device-resident loop state (all int32 arrays live in the caller's arena).
struct LoopState {
    int* n;            // [B] committed tokens per sequence (prompt included); position n-1 is pending
    int* pending;      // [B] the pending token c[n-1]
    int* drafts;       // [B][gamma_limit]   d_1..d_gamma of the current iteration
    int* targets;      // [B][gamma_limit+1] the large model's arg-max per block row
    int* accept_len;   // [B]
    int* emitted;      // [B] tokens written to out_ids since the generate call began
    int* done;         // [B]
    int* out_ids;      // [B][out_cap]
    int* counters;     // [0] iteration index since prefill (advances while sequences are live), [1] live sequences,
                       // [2] error flags, [3] max_b n_b, [4] sum_b n_b, [5] live iterations of the current call,
                       // [6] verify kernels executed since the context was created (the host's ticket),
                       // [7] sequences still drafting (adaptive block length), [8] router launches since the context was created,
                       // [9] CTAs of the running router launch that have finished
    volatile int* host_flags;   // mapped pinned host memory: [0] ticket, [1] live, [2] n_max, [3] n_sum, [4] iterations,
                                // [5] router ticket, [6] sequences still drafting, [7] most tokens any live sequence still wants
    int* block_len;    // [B] adaptive block length: drafts made in the current iteration
    int* drafting;     // [B] adaptive block length: 1 while the router lets the sequence go on drafting
    float* confidence; // [B][gamma_limit] the router's 1 - s for every draft of the current iteration
    unsigned long long* hist;   // [gamma_limit+1] accept-length histogram of live sequences
    int out_cap;
    int gamma_limit;
};

// x^(0) = Emb(t) + Pos(index) of one row (Eq. 1) into the fp32 residual stream, 16 bytes of the tables at a time, with what
// the first LayerNorm's GEMM wants of it (LN, bf16; `row` is its row there; red: one float per warp).  d is a multiple of 8.
// All threads of a block of BLOCK take part.
template <typename T, int BLOCK, bool LN>
__device__ __forceinline__ void embed_row(const T* __restrict__ er, const T* __restrict__ pr, float* __restrict__ hr, float* __restrict__ snap, int d,
                                          const NextLn& ln, int row, float* red) {
    constexpr int VN = VecN<T>::N;
    const bool once = d <= BLOCK * VN;   // the row stays in registers
    float v[VN], gain[LN ? VN : 1], sum = 0.f;
    auto fetch = [&](int i) {
        float p[VN];
        load_vec(er + i, v);
        load_vec(pr + i, p);
#pragma unroll
        for (int u = 0; u < VN; ++u) v[u] += p[u];
    };
    auto fetch_gain = [&](int i) {
        if constexpr (LN) {
#pragma unroll
            for (int u = 0; u < VN; u += 4) {
                const float4 g = __ldg(reinterpret_cast<const float4*>(ln.gain + i + u));
                gain[u] = g.x; gain[u + 1] = g.y; gain[u + 2] = g.z; gain[u + 3] = g.w;
            }
        }
    };
    for (int i0 = 0; i0 < d; i0 += BLOCK * VN) {
        const int i = i0 + threadIdx.x * VN;
#pragma unroll
        for (int u = 0; u < VN; ++u) v[u] = 0.f;
        if (i < d) {
            fetch(i);
            if (once) fetch_gain(i);
#pragma unroll
            for (int u = 0; u < VN; u += 4) {
                const float4 t = make_float4(v[u], v[u + 1], v[u + 2], v[u + 3]);
                *reinterpret_cast<float4*>(hr + i + u) = t;
                if (snap) *reinterpret_cast<float4*>(snap + i + u) = t;
            }
        }
        if constexpr (LN) {   // four neighbouring threads hold a group of 32 features
            const float n = (float)min(32, d - (i & ~31));
            float s = 0.f, q = 0.f;
#pragma unroll
            for (int u = 0; u < VN; ++u) s += v[u];
            sum += s;
            s += __shfl_xor_sync(0xffffffffu, s, 1);
            s += __shfl_xor_sync(0xffffffffu, s, 2);
            const float mean = s / n;
            if (i < d) {
#pragma unroll
                for (int u = 0; u < VN; ++u) { const float c = v[u] - mean; q = fmaf(c, c, q); }
            }
            q += __shfl_xor_sync(0xffffffffu, q, 1);
            q += __shfl_xor_sync(0xffffffffu, q, 2);
            if (i < d && (threadIdx.x & 3) == 0) ln.stats[(size_t)row * ln.groups + (i >> 5)] = make_float2(mean, q);
        }
    }
    if constexpr (LN) {
        sum = warp_sum(sum);
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = sum;
        __syncthreads();
        float c = 0.f;
#pragma unroll
        for (int w = 0; w < BLOCK / 32; ++w) c += red[w];
        c /= (float)d;
        if (threadIdx.x == 0) ln.ref[row] = c;
        for (int i = threadIdx.x * VN; i < d; i += BLOCK * VN) {
            if (!once) { fetch(i); fetch_gain(i); }
            uint4 hi, lo;
            uint32_t *ph = &hi.x, *pl = &lo.x;
#pragma unroll
            for (int u = 0; u < VN; u += 2) {
                const float x0 = (v[u] - c) * gain[u], x1 = (v[u + 1] - c) * gain[u + 1];
                const __nv_bfloat162 a = __floats2bfloat162_rn(x0, x1);
                const __nv_bfloat162 r = __floats2bfloat162_rn(x0 - __low2float(a), x1 - __high2float(a));
                ph[u / 2] = *reinterpret_cast<const uint32_t*>(&a);
                pl[u / 2] = *reinterpret_cast<const uint32_t*>(&r);
            }
            *reinterpret_cast<uint4*>(ln.hi + (size_t)row * d + i) = hi;
            *reinterpret_cast<uint4*>(ln.lo + (size_t)row * d + i) = lo;
        }
    }
}

// One LayerNorm's parameters and where its four rows go that ride along in the GEMM behind it: gain, the gain's bf16
// remainder, bias, its remainder ([4][d]).
struct LnSource { const float* g; const float* b; bf16* rows; int d; };

// Start of a generate or step call: the first block says that nobody has emitted anything (a generate call also clears the
// histogram); the others write the LayerNorms' rows from the parameters as they are now (bf16: the decode GEMMs multiply by the live gain too,
// so parameters that the caller changed since the prompt pass hold for the whole call).  Not launched behind a running
// kernel: the GEMMs that read the rows ahead of their wait start two launches later.
// grid: 1 + LayerNorms; block: 256 (batch <= 256).
__global__ void __launch_bounds__(256) call_begin_kernel(LoopState st, int batch, bool clear_hist, const LnSource* __restrict__ lns) {
    if (blockIdx.x > 0) {
        const LnSource l = lns[blockIdx.x - 1];
        for (int i = threadIdx.x; i < l.d; i += 256) {
            const float g = l.g[i], b = l.b[i];
            const bf16 gh = __float2bfloat16_rn(g), bh = __float2bfloat16_rn(b);
            l.rows[i] = gh;
            l.rows[l.d + i] = __float2bfloat16_rn(g - __bfloat162float(gh));
            l.rows[2 * l.d + i] = bh;
            l.rows[3 * l.d + i] = __float2bfloat16_rn(b - __bfloat162float(bh));
        }
        return;
    }
    const int b = threadIdx.x;
    if (b < batch) { st.emitted[b] = 0; st.done[b] = 0; }
    if (clear_hist && b <= st.gamma_limit) st.hist[b] = 0ull;
    if (b == 0) { st.counters[1] = batch; st.counters[5] = 0; }
}

// What a prompt pass needs on the device, staged in one copy: per query its length and its offsets among the token ids,
// the processed rows and the attention groups ([4][n_queries]), then the ids, query after query.
struct PromptStage {
    const int* len; const int* id_off; const int* row_off; const int* grp_off; const int* ids;
    int n_queries, samples, rows, group;   // sequences per query; processed rows; queries per attention group
};

// Start of a prompt pass: block m < rows sets up processed row m (token, sequence, position, its attention group if it
// starts one) and embeds it; the last block sets the loop state of every sequence.  The tickets are the host's counts of
// the verify and router kernels it has enqueued, which the device's counts equal by then.
// grid: rows + 1; block: 128.
template <typename T>
__global__ void __launch_bounds__(128) prompt_begin_kernel(LoopState st, PromptStage ps, int* row_tok, int* row_seq, int* row_pos, int* grp_row0, int* grp_cnt,
                                                           const T* __restrict__ emb, const T* __restrict__ pos, float* __restrict__ h, int d,
                                                           int ticket, int router_ticket) {
    const int m = blockIdx.x;
    if (m == ps.rows) {
        for (int b = threadIdx.x; b < ps.n_queries * ps.samples; b += 128) {
            const int q = b / ps.samples, len = ps.len[q];
            st.n[b] = len;
            st.pending[b] = ps.ids[ps.id_off[q] + len - 1];
        }
        if (threadIdx.x == 0) { st.counters[6] = ticket; st.counters[8] = router_ticket; }
        return;
    }
    int lo = 0, hi = ps.n_queries - 1;   // the last query whose rows begin at or before m (queries without rows share a start: the last one has it)
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (ps.row_off[mid] <= m) lo = mid; else hi = mid - 1;
    }
    const int p = m - ps.row_off[lo], tok = ps.ids[ps.id_off[lo] + p];
    if (threadIdx.x == 0) {
        row_tok[m] = tok; row_seq[m] = lo * ps.samples; row_pos[m] = p;
        if (p % ps.group == 0) {
            const int g = ps.grp_off[lo] + p / ps.group;
            grp_row0[g] = m;
            grp_cnt[g] = min(ps.group, ps.len[lo] - 1 - p);
        }
    }
    embed_row<T, 128, false>(emb + (size_t)tok * d, pos + (size_t)p * d, h + (size_t)m * d, nullptr, d, NextLn{}, 0, nullptr);
}

// Keys / values of a query's first sequence to its other samples: one block per (layer and K or V, key/value head, query),
// 16 bytes at a time, read once and written samples - 1 times.  cache: [layers * 2][batch][heads][t_max][row_bytes].
// grid: (layers * 2, heads, queries); block: 256.
__global__ void __launch_bounds__(256) copy_samples_kernel(unsigned char* cache, size_t layer_bytes, int samples, int t_max, int row_bytes,
                                                           const int* __restrict__ len) {
    const size_t pitch = (size_t)t_max * row_bytes, seq = pitch * gridDim.y;
    unsigned char* src = cache + blockIdx.x * layer_bytes + (size_t)blockIdx.z * samples * seq + blockIdx.y * pitch;
    const int n16 = (len[blockIdx.z] - 1) * (row_bytes >> 4);
    for (int i = threadIdx.x; i < n16; i += 256) {
        const uint4 v = reinterpret_cast<const uint4*>(src)[i];
        for (int j = 1; j < samples; ++j) reinterpret_cast<uint4*>(src + j * seq)[i] = v;
    }
}

// Arg-max of one row from the per-tile (value, index) pairs an output-head GEMM left behind; lowest index
// on ties.  Warp-wide; every lane returns the result.
__device__ __forceinline__ int argmax_from_tiles(const float* val, const int* idx, int n_tiles) {
    const int lane = threadIdx.x & 31;
    float bv = -INFINITY;
    int bi = INT_MAX;
    for (int t0 = lane; t0 < n_tiles; t0 += 256) {   // eight loads in flight per lane
        float v[8];
        int ix[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int t = t0 + 32 * u;
            v[u] = t < n_tiles ? __ldcg(val + t) : -INFINITY;
            ix[u] = t < n_tiles ? __ldcg(idx + t) : INT_MAX;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u)
            if (v[u] > bv || (v[u] == bv && ix[u] < bi)) { bv = v[u]; bi = ix[u]; }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float ov = __shfl_xor_sync(0xffffffffu, bv, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (ov > bv || (ov == bv && oi < bi)) { bv = ov; bi = oi; }
    }
    return bi == INT_MAX ? 0 : bi;
}

// Start of a pass over decode rows: row set-up and x^(0) = Emb(t) + Pos(index) in one kernel (Eq. 1).
// Row m = b*nq + (r - r0) carries block row r of sequence b (row 0 = pending token, row r = draft r).
// The token of block row fin_r is not known yet as an id: it is the arg-max of the small model's last
// output-head GEMM, finished here from its per-tile results and recorded as draft fin_r.  grid: rows; block: 128.
template <typename T>
__global__ void __launch_bounds__(128) step_begin_kernel(LoopState st, int r0, int nq, int fin_r, const float* amax_val,
                                                         const int* amax_idx, int amax_stride, int n_tiles, int* row_tok,
                                                         int* row_seq, int* row_pos, const T* __restrict__ emb,
                                                         const T* __restrict__ pos, float* __restrict__ h, int d, float* snap, NextLn ln) {
    __shared__ int s_tok, s_pos;
    __shared__ float s_red[4];
    pdl_wait();
    pdl_launch_dependents();
    const int m = blockIdx.x;
    const int b = m / nq, r = r0 + (m - b * nq);
    if (threadIdx.x < 32) {
        int tok;
        if (r == 0) tok = st.pending[b];
        else if (r == fin_r) tok = argmax_from_tiles(amax_val + (size_t)b * amax_stride, amax_idx + (size_t)b * amax_stride, n_tiles);
        else tok = st.drafts[b * st.gamma_limit + r - 1];
        if (threadIdx.x == 0) {
            if (r == fin_r && r > 0) st.drafts[b * st.gamma_limit + r - 1] = tok;
            const int p = st.n[b] - 1 + r;
            s_tok = tok; s_pos = p;
            row_tok[m] = tok; row_seq[m] = b; row_pos[m] = p;
        }
    }
    __syncthreads();
    // (snap: copy for the FF_Tandem projection of x^(0))
    embed_row<T, 128, sizeof(T) == 2>(emb + (size_t)s_tok * d, pos + (size_t)s_pos * d, h + (size_t)m * d, snap ? snap + (size_t)m * d : nullptr, d, ln, m, s_red);
}

__device__ __forceinline__ float block_sum_128(float v, float* red) {
    v = warp_sum(v);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    return red[0] + red[1] + red[2] + red[3];
}

// Four normalised values to the output row: fp32 as they are, bf16 rounded.
__device__ __forceinline__ void ln_store4(float* orow, int k4, float y0, float y1, float y2, float y3) {
    reinterpret_cast<float4*>(orow)[k4] = make_float4(y0, y1, y2, y3);
}
__device__ __forceinline__ void ln_store4(bf16* orow, int k4, float y0, float y1, float y2, float y3) {
    const __nv_bfloat162 lo = __floats2bfloat162_rn(y0, y1), hi = __floats2bfloat162_rn(y2, y3);
    reinterpret_cast<uint2*>(orow)[k4] = make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
}
// The same as value + remainder, the remainder `lo` elements behind the value (lo == 0: the value alone).
template <bool PL, typename TO>
__device__ __forceinline__ void ln_put4(TO* orow, size_t lo, int k4, float y0, float y1, float y2, float y3) {
    if constexpr (PL) {
        const __nv_bfloat162 a = __floats2bfloat162_rn(y0, y1), b = __floats2bfloat162_rn(y2, y3);
        reinterpret_cast<uint2*>(orow)[k4] = make_uint2(*reinterpret_cast<const uint32_t*>(&a), *reinterpret_cast<const uint32_t*>(&b));
        ln_store4(orow + lo, k4, y0 - __low2float(a), y1 - __high2float(a), y2 - __low2float(b), y3 - __high2float(b));
    } else {
        ln_store4(orow, k4, y0, y1, y2, y3);
    }
}
// LayerNorm of fp32 rows (biased variance, eps 1e-5) ahead of the GEMMs, output in the storage type: the row sits in
// registers between the passes (up to 4096 elements), loads and stores are 16 bytes wide (8191 rows of 4096: 56 us with
// scalar accesses in three passes).  raw (nullable): bf16 copy of the row as it is, for the FF_Tandem projection that reads
// the same residual stream (a pass of its own over it took 120 us there).  A block keeps gain and bias in registers over its
// rows and fetches a row ahead: with one row per block those 32 KB per 16 KB of row made the L2 traffic (51 us at 8191 rows).
// PL (TO = bf16): output and raw copy as two planes, values and, `lo` elements behind them, remainders.
// grid: at most M blocks; block: 128; d % 4 == 0.
template <typename TO, bool PL = false>
__global__ void __launch_bounds__(128) layernorm_rows_kernel(const float* __restrict__ x, const float* __restrict__ gain,
                                                             const float* __restrict__ bias, TO* __restrict__ out, int d,
                                                             int M, bf16* raw, size_t lo = 0) {
    __shared__ float red[4];
    const int d4 = d >> 2;
    if (d4 <= 8 * 128) {
        // gains and biases are parameters: fetched while the kernel that writes x is still running
        float4 gq[8], bq[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int k4 = threadIdx.x + 128 * u;
            gq[u] = k4 < d4 ? __ldg(reinterpret_cast<const float4*>(gain) + k4) : make_float4(0.f, 0.f, 0.f, 0.f);
            bq[u] = k4 < d4 ? __ldg(reinterpret_cast<const float4*>(bias) + k4) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        pdl_wait();
        pdl_launch_dependents();
        float4 tn[8];
        auto fetch = [&](int row) {
            const float4* xr = reinterpret_cast<const float4*>(x + (size_t)row * d);
#pragma unroll
            for (int u = 0; u < 8; ++u) tn[u] = (threadIdx.x + 128 * u < d4) ? __ldcg(xr + threadIdx.x + 128 * u) : make_float4(0.f, 0.f, 0.f, 0.f);
        };
        fetch(blockIdx.x);
        for (int row = blockIdx.x; row < M; row += gridDim.x) {
            float4 t[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) t[u] = tn[u];
            if (row + gridDim.x < M) fetch(row + gridDim.x);   // under this row's reductions
            TO* orow = out + (size_t)row * d;
            if (raw) {
#pragma unroll
                for (int u = 0; u < 8; ++u)
                    if (threadIdx.x + 128 * u < d4) ln_put4<PL>(raw + (size_t)row * d, lo, threadIdx.x + 128 * u, t[u].x, t[u].y, t[u].z, t[u].w);
            }
            float s = 0.f;
#pragma unroll
            for (int u = 0; u < 8; ++u) s += (t[u].x + t[u].y) + (t[u].z + t[u].w);
            const float mu = block_sum_128(s, red) / d;
            float q = 0.f;
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                if (threadIdx.x + 128 * u < d4) {
                    const float d0 = t[u].x - mu, d1 = t[u].y - mu, d2 = t[u].z - mu, d3 = t[u].w - mu;
                    q = fmaf(d0, d0, q); q = fmaf(d1, d1, q); q = fmaf(d2, d2, q); q = fmaf(d3, d3, q);
                }
            }
            const float rs = 1.0f / sqrtf(block_sum_128(q, red) / d + 1e-5f);
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int k4 = threadIdx.x + 128 * u;
                if (k4 < d4) {
                    const float4 g = gq[u], b = bq[u];
                    ln_put4<PL>(orow, lo, k4, (t[u].x - mu) * rs * g.x + b.x, (t[u].y - mu) * rs * g.y + b.y,
                              (t[u].z - mu) * rs * g.z + b.z, (t[u].w - mu) * rs * g.w + b.w);
                }
            }
        }
    } else {
        pdl_wait();
        pdl_launch_dependents();
        for (int row = blockIdx.x; row < M; row += gridDim.x) {
            const float4* xr = reinterpret_cast<const float4*>(x + (size_t)row * d);
            TO* orow = out + (size_t)row * d;
            float s = 0.f;
            for (int k4 = threadIdx.x; k4 < d4; k4 += 128) {
                const float4 t = __ldcg(xr + k4);
                s += (t.x + t.y) + (t.z + t.w);
                if (raw) ln_put4<PL>(raw + (size_t)row * d, lo, k4, t.x, t.y, t.z, t.w);
            }
            const float mu = block_sum_128(s, red) / d;
            float q = 0.f;
            for (int k4 = threadIdx.x; k4 < d4; k4 += 128) {
                const float4 t = __ldcg(xr + k4);
                const float d0 = t.x - mu, d1 = t.y - mu, d2 = t.z - mu, d3 = t.w - mu;
                q = fmaf(d0, d0, q); q = fmaf(d1, d1, q); q = fmaf(d2, d2, q); q = fmaf(d3, d3, q);
            }
            const float rs = 1.0f / sqrtf(block_sum_128(q, red) / d + 1e-5f);
            for (int k4 = threadIdx.x; k4 < d4; k4 += 128) {
                const float4 t = __ldcg(xr + k4);
                const float4 g = __ldg(reinterpret_cast<const float4*>(gain) + k4), b = __ldg(reinterpret_cast<const float4*>(bias) + k4);
                ln_put4<PL>(orow, lo, k4, (t.x - mu) * rs * g.x + b.x, (t.y - mu) * rs * g.y + b.y, (t.z - mu) * rs * g.z + b.z,
                          (t.w - mu) * rs * g.w + b.w);
            }
        }
    }
}

// The same for more rows: a warp per row, the row in its registers, no barrier between the passes.  V: float4s per lane, d <= 128 V; up
// to 1024 elements gain and bias stay in registers, beyond they come from L1 for every row.
// Prompt passes with it: small pair (28 LayerNorms of 511 rows of 1024 or 512) 731 -> 696 us, 3999 rows 2.49 -> 2.31 ms; medium pair,
// 1999 rows of 2048, 5.99 -> 5.73 ms; rows of 4096 no faster than with a block per row.
// grid: at most ceil(M / 4) blocks; block: 128; d % 4 == 0.
constexpr int LNW_MAX = 2048;
template <typename TO, bool PL, int V>
__global__ void __launch_bounds__(128) layernorm_warp_kernel(const float* __restrict__ x, const float* __restrict__ gain, const float* __restrict__ bias,
                                                             TO* __restrict__ out, int d, int M, bf16* raw, size_t lo) {
    constexpr bool KEEP = V <= 8;
    const int lane = threadIdx.x & 31, d4 = d >> 2;
    auto parameter = [&](const float* p, int v) {
        return lane + 32 * v < d4 ? __ldg(reinterpret_cast<const float4*>(p) + lane + 32 * v) : make_float4(0.f, 0.f, 0.f, 0.f);
    };
    float4 g[KEEP ? V : 1], b[KEEP ? V : 1];
    if constexpr (KEEP) {
#pragma unroll
        for (int v = 0; v < V; ++v) { g[v] = parameter(gain, v); b[v] = parameter(bias, v); }
    }
    pdl_wait();
    pdl_launch_dependents();
    for (int row = blockIdx.x * 4 + (threadIdx.x >> 5); row < M; row += 4 * gridDim.x) {
        const float4* xr = reinterpret_cast<const float4*>(x + (size_t)row * d);
        TO* orow = out + (size_t)row * d;
        float4 t[V];
        float s = 0.f, q = 0.f;
#pragma unroll
        for (int v = 0; v < V; ++v) t[v] = lane + 32 * v < d4 ? __ldcg(xr + lane + 32 * v) : make_float4(0.f, 0.f, 0.f, 0.f);
        if (raw) {
#pragma unroll
            for (int v = 0; v < V; ++v)
                if (lane + 32 * v < d4) ln_put4<PL>(raw + (size_t)row * d, lo, lane + 32 * v, t[v].x, t[v].y, t[v].z, t[v].w);
        }
#pragma unroll
        for (int v = 0; v < V; ++v) s += (t[v].x + t[v].y) + (t[v].z + t[v].w);
        const float mu = warp_sum(s) / d;
#pragma unroll
        for (int v = 0; v < V; ++v)
            if (lane + 32 * v < d4) {
                const float d0 = t[v].x - mu, d1 = t[v].y - mu, d2 = t[v].z - mu, d3 = t[v].w - mu;
                q = fmaf(d0, d0, q); q = fmaf(d1, d1, q); q = fmaf(d2, d2, q); q = fmaf(d3, d3, q);
            }
        const float rs = 1.0f / sqrtf(warp_sum(q) / d + 1e-5f);
#pragma unroll
        for (int v = 0; v < V; ++v)
            if (lane + 32 * v < d4) {
                const float4 gv = KEEP ? g[KEEP ? v : 0] : parameter(gain, v), bv = KEEP ? b[KEEP ? v : 0] : parameter(bias, v);
                ln_put4<PL>(orow, lo, lane + 32 * v, (t[v].x - mu) * rs * gv.x + bv.x, (t[v].y - mu) * rs * gv.y + bv.y,
                            (t[v].z - mu) * rs * gv.z + bv.z, (t[v].w - mu) * rs * gv.w + bv.w);
            }
    }
}

// bf16 copy of the residual stream for a projection that no LayerNorm of the large model follows.  n a multiple of 8.  PL: two planes,
// the remainders `lo` elements behind the values.
// grid: enough blocks of 256 for n / 8.
template <bool PL>
__global__ void __launch_bounds__(256) cast_rows_kernel(const float* __restrict__ x, bf16* __restrict__ out, size_t n, size_t lo) {
    pdl_wait();
    pdl_launch_dependents();
    const size_t i = ((size_t)blockIdx.x * 256 + threadIdx.x) * 8;
    if (i >= n) return;
    const float4 a = __ldcg(reinterpret_cast<const float4*>(x + i)), b = __ldcg(reinterpret_cast<const float4*>(x + i) + 1);
    ln_put4<PL>(out + i, lo, 0, a.x, a.y, a.z, a.w);
    ln_put4<PL>(out + i, lo, 1, b.x, b.y, b.z, b.w);
}

// Verify / accept / rollback (Section 3.1), one warp per sequence, one CTA.
//   a = longest prefix of drafts equal to the large model's tokens (or forced);
//   the sequence gains d_1..d_a and g_{a+1}; n advances; g_{a+1} becomes pending.
// Rolling the caches back is the update of n: positions >= n-1 are rewritten by the next iteration.
// When amax_val is given, the large model's arg-max per block row is first finished from the per-tile results of
// its output-head GEMM.
// mode 3 is the round of stand-alone Tandem without the free token (Section 3 "Inference", "Representation
// Generation Only"; Figure 3): the large model has read gamma rows and predicted nothing, all gamma tokens of the
// small model are kept and the last one becomes pending.  The last draft is then not a block row, so nobody has
// turned it into a token id yet: when fin_val is given it is finished here from the small head's per-tile results.
// mode 4 is sampled SPEED: sample_verify_kernel has already written each sequence's accept length and, at that index
// of its targets, the token drawn after the kept drafts; this kernel only does the bookkeeping.
// block_len (nullable): per-sequence number of drafts of this iteration when the router chose it.
// A lone CTA at the end of the iteration's chain, bound by the latency of dependent loads: 32 warps finish up to 32
// arg-max rows side by side, a sequence's drafts and targets are fetched by the lanes of its warp in one round trip, and
// the totals for the host are summed in shared memory.
// block: VERIFY_THREADS; batch * (gamma + 1) <= 256.
constexpr int VERIFY_THREADS = 1024;
__global__ void __launch_bounds__(VERIFY_THREADS) verify_kernel(LoopState st, int batch, int gamma, int mode, unsigned long long seed,
                                                     int max_new, const float* amax_val, const int* amax_idx, int amax_stride,
                                                     int n_tiles, const float* fin_val, const int* fin_idx, const int* block_len) {
    __shared__ int s_tok[256];                     // the large model's token per block row (mode 3: the last draft per sequence)
    __shared__ int s_live, s_nmax, s_nsum, s_left;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr int WARPS = VERIFY_THREADS / 32;
    if (threadIdx.x == 0) { s_live = 0; s_nmax = 0; s_nsum = 0; s_left = 0; }
    pdl_wait();
    pdl_launch_dependents();
    const bool finish_last = mode == 3 && fin_val != nullptr && gamma > 0;
    const bool finish_rows = mode != 3 && mode != 4 && amax_val != nullptr;   // (mode 4: the sampled decisions are already in place)
    const int rows = finish_last ? batch : (finish_rows ? batch * (gamma + 1) : 0);
    const float* val = finish_last ? fin_val : amax_val;
    const int* idx = finish_last ? fin_idx : amax_idx;
    for (int m = warp; m < rows; m += WARPS) {
        const int tok = argmax_from_tiles(val + (size_t)m * amax_stride, idx + (size_t)m * amax_stride, n_tiles);
        if (lane == 0) s_tok[m] = tok;
    }
    __syncthreads();
    const int iteration = st.counters[0];
    const int live_before = st.counters[1];
    for (int b = warp; b < batch; b += WARPS) {
        int* dp = st.drafts + b * st.gamma_limit;
        int* gp = st.targets + b * (st.gamma_limit + 1);
        // lane i: draft d_{i+1} and target g_{i+1}, as far as the block goes
        int d = lane < gamma ? __ldcg(dp + lane) : -1;
        if (finish_last && lane == gamma - 1) { d = s_tok[b]; dp[lane] = d; }
        int g = -1;
        if (lane <= gamma && mode != 3) {
            if (finish_rows) { g = s_tok[b * (gamma + 1) + lane]; gp[lane] = g; }
            else g = __ldcg(gp + lane);
        }
        const int done = st.done[b], em = st.emitted[b], n = st.n[b], pending = st.pending[b];
        const int gamma_b = block_len ? min(block_len[b], gamma) : gamma;
        const int sampled_a = mode == 4 ? st.accept_len[b] : 0;
        int n_new = n, left = 0, live = 0;
        if (!done) {
            int a;
            if (mode == 1 || mode == 3) a = gamma;
            else if (mode == 4) a = min(max(sampled_a, 0), gamma);   // sampled SPEED: decided by sample_verify_kernel, with g[a] the token it drew
            else if (mode == 2) a = (int)(splitmix64(splitmix64(splitmix64(seed) ^ (unsigned long long)b) ^ (unsigned long long)iteration) % (unsigned long long)(gamma + 1));
            else a = __ffs(~__ballot_sync(0xffffffffu, lane < gamma_b && d == g)) - 1;   // adaptive block length: only the drafts really made count
            const int bonus = __shfl_sync(0xffffffffu, g, a);
            const int take = min(mode == 3 ? a : a + 1, max_new - em);
            const int tok = lane < a ? d : bonus;          // the block's token number lane + 1
            if (lane < take && em + lane < st.out_cap) st.out_ids[(size_t)b * st.out_cap + em + lane] = tok;
            const int last = __shfl_sync(0xffffffffu, tok, max(take - 1, 0));
            n_new = n + take;
            live = em + take < max_new;
            left = max_new - em - take;
            if (lane == 0) {
                st.accept_len[b] = a;
                atomicAdd(st.hist + a, 1ull);
                st.emitted[b] = em + take;
                st.n[b] = n_new;
                st.pending[b] = take > 0 ? last : pending;
                if (!live) st.done[b] = 1;
            }
        }
        if (lane == 0) {
            atomicAdd(&s_live, live);
            atomicMax(&s_nmax, n_new);
            atomicAdd(&s_nsum, n_new);
            atomicMax(&s_left, left);
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        const int iters = st.counters[5] + (live_before > 0 ? 1 : 0);
        const int ticket = st.counters[6] + 1;
        // publish to the host: data first, then the ticket it polls on
        st.host_flags[1] = s_live;
        st.host_flags[2] = s_nmax;
        st.host_flags[3] = s_nsum;
        st.host_flags[4] = iters;
        st.host_flags[7] = s_left;
        __threadfence_system();
        st.host_flags[0] = ticket;
        if (live_before > 0) st.counters[0] = iteration + 1;
        st.counters[1] = s_live;
        st.counters[3] = s_nmax;
        st.counters[4] = s_nsum;
        st.counters[5] = iters;
        st.counters[6] = ticket;
    }
}

// Teacher-forced Tandem forward, bf16: all given tokens that have a next one are rows of one pass (or of a few, where the work space is
// short), sequence after sequence.
struct ForcedRows {
    const int* ids;      // the sequences, one after the other: row v of sequence b is ids[v + b], its next token ids[v + b + 1]
    const int* start;    // [batch + 1] first row of each sequence, over all passes
    int batch, v0, rows; // this pass: rows v0 .. v0 + rows - 1, whole blocks
    int gamma, vocab;    // positions per block (a sequence's last one may be shorter)
    int group;           // queries per attention group: of the large model, or a block of the small model's
    int* row_seq; int* row_pos;
    int* keep;           // [rows] where the row's logits stay readable: step within the block * batch + sequence for a sequence's last block, else -1
    int* truth;          // [rows] the next token
    int* grp; int* grp_pos;                      // attention groups, see AttnArgs::pass_grp
    float* nll; int* top;                        // [rows of all passes] scores
    const float* hidden; int d_large;            // the large model's final residual stream [rows][d_large]
    float* last_hidden; float* last_logits;      // readable afterwards, of the sequences' last blocks: [batch][gamma][d_large], [gamma][batch][vocab]
};

// Start of one model's part of such a pass: row set-up and embedding, and in one more block the attention groups and the sequences' loop
// state.  The small model's part has batch * gamma blocks more: the large model's final stream of the sequences' last blocks, and
// zeros where a block ends before gamma positions.
// grid: rows + 1 (+ batch * gamma); block: 128.
__global__ void __launch_bounds__(128) forced_rows_kernel(LoopState st, ForcedRows f, const bf16* __restrict__ emb, const bf16* __restrict__ pos,
                                                          float* __restrict__ h, int d, int ticket, int router_ticket) {
    __shared__ int s_first[128], s_n[128];
    pdl_wait();
    pdl_launch_dependents();
    const int m = blockIdx.x;
    if (m > f.rows) {
        const int i = m - f.rows - 1, b = i / f.gamma, s = i - b * f.gamma, n = f.start[b + 1] - f.start[b];
        const int last = (n - 1) / f.gamma * f.gamma, row = f.start[b] + last + s - f.v0;   // the last block's first position
        float* dst = f.last_hidden + (size_t)i * f.d_large;
        if (last + s >= n) {
            for (int k = threadIdx.x; k < f.d_large; k += 128) dst[k] = 0.f;
            float* row = f.last_logits + (size_t)(s * f.batch + b) * f.vocab;
            if ((f.vocab & 3) == 0) { for (int k = threadIdx.x; k < f.vocab >> 2; k += 128) reinterpret_cast<float4*>(row)[k] = make_float4(0.f, 0.f, 0.f, 0.f); }
            else for (int k = threadIdx.x; k < f.vocab; k += 128) row[k] = 0.f;
        } else if (row >= 0 && row < f.rows) {
            const float4* src = reinterpret_cast<const float4*>(f.hidden + (size_t)row * f.d_large);
            for (int k = threadIdx.x; k < f.d_large >> 2; k += 128) reinterpret_cast<float4*>(dst)[k] = __ldcg(src + k);
        }
        return;
    }
    if (m == f.rows) {
        const int b = threadIdx.x;   // (batch <= 128: at least two rows per sequence in every context)
        s_first[b] = s_n[b] = 0;
        if (b < f.batch) {
            const int first = max(f.start[b], f.v0);
            s_first[b] = first - f.v0;
            s_n[b] = max(0, min(f.start[b + 1], f.v0 + f.rows) - first);
            st.n[b] = f.start[b + 1] - f.start[b] + 1;
            st.pending[b] = f.ids[f.start[b + 1] + b];
        }
        __syncthreads();
        for (int i = 0, g = 0; i < f.batch; ++i) {
            const int n = s_n[i], groups = (n + f.group - 1) / f.group;
            for (int j = threadIdx.x; j < groups; j += 128) {
                f.grp[g + j] = (s_first[i] + j * f.group) | min(f.group, n - j * f.group) << 16 | i << 20;
                f.grp_pos[g + j] = f.v0 + s_first[i] - f.start[i] + j * f.group;
            }
            g += groups;
        }
        if (b == 0) { st.counters[6] = ticket; st.counters[8] = router_ticket; }
        return;
    }
    const int v = f.v0 + m;
    int lo = 0, hi = f.batch - 1;   // the last sequence that begins at or before row v
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (f.start[mid] <= v) lo = mid; else hi = mid - 1;
    }
    const int p = v - f.start[lo], tok = f.ids[v + lo];
    if (threadIdx.x == 0) {
        const int s = p - (f.start[lo + 1] - f.start[lo] - 1) / f.gamma * f.gamma;
        f.row_seq[m] = lo; f.row_pos[m] = p;
        f.keep[m] = s >= 0 ? s * f.batch + lo : -1;
        f.truth[m] = f.ids[v + lo + 1];
    }
    embed_row<bf16, 128, false>(emb + (size_t)tok * d, pos + (size_t)p * d, h + (size_t)m * d, nullptr, d, NextLn{}, 0, nullptr);
}

// Scores of rows whose output head left (maximum, its index, sum of exponentials) per tile of features and the true token's
// logit (in nll): negative log-likelihood and arg-max (lowest index on ties).  One warp per row; n_tiles values each, 500 at 32000 logits.
// grid: ceil(rows / 8); block: 256.
__global__ void __launch_bounds__(256) score_tiles_kernel(int rows, int n_tiles, const float* __restrict__ tile_max, const int* __restrict__ tile_idx,
                                                          const float* __restrict__ tile_sum, float* __restrict__ nll, int* __restrict__ top1) {
    pdl_wait();
    pdl_launch_dependents();
    const int m = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (m >= rows) return;
    const size_t base = (size_t)m * n_tiles;
    const int top = argmax_from_tiles(tile_max + base, tile_idx + base, n_tiles);
    float best = -INFINITY;
    for (int t = lane; t < n_tiles; t += 32) best = fmaxf(best, __ldcg(tile_max + base + t));
    best = warp_max(best);
    float tot = 0.f;
    for (int t = lane; t < n_tiles; t += 32) {
        const float z = __ldcg(tile_sum + base + t);
        tot += z > 0.f ? z * expf(__ldcg(tile_max + base + t) - best) : 0.f;
    }
    tot = warp_sum(tot);
    if (lane == 0) {
        nll[m] = best + logf(tot) - nll[m];
        top1[m] = top;
    }
}

// Teacher-forced Tandem forward in rounds (fp32): the next gamma tokens of every sequence become the
// "drafts" of the round, so that draft step s reads the true token of its position.  forced: [batch][stride] token
// ids; positions at or beyond forced_len[b] read as token 0 (rows past a sequence's end are computed and ignored).
// grid: 1; block: 256.
__global__ void __launch_bounds__(256) forced_fill_kernel(LoopState st, int batch, int gamma, const int* __restrict__ forced,
                                                          const int* __restrict__ forced_len, int stride) {
    pdl_wait();
    pdl_launch_dependents();
    for (int i = threadIdx.x; i < batch * gamma; i += 256) {
        const int b = i / gamma, r = i - b * gamma;
        const int p = st.n[b] + r;                       // position of the token that draft r + 1 stands for
        st.drafts[b * st.gamma_limit + r] = p < forced_len[b] ? forced[(size_t)b * stride + p] : 0;
    }
}

// Scores of a teacher-forced round: for draft step s of sequence b, at position p = n_b - 1 + s, the negative
// log-likelihood of the true token at p + 1 under softmax(logits) and the arg-max (lowest id on ties).
// Bound by the latency of a row's passes: a row is dealt to the 64 warps of a cluster, whose ranges stay in registers between the
// maximum and the sum (up to 32768 logits, else they are read again: 9.7 us a launch at 32768 and 32776 logits, 11.3 at 65536,
// 13.8 at 131072); the warps' maxima, positions and sums meet in the first
// CTA.  32000 logits, 16 rows: 19 us with one CTA per row and two passes over it, about 6 us like this.
// logits: [gamma][batch][V].  grid: (SCR_CLUSTER, gamma, batch), a cluster per row; block: SCR_THREADS.
constexpr int SCR_CLUSTER = 8, SCR_THREADS = 256, SCR_RANGES = SCR_CLUSTER * SCR_THREADS / 32, SCR_REGS = 16;
__global__ void __launch_bounds__(SCR_THREADS) score_rows_kernel(LoopState st, int batch, const float* __restrict__ logits, int V,
                                                                 const int* __restrict__ forced, const int* __restrict__ forced_len, int stride,
                                                                 float* __restrict__ nll, int* __restrict__ top1) {
    __shared__ float s_max[SCR_RANGES], s_sum[SCR_RANGES], s_pos[SCR_RANGES];   // first CTA: one entry per range (s_pos: the bits of an int)
    cluster_arrive_relaxed();   // opening handshake
    pdl_wait();
    pdl_launch_dependents();
    cluster_wait();
    const int s = blockIdx.y, b = blockIdx.z, lane = threadIdx.x & 31;
    const int p = st.n[b] - 1 + s;
    if (p + 1 >= forced_len[b]) return;                  // no true next token: nothing to score (the same for the whole cluster)
    const float* row = logits + ((size_t)s * batch + b) * V;
    const int id = blockIdx.x * (SCR_THREADS / 32) + (threadIdx.x >> 5);
    const int chunk = (((V + SCR_RANGES - 1) / SCR_RANGES) + 31) & ~31;
    const int i0 = min(V, id * chunk), i1 = min(V, i0 + chunk);
    float best = -INFINITY, z = 0.f;
    int bi = INT_MAX;
    auto take = [&](float v, int i) {
        if (v > best || (v == best && i < bi)) { best = v; bi = i; }
    };
    auto across = [&]() {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float ov = __shfl_xor_sync(0xffffffffu, best, o);
            take(ov, __shfl_xor_sync(0xffffffffu, bi, o));
        }
    };
    if (chunk <= 32 * SCR_REGS) {
        float x[SCR_REGS];
#pragma unroll
        for (int j = 0; j < SCR_REGS; ++j) x[j] = __ldcg(row + min(i0 + 32 * j + lane, V - 1));
#pragma unroll
        for (int j = 0; j < SCR_REGS; ++j) if (i0 + 32 * j + lane < i1) take(x[j], i0 + 32 * j + lane);
        across();
#pragma unroll
        for (int j = 0; j < SCR_REGS; ++j) z += i0 + 32 * j + lane < i1 ? expf(x[j] - best) : 0.f;
    } else {
#pragma unroll 8
        for (int i = i0 + lane; i < i1; i += 32) take(__ldcg(row + i), i);
        across();
#pragma unroll 8
        for (int i = i0 + lane; i < i1; i += 32) z += expf(__ldcg(row + i) - best);
    }
    z = warp_sum(z);
    if (lane == 0) {
        st_dsmem_f32(smem_u32(&s_max[id]), 0, best);
        st_dsmem_f32(smem_u32(&s_sum[id]), 0, z);
        st_dsmem_f32(smem_u32(&s_pos[id]), 0, __int_as_float(bi));
    }
    cluster_sync_all();
    if (blockIdx.x != 0 || threadIdx.x >= 32) return;
    best = -INFINITY;
    bi = INT_MAX;
    for (int r = lane; r < SCR_RANGES; r += 32) take(s_max[r], __float_as_int(s_pos[r]));
    across();
    float tot = 0.f;
    for (int r = lane; r < SCR_RANGES; r += 32) tot += s_sum[r] > 0.f ? s_sum[r] * expf(s_max[r] - best) : 0.f;   // (an empty range: 0)
    tot = warp_sum(tot);
    if (lane == 0) {
        const int truth = forced[(size_t)b * stride + p + 1];
        nll[(size_t)b * stride + p] = best + logf(tot) - __ldcg(row + truth);
        top1[(size_t)b * stride + p] = bi;
    }
}

// Test hook: gathers K or V of one (layer, sequence) from [H][t_max][dh] into fp32 [n][H*dh].
template <typename T>
__global__ void gather_kv_kernel(const T* __restrict__ cache_seq, float* __restrict__ dst, int n, int n_heads, int d_head, int t_max) {
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int d = n_heads * d_head;
    if (i >= (size_t)n * d) return;
    const int t = (int)(i / d), c = (int)(i - (size_t)t * d);
    const int h = c / d_head, el = c - h * d_head;
    dst[i] = to_float(cache_seq[((size_t)h * t_max + t) * d_head + el]);
}

}  // namespace tandem
