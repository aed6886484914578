// SIMT GEMMs  y[m][n] = sum_k x[m][k] * W[n][k]  (weights [out][in]) with fused epilogues.
//
//  gemm_rows_kernel    few rows (the decode passes; prompts of up to 64 rows): one warp per one or four output
//                      columns streams the weight rows with 16-byte loads; the rows of x sit in shared memory,
//                      normalised on the way where LayerNorm precedes the map.
//                      Each output element is reduced in an order that depends only on K, never on the
//                      number of rows, so a block pass and a one-row pass give identical bits.
//  gemm_tiled_kernel   prompt path (many rows), classic shared-memory tiling.
//
// Both are the exact-arithmetic (fp32 FMA) paths of the fp32 test mode.
#pragma once
#include <limits.h>
#include <math.h>
#include "common.cuh"
#include "tc_common.cuh"

namespace tandem {

enum { EPI_STORE = 0, EPI_STORE_F32 = 1, EPI_GELU = 2, EPI_RESID = 3, EPI_QKV = 4, EPI_KV = 5 };
constexpr int EPI_ARGMAX = 6;   // few rows: fp32 store plus the (max, index) of each row within a tile of features (fp32 mode: a block's columns)

struct EpiArgs {
    void* out;            // EPI_STORE/GELU: T [M][ldo] (GELU on the tensor-core decode path: float);  STORE_F32/RESID: float [M][ldo];  QKV: q as T [M][ldo]
    int ldo;
    void* kcache;         // QKV / KV: this layer's keys   [B][H][t_max][d_head] (T)
    void* vcache;         //           this layer's values
    const int* row_seq;   // [M] sequence of each row (null: row j is sequence j at position 0 on the tensor-core decode path, position j of one sequence elsewhere)
    const int* row_pos;   // [M] absolute position of each row
    int n_heads, d_head, t_max;   // n_heads: key/value heads of the cache
    int seg0;             // QKV / KV: columns of the first segment (QKV: the queries, d_model; KV: the keys)
    int seg;              //           columns of every further segment (keys / values: kv heads * d_head)
    void* out_lo;         // EPI_GELU on the tensor-core decode path, optional: `out` is then the bf16 plane of the values and this
                          // the bf16 plane of the remainders (x = value + remainder), both [M][ldo], for a consumer that loads them by TMA
    void* snap;           // EPI_RESID in decode passes: optional fp32 copy of the new values [M][snap_ld]
    int snap_ld;
    NextLn ln;            // EPI_RESID on the tensor-core decode path, see NextLn
};

struct WSegs {            // up to three weight matrices stacked along N: [seg_rows0][K], then [seg_rows][K] each
    const void* w[3];
    int seg_rows0;
    int seg_rows;
};

template <typename T>
__device__ __forceinline__ const T* weight_row(const WSegs& ws, int n, int K) {
    if (n < ws.seg_rows0) return static_cast<const T*>(ws.w[0]) + (size_t)n * K;
    const int r = n - ws.seg_rows0, s = r / ws.seg_rows;
    return static_cast<const T*>(ws.w[1 + s]) + (size_t)(r - s * ws.seg_rows) * K;
}

template <typename T, int EPI>
__device__ __forceinline__ void epilogue(const EpiArgs& e, int m, int n, float v) {
    if (EPI == EPI_STORE) {
        static_cast<T*>(e.out)[(size_t)m * e.ldo + n] = from_float<T>(v);
    } else if (EPI == EPI_STORE_F32) {
        static_cast<float*>(e.out)[(size_t)m * e.ldo + n] = v;
    } else if (EPI == EPI_GELU) {
        static_cast<T*>(e.out)[(size_t)m * e.ldo + n] = from_float<T>(sizeof(T) == 2 ? gelu_bf16_out(v) : gelu_exact(v));
    } else if (EPI == EPI_RESID) {
        float* p = static_cast<float*>(e.out) + (size_t)m * e.ldo + n;
        const float h = *p + v;
        *p = h;
        if (sizeof(T) == 4 && e.snap) static_cast<float*>(e.snap)[(size_t)m * e.snap_ld + n] = h;   // (bf16: the few-row kernel has its own epilogue)
    } else {
        int s = 0, c = n;
        if (n >= e.seg0) { s = 1 + (n - e.seg0) / e.seg; c = (n - e.seg0) - (s - 1) * e.seg; }
        if (EPI == EPI_QKV) {
            if (s == 0) {
                static_cast<T*>(e.out)[(size_t)m * e.ldo + c] = from_float<T>(v);
                return;
            }
            s -= 1;
        }
        const int h = c / e.d_head, el = c - h * e.d_head;
        const bool rows = sizeof(T) == 4 || e.row_seq;
        const size_t seq = rows ? e.row_seq[m] : 0, pos = rows ? e.row_pos[m] : m;
        const size_t idx = ((seq * e.n_heads + h) * e.t_max + pos) * e.d_head + el;
        T* base = static_cast<T*>(s == 0 ? e.kcache : e.vcache);
        base[idx] = from_float<T>(v);
    }
}

constexpr int GS_THREADS = 256;
constexpr int GS_WARPS = GS_THREADS / 32;
constexpr int GS_KC = 2048;      // K elements of x staged in shared memory at a time; the longest row whose LayerNorm is fused

// Sums NV values over the warp's lanes, NV a power of two up to 32: halves the number of values a lane carries while it
// halves the distance, so NV values cost NV - 1 + (5 - log2 NV) shuffles instead of 5 NV.  Lane L returns the sum of value
// L >> (5 - log2 NV).  The tree of additions is the butterfly 16, 8, 4, 2, 1 for every value and every NV.
template <int NV>
__device__ __forceinline__ float warp_sum_many(float (&v)[NV], int lane) {
    int off = 16;
#pragma unroll
    for (int n = NV; n > 1; n >>= 1, off >>= 1) {
        const bool up = (lane & off) != 0;
#pragma unroll
        for (int i = 0; i < n / 2; ++i) {
            const float keep = up ? v[i + n / 2] : v[i], send = up ? v[i] : v[i + n / 2];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
        }
    }
#pragma unroll
    for (; off > 0; off >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], off);
    return v[0];
}

// Few rows, fp32: one warp per NC output columns, the rows of x in shared memory, LayerNorm fused (LN, K <= GS_KC).
// Bound by latency (the fp32 pair's matrices are 0.06-1 MB): NC = 1 spreads N = 256..1024 over the whole GPU, NC = 4 reads
// the staged rows once per four columns when there are columns enough; a warp's first weights are fetched before the wait
// on the preceding kernel; the row sums leave the warp through warp_sum_many and are finished by several lanes side by
// side.  One short row goes from L2 straight into the registers of every warp; more rows are staged by copies that pass no register.  Short
// rows are normalised in a warp's registers on their way, with gain and bias fetched ahead of the wait.
// At most 128 registers (FORM keeps apart what a launch never needs together), so that two CTAs fit a multiprocessor and a successor can
// set up beside its predecessor.  Requests of the 256 / 128-wide pair, 48 tokens at gamma 4, 1 / 4 / 8 / 16 sequences: 4.61 / 5.80 / 8.04 /
// 11.2 ms with staged rows in registers (up to 236: one CTA), 4.37 / 4.70 / 5.99 / 7.56 like this (1: 64 tokens), 4.45 / 4.85 / 6.15 / 7.03 squeezed
// into 80 registers for three CTAs.  1024 / 512-wide, 24 tokens at gamma 3, 4 sequences: 16.7, 13.7, 14.3.
// grid: (ceil(N / (GS_WARPS * NC)), ceil(M / MT)); dynamic smem: MT * min(K, GS_KC) floats.
enum { ROWS_PLAIN = 0, ROWS_LN_REGS = 1, ROWS_LN_SMEM = 2 };
// Longest row that a warp normalises in its registers: 512 elements with one column per warp, 256 with four.
__host__ __device__ constexpr int rows_ln_regs_max(int nc) { return 128 * (8 / nc < 4 ? 8 / nc : 4); }
template <int MT, int NC, int FORM, int EPI>
__global__ void __launch_bounds__(GS_THREADS, 2)
gemm_rows_kernel(const float* __restrict__ x, int ldx, int M, int K, WSegs ws, int N, const float* __restrict__ ln_g,
                 const float* __restrict__ ln_b, EpiArgs e, float* amax_val, int* amax_idx, int amax_stride) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    float* xs = reinterpret_cast<float*>(smem_raw);
    constexpr bool LN_REGS = FORM == ROWS_LN_REGS;
    constexpr int LV = rows_ln_regs_max(NC) / 128;   // float4s per lane of a row that is normalised in registers
    constexpr int PF = LN_REGS ? LV : 8 / NC;        // float4s of each column fetched ahead of the wait
    constexpr int NV = MT * NC;
    constexpr int LOG = NV == 1 ? 0 : (NV == 4 ? 2 : (NV == 8 ? 3 : (NV == 16 ? 4 : 5)));
    static_assert(MT <= GS_WARPS, "a warp per row where rows are normalised");
    static_assert(NV == 1 || NV == 4 || NV == 8 || NV == 16 || NV == 32, "warp_sum_many");
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n0 = (blockIdx.x * GS_WARPS + warp) * NC;
    const int m0 = blockIdx.y * MT, rows = min(MT, M - m0);
    const int KS = min(K, GS_KC);      // row stride in shared memory

    const float* wrow[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) wrow[c] = (n0 + c < N) ? weight_row<float>(ws, n0 + c, K) : nullptr;
    float4 wpre[NC][PF];               // weights are parameters: no need to wait for them
#pragma unroll
    for (int c = 0; c < NC; ++c)
#pragma unroll
        for (int i = 0; i < PF; ++i) {
            const int kk = (lane + 32 * i) * 4;
            wpre[c][i] = (wrow[c] != nullptr && kk < K) ? __ldg(reinterpret_cast<const float4*>(wrow[c] + kk)) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
    const bool direct = MT == 1 && (LN_REGS || (FORM == ROWS_PLAIN && K <= 128 * PF));
    float4 g[LN_REGS ? LV : 1], b[LN_REGS ? LV : 1];
    if constexpr (LN_REGS) {
#pragma unroll
        for (int v = 0; v < LV; ++v) {
            const int kk = (lane + 32 * v) * 4;
            g[v] = kk < K ? __ldg(reinterpret_cast<const float4*>(ln_g + kk)) : make_float4(0.f, 0.f, 0.f, 0.f);
            b[v] = kk < K ? __ldg(reinterpret_cast<const float4*>(ln_b + kk)) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
    }
    // where this thread's first float4 of a staging pass lies (the division ahead of the wait)
    const int r_first = threadIdx.x / (KS >> 2), v_first = threadIdx.x - r_first * (KS >> 2);
    pdl_wait();
    pdl_launch_dependents();

    float acc[NV];
#pragma unroll
    for (int i = 0; i < NV; ++i) acc[i] = 0.f;
    auto step = [&](const float4 (&w)[NC], int kk) {
#pragma unroll
        for (int r = 0; r < MT; ++r) {
            if (r >= rows) break;
            const float4 xv = *reinterpret_cast<const float4*>(xs + r * KS + kk);
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                float t = acc[r * NC + c];
                t = fmaf(xv.x, w[c].x, t); t = fmaf(xv.y, w[c].y, t); t = fmaf(xv.z, w[c].z, t); t = fmaf(xv.w, w[c].w, t);
                acc[r * NC + c] = t;
            }
        }
    };
    // A row of up to 128 * V elements into a warp's registers, normalised where LayerNorm precedes the map (biased variance, eps 1e-5)
    auto load_row = [&](auto& t, int m) {
        constexpr int V = sizeof(t) / sizeof(t[0]);
#pragma unroll
        for (int v = 0; v < V; ++v) {
            const int kk = (lane + 32 * v) * 4;
            t[v] = kk < K ? __ldcg(reinterpret_cast<const float4*>(x + (size_t)m * ldx + kk)) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        if constexpr (LN_REGS) {
            float sum = 0.f, q = 0.f;
#pragma unroll
            for (int v = 0; v < V; ++v) if ((lane + 32 * v) * 4 < K) sum += (t[v].x + t[v].y) + (t[v].z + t[v].w);
            const float mu = warp_sum(sum) / (float)K;
#pragma unroll
            for (int v = 0; v < V; ++v)
                if ((lane + 32 * v) * 4 < K) {
                    const float d0 = t[v].x - mu, d1 = t[v].y - mu, d2 = t[v].z - mu, d3 = t[v].w - mu;
                    q = fmaf(d0, d0, q); q = fmaf(d1, d1, q); q = fmaf(d2, d2, q); q = fmaf(d3, d3, q);
                }
            const float rs = 1.0f / sqrtf(warp_sum(q) / (float)K + 1e-5f);
#pragma unroll
            for (int v = 0; v < V; ++v) {
                t[v].x = (t[v].x - mu) * rs * g[v].x + b[v].x; t[v].y = (t[v].y - mu) * rs * g[v].y + b[v].y;
                t[v].z = (t[v].z - mu) * rs * g[v].z + b[v].z; t[v].w = (t[v].w - mu) * rs * g[v].w + b[v].w;
            }
        }
    };
    auto dot = [&](float& a, const float4& xv, const float4& w) { a = fmaf(xv.x, w.x, a); a = fmaf(xv.y, w.y, a); a = fmaf(xv.z, w.z, a); a = fmaf(xv.w, w.w, a); };
    if (direct) {
        float4 t[PF];
        load_row(t, m0);
#pragma unroll
        for (int v = 0; v < PF; ++v)
#pragma unroll
            for (int c = 0; c < NC; ++c) if ((lane + 32 * v) * 4 < K) dot(acc[c], t[v], wpre[c][v]);
    } else
    for (int k0 = 0; k0 < K; k0 += GS_KC) {
        const int kc = min(GS_KC, K - k0), vec = kc >> 2;
        __syncthreads();
        if constexpr (LN_REGS) {   // (the only staging pass) a warp per row
            if (warp < rows) {
                float4 t[LV];
                load_row(t, m0 + warp);
#pragma unroll
                for (int v = 0; v < LV; ++v)
                    if ((lane + 32 * v) * 4 < K) *reinterpret_cast<float4*>(xs + warp * KS + (lane + 32 * v) * 4) = t[v];
            }
        } else {   // all of this thread's copies in flight, none in registers
            int r = r_first, v = v_first;
            if (kc != KS) { r = threadIdx.x / vec; v = threadIdx.x - r * vec; }
            while (r < rows) {
                cp_async16(xs + r * KS + v * 4, x + (size_t)(m0 + r) * ldx + k0 + v * 4);
                for (v += GS_THREADS; v >= vec; v -= vec) ++r;
            }
            cp_async_commit();
            cp_async_wait_all();
        }
        __syncthreads();
        if constexpr (FORM == ROWS_LN_SMEM) {   // one warp per row, fixed lane-strided order (biased variance, eps 1e-5)
            if (warp < rows) {
                float* xr = xs + warp * KS;
                float s = 0.f;
#pragma unroll 4
                for (int k = lane * 4; k < K; k += 128) { const float4 t = *reinterpret_cast<const float4*>(xr + k); s += (t.x + t.y) + (t.z + t.w); }
                const float mu = warp_sum(s) / (float)K;
                float q = 0.f;
#pragma unroll 4
                for (int k = lane * 4; k < K; k += 128) {
                    const float4 t = *reinterpret_cast<const float4*>(xr + k);
                    const float d0 = t.x - mu, d1 = t.y - mu, d2 = t.z - mu, d3 = t.w - mu;
                    q = fmaf(d0, d0, q); q = fmaf(d1, d1, q); q = fmaf(d2, d2, q); q = fmaf(d3, d3, q);
                }
                const float rs = 1.0f / sqrtf(warp_sum(q) / (float)K + 1e-5f);
#pragma unroll 4
                for (int k = lane * 4; k < K; k += 128) {
                    float4 t = *reinterpret_cast<const float4*>(xr + k);
                    const float4 g = __ldg(reinterpret_cast<const float4*>(ln_g + k)), b = __ldg(reinterpret_cast<const float4*>(ln_b + k));
                    t.x = (t.x - mu) * rs * g.x + b.x; t.y = (t.y - mu) * rs * g.y + b.y;
                    t.z = (t.z - mu) * rs * g.z + b.z; t.w = (t.w - mu) * rs * g.w + b.w;
                    *reinterpret_cast<float4*>(xr + k) = t;
                }
            }
            __syncthreads();
        }
        int i = 0;
        if (k0 == 0) {
#pragma unroll
            for (int p = 0; p < PF; ++p) {
                const int kk = (lane + 32 * p) * 4;
                float4 w[NC];
#pragma unroll
                for (int c = 0; c < NC; ++c) w[c] = wpre[c][p];
                if (kk < kc) step(w, kk);
            }
            i = PF;
        }
        if constexpr (LN_REGS) break;   // (a row that fits a warp's registers has had all its products)
#pragma unroll 2
        for (int kk = (lane + 32 * i) * 4; kk < kc; kk += 128) {
            float4 w[NC];
#pragma unroll
            for (int c = 0; c < NC; ++c)
                w[c] = wrow[c] != nullptr ? __ldg(reinterpret_cast<const float4*>(wrow[c] + k0 + kk)) : make_float4(0.f, 0.f, 0.f, 0.f);
            step(w, kk);
        }
    }
    const float v = warp_sum_many<NV>(acc, lane);
    const int idx = lane >> (5 - LOG), r = idx / NC, n = n0 + idx % NC;
    const bool mine = (lane & ((32 >> LOG) - 1)) == 0 && r < rows;
    if constexpr (EPI == EPI_ARGMAX) {   // the block's columns, lowest feature on ties; the consumer finishes the row from the blocks' results
        __shared__ float s_v[GS_WARPS * NC][MT];
        if (mine) {
            if (n < N) static_cast<float*>(e.out)[(size_t)(m0 + r) * e.ldo + n] = v;
            s_v[warp * NC + idx % NC][r] = n < N ? v : -INFINITY;
        }
        __syncthreads();
        if (threadIdx.x < rows) {
            float best = -INFINITY;
            int bi = INT_MAX;
#pragma unroll
            for (int c = 0; c < GS_WARPS * NC; ++c) {
                const float t = s_v[c][threadIdx.x];
                if (t > best) { best = t; bi = blockIdx.x * GS_WARPS * NC + c; }
            }
            amax_val[(size_t)(m0 + threadIdx.x) * amax_stride + blockIdx.x] = best;
            amax_idx[(size_t)(m0 + threadIdx.x) * amax_stride + blockIdx.x] = bi;
        }
        return;
    }
    if (mine && n < N) epilogue<float, EPI>(e, m0 + r, n, v);
}

// Shared-memory tiled GEMM for many rows.  64x64 output tile, 16-deep K slices, 4x4 outputs per thread.
constexpr int GT_BM = 64, GT_BN = 64, GT_BK = 16, GT_THREADS = 256;

template <typename T, int EPI>
__global__ void __launch_bounds__(GT_THREADS)
gemm_tiled_kernel(const T* __restrict__ x, int ldx, int M, int K, WSegs ws, int N, EpiArgs e) {
    __shared__ float xs[GT_BK][GT_BM + 4];
    __shared__ float wsm[GT_BK][GT_BN + 4];
    const int tid = threadIdx.x;
    const int tx = tid & 15, ty = tid >> 4;
    const int m0 = blockIdx.y * GT_BM, n0 = blockIdx.x * GT_BN;
    // loader mapping: 64 rows x 16 k; each thread moves 4 consecutive k of one row
    const int lrow = tid >> 2, lk = (tid & 3) * 4;
    const T* xrow = (m0 + lrow < M) ? x + (size_t)(m0 + lrow) * ldx : nullptr;
    const T* wrow = (n0 + lrow < N) ? weight_row<T>(ws, n0 + lrow, K) : nullptr;

    float acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;

    for (int k0 = 0; k0 < K; k0 += GT_BK) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int k = k0 + lk + i;
            xs[lk + i][lrow] = (xrow != nullptr && k < K) ? to_float(xrow[k]) : 0.f;
            wsm[lk + i][lrow] = (wrow != nullptr && k < K) ? to_float(wrow[k]) : 0.f;
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < GT_BK; ++k) {
            float a[4], b[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) a[i] = xs[k][ty * 4 + i];
#pragma unroll
            for (int j = 0; j < 4; ++j) b[j] = wsm[k][tx * 4 + j];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int m = m0 + ty * 4 + i, n = n0 + tx * 4 + j;
            if (m < M && n < N) epilogue<T, EPI>(e, m, n, acc[i][j]);
        }
}

}  // namespace tandem
