// Attention over a KV cache laid out [seq][head][position][d_head].
//
// attn_kernel (fp32 mode; prompt pass at head size 32) serves three uses (Eq. 1 and Eq. 2, second line):
//   * the small model's decode step: one query per (sequence, head) over the mixed context; positions
//     the large model has processed hold large-derived keys/values, later ones the small model's own,
//     in one contiguous cache, so the boundary needs no special handling here;
//   * the large model's block pass: gamma+1 queries per sequence share one sweep over the cache, each
//     limited to its own position (causal inside the block);
//   * the prompt pass (LOOP = true): a group of consecutive queries sweeps all chunks up to its last position.
//
// The context is cut into chunks of ATT_CH positions anchored at absolute position 0.  In split mode one
// CTA handles one chunk and writes (max, sum, weighted values) per query; the CTA of a (group, head)
// that finishes last combines the chunks in position order.  A query's arithmetic never depends on how many other queries ride along,
// so a block pass and single-token passes produce identical bits.
#pragma once
#include <limits.h>
#include <math.h>
#include "common.cuh"
#include "tc_common.cuh"

namespace tandem {

constexpr int ATT_CH = 128;       // positions per chunk
constexpr int ATT_NQ = 16;        // most queries per CTA (gamma limit + 1)
constexpr int ATT_THREADS = 256;

struct AttnArgs {
    const void* q; int ldq;              // T [M][ldq]; head h at columns h*DH..
    const void* kcache; const void* vcache;   // [seq][head][t_max][DH]
    const void* k2; const void* v2;            // optional second segment [seq][head][t_max2][DH] holding
    int split, t_max2;                         //   positions >= split (used when k2 != nullptr)
    //   (attn_decode_kernel, ATD_PASS: the second segment is [head][t_max2][DH], indexed by the rows of the pass, and holds the
    //   positions from the group's first row on; split unused)
    void* out; int ldo;                  // T [M][ldo]
    const int* row_seq; const int* row_pos;    // attn_decode_kernel: row_seq may be null, then group g is sequence g and every
    int pos_all;                               //   sequence's first row sits at position pos_all (no row arrays to fill and fetch)
    int wait_first;                            // attn_decode_kernel: 1 = nothing is read before the wait on the preceding kernel
                                               //   (a stand-alone call: whatever precedes it may be writing the keys and values)
    const int* grp_row0; const int* grp_cnt;   // nullable: then group g = rows g*nq .. g*nq+nq-1
    const int* pass_grp; const int* pass_pos;  // ATD_PASS: per group first row | rows << 16 | sequence << 20, and the first row's position
    int nq;
    int units, log_parts;                // ATD_PASS: groups * head groups; 2^log_parts warps (1, 2 or 4) share the keys of each
    int n_heads, t_max;
    int n_kv_heads;                      // key/value heads of the caches; 0 = n_heads.  Query head h reads kv head h / (n_heads / n_kv_heads)
    int* err_flag;                       // attn_decode_kernel: where a bounded wait that ran out records its code (nullable)
    void* out_lo;                        // attn_decode_kernel, optional: `out` is then the bf16 plane of the values and this the bf16
                                         // plane of the remainders (fp32 result = value + remainder), both [M][ldo]
    int heads_per_cta;                   // attn_decode_kernel: query heads of one key/value head served by one CTA (their rows share
                                         // the 16-row tile: heads_per_cta * nq <= 16); 0 = 1.  grid.y = n_heads / heads_per_cta
    float* part_ml;                      // split mode: [M][H][n_chunks_max][2]
    float* part_acc;                     //             [M][H][n_chunks_max][DH]
    int n_chunks_max;
    float scale;
    int* merge_counters;                 // split mode: [groups][H], zero between launches
};

template <typename T, int DH>
constexpr size_t attn_smem_bytes() {
    return (size_t)2 * ATT_CH * (DH + 2 * VecN<T>::N) * sizeof(T) + (size_t)ATT_NQ * DH * sizeof(float) +
           (size_t)ATT_NQ * ATT_CH * sizeof(float) + (size_t)2 * ATT_NQ * sizeof(float);
}

// grid: (chunks, heads, groups) in split mode; (1, heads, groups) in loop mode; block: ATT_THREADS.
// Exact-arithmetic kernel, bound by the latency of its phases on short contexts (a draft step of the fp32 mode has one
// CTA per head): two threads share a key's dot products, and in the value phase ATT_THREADS / DH threads share an output
// element, each summing its own groups of four positions for all queries at once (four values and one 16-byte load of
// probabilities per query and step), before their sums are added in a fixed order.  A block of five queries over 100
// positions of 64-wide heads: 5.3 us, against 11.4 us with one thread per key and a query-by-query walk over the values.
template <typename T, int DH, bool LOOP>
__global__ void __launch_bounds__(ATT_THREADS) attn_kernel(AttnArgs a) {
    constexpr int VN = VecN<T>::N;
    constexpr int LD = DH + 2 * VN;             // padded row: keeps 16-byte alignment, spreads banks
    constexpr int VPR = DH / VN;                // 16-byte vectors per row
    constexpr int PARTS = ATT_THREADS / DH;     // threads that share an output element in the value phase
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int s_last;
    __shared__ float fo[ATT_NQ];   // LOOP: factor of what the earlier chunks contributed, per query
    if (LOOP) pdl_wait();      // queries and keys/values come from earlier kernels
    T* ks = reinterpret_cast<T*>(smem_raw);
    T* vs = ks + ATT_CH * LD;
    float* qs = reinterpret_cast<float*>(vs + ATT_CH * LD);
    float* ss = qs + ATT_NQ * DH;
    float* cm = ss + ATT_NQ * ATT_CH;
    float* cl = cm + ATT_NQ;
    float* red = reinterpret_cast<float*>(smem_raw);   // [PARTS][cnt][DH] where the keys were, once they are done with
    static_assert((size_t)ATT_THREADS * ATT_NQ * sizeof(float) <= (size_t)2 * ATT_CH * LD * sizeof(T), "the parts' sums fit where the keys and values were");

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int g = blockIdx.z, h = blockIdx.y;
    // A decode pass has written its row arrays at least two kernels back: they, and the keys and values of the positions before the
    // block, are fetched ahead of the wait (one query, 32-wide heads, 60 positions: 2.85 -> 2.24 us of the chain; five, 64-wide: 5.0 -> 4.3).
    const int row0 = LOOP && a.grp_row0 ? a.grp_row0[g] : g * a.nq;
    const int cnt = LOOP && a.grp_cnt ? a.grp_cnt[g] : a.nq;
    if (cnt <= 0) return;
    const int b = __ldcg(a.row_seq + row0);
    const int pos_first = __ldcg(a.row_pos + row0);
    const int pos_last = pos_first + cnt - 1;
    const int c_begin = LOOP ? 0 : blockIdx.x;
    const int c_end = LOOP ? pos_last / ATT_CH + 1 : blockIdx.x + 1;
    if (c_begin * ATT_CH > pos_last) {
        if (!LOOP) { pdl_wait(); pdl_launch_dependents(); }
        return;
    }
    const int n_kv = a.n_kv_heads > 0 ? a.n_kv_heads : a.n_heads;
    const int kvh = h / (a.n_heads / n_kv);            // grouped-query attention: several query heads share one key/value head
    const size_t head_base = ((size_t)b * n_kv + kvh) * a.t_max;
    auto fetch = [&](int t0, int t_lo, int t_hi) {     // positions t0 + t_lo .. t0 + t_hi - 1 into the chunk's rows
        for (int i = t_lo * VPR + tid; i < t_hi * VPR; i += ATT_THREADS) {
            const int t = i / VPR, v = i - t * VPR;
            const size_t src = (head_base + t0 + t) * DH + v * VN;
            cp_async16(ks + t * LD + v * VN, static_cast<const T*>(a.kcache) + src);
            cp_async16(vs + t * LD + v * VN, static_cast<const T*>(a.vcache) + src);
        }
    };
    const int n_old = LOOP ? 0 : max(0, min(ATT_CH, pos_first - c_begin * ATT_CH));   // of the (one) chunk's positions
    if (!LOOP) {
        fetch(c_begin * ATT_CH, 0, n_old);
        pdl_wait();
    }
    pdl_launch_dependents();   // the next kernel may start fetching its weights

    const T* qg = static_cast<const T*>(a.q);
    for (int i = tid; i < cnt * DH; i += ATT_THREADS) {
        const int qi = i / DH, el = i - qi * DH;
        qs[qi * DH + el] = to_float(qg[(size_t)(row0 + qi) * a.ldq + h * DH + el]);
    }

    const int e = tid % DH, part = tid / DH;
    float acc[ATT_NQ];
#pragma unroll
    for (int i = 0; i < ATT_NQ; ++i) acc[i] = 0.f;
    if (LOOP && tid < ATT_NQ) { cm[tid] = -INFINITY; cl[tid] = 0.f; }

    for (int c = c_begin; c < c_end; ++c) {
        const int t0 = c * ATT_CH;
        const int nt = min(ATT_CH, pos_last + 1 - t0);
        const int nt4 = (nt + 3) & ~3;
        __syncthreads();   // previous chunk fully consumed (and qs written, first time round)
        fetch(t0, n_old, nt);
        for (int i = nt * VPR + tid; i < nt4 * VPR; i += ATT_THREADS) {   // up to three rows that fill the last group of four: a zero weight times them stays zero
            const int t = i / VPR, v = i - t * VPR;
            *reinterpret_cast<uint4*>(vs + t * LD + v * VN) = make_uint4(0u, 0u, 0u, 0u);
        }
        cp_async_commit();
        cp_async_wait_all();
        __syncthreads();

        // scores: threads 2t and 2t+1 own key t0+t for every query (even / odd 16-byte vectors of the row)
        {
            const int t = tid >> 1, half = tid & 1;
            static_assert(ATT_THREADS == 2 * ATT_CH, "two threads per key");
            float dot[ATT_NQ];
#pragma unroll
            for (int qi = 0; qi < ATT_NQ; ++qi) dot[qi] = 0.f;
            if (t < nt) {
#pragma unroll 2
                for (int v = half; v < VPR; v += 2) {
                    float kv[VN];
                    load_vec(ks + t * LD + v * VN, kv);
#pragma unroll
                    for (int qi = 0; qi < ATT_NQ; ++qi) {
                        if (qi >= cnt) break;
#pragma unroll
                        for (int i = 0; i < VN; i += 4) {
                            const float4 q4 = *reinterpret_cast<const float4*>(qs + qi * DH + v * VN + i);
                            dot[qi] = fmaf(q4.x, kv[i], dot[qi]); dot[qi] = fmaf(q4.y, kv[i + 1], dot[qi]);
                            dot[qi] = fmaf(q4.z, kv[i + 2], dot[qi]); dot[qi] = fmaf(q4.w, kv[i + 3], dot[qi]);
                        }
                    }
                }
            }
#pragma unroll
            for (int qi = 0; qi < ATT_NQ; ++qi) {
                if (qi >= cnt) break;
                const float d = dot[qi] + __shfl_xor_sync(0xffffffffu, dot[qi], 1);
                if (half == 0 && t < nt4) ss[qi * ATT_CH + t] = (t < nt && t0 + t <= pos_first + qi) ? d * a.scale : -INFINITY;
            }
        }
        __syncthreads();

        // per query: maximum (LOOP: of everything so far), exponentials, sum
        for (int qi = warp; qi < cnt; qi += ATT_THREADS / 32) {
            float m = LOOP ? cm[qi] : -INFINITY;
            const float m_old = m;
            for (int t = lane; t < nt; t += 32) m = fmaxf(m, ss[qi * ATT_CH + t]);
            m = warp_max(m);
            float l = 0.f;
            for (int t = lane; t < nt4; t += 32) {
                const float p = m > -INFINITY ? expf(ss[qi * ATT_CH + t] - m) : 0.f;
                ss[qi * ATT_CH + t] = p;
                l += p;
            }
            l = warp_sum(l);
            __syncwarp();
            if (lane == 0) {
                if (LOOP) {
                    const float f = m_old > -INFINITY ? expf(m_old - m) : 0.f;
                    fo[qi] = f;
                    l = fmaf(cl[qi], f, l);
                }
                cm[qi] = m;
                cl[qi] = l;
            }
        }
        __syncthreads();

        // weighted values: this thread's groups of four positions, element e, every query
        if (LOOP) {
#pragma unroll
            for (int qi = 0; qi < ATT_NQ; ++qi) {
                if (qi >= cnt) break;
                acc[qi] *= fo[qi];
            }
        }
        for (int t = 4 * part; t < nt4; t += 4 * PARTS) {
            float v[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) v[i] = to_float(vs[(t + i) * LD + e]);
#pragma unroll
            for (int qi = 0; qi < ATT_NQ; ++qi) {
                if (qi >= cnt) break;
                const float4 p = *reinterpret_cast<const float4*>(ss + qi * ATT_CH + t);
                acc[qi] = fmaf(p.x, v[0], acc[qi]); acc[qi] = fmaf(p.y, v[1], acc[qi]);
                acc[qi] = fmaf(p.z, v[2], acc[qi]); acc[qi] = fmaf(p.w, v[3], acc[qi]);
            }
        }
    }
    // the parts' sums of every (query, element), added in part order
    __syncthreads();
#pragma unroll
    for (int qi = 0; qi < ATT_NQ; ++qi) {
        if (qi >= cnt) break;
        red[((size_t)part * cnt + qi) * DH + e] = acc[qi];
    }
    __syncthreads();
    T* og = static_cast<T*>(a.out);
    const int n_active = pos_last / ATT_CH + 1;        // CTAs of this (group, head) in split mode
    for (int i = tid; i < cnt * DH; i += ATT_THREADS) {
        const int qi = i / DH, el = i - qi * DH;
        float o = 0.f;
#pragma unroll
        for (int p = 0; p < PARTS; ++p) o += red[(size_t)p * cnt * DH + i];
        if (LOOP || n_active == 1) {
            og[(size_t)(row0 + qi) * a.ldo + h * DH + el] = from_float<T>(o / cl[qi]);
        } else if (cm[qi] > -INFINITY) {
            const size_t p = ((size_t)(row0 + qi) * a.n_heads + h) * a.n_chunks_max + c_begin;
            a.part_acc[p * DH + el] = o;
            if (el == 0) { a.part_ml[p * 2] = cm[qi]; a.part_ml[p * 2 + 1] = cl[qi]; }
        }
    }
    if (!LOOP && n_active > 1) {
        // The CTA that finishes last for this (group, head) merges every query's chunks in position order.
        __threadfence();
        __syncthreads();
        if (tid == 0) {
            const int active = min((int)gridDim.x, n_active);   // CTAs that got this far
            int* counter = a.merge_counters + (size_t)g * a.n_heads + h;
            const int t = atomicAdd(counter, 1);
            s_last = (t == active - 1);
            if (t == active - 1) *counter = 0;   // ready for the next launch
        }
        __syncthreads();
        if (!s_last) return;
        __threadfence();
        for (int i = tid; i < cnt * DH; i += ATT_THREADS) {
            const int qi = i / DH, el = i - qi * DH;
            const int nc = (pos_first + qi) / ATT_CH + 1;
            const size_t base = ((size_t)(row0 + qi) * a.n_heads + h) * a.n_chunks_max;
            float mx = -INFINITY;
#pragma unroll 8
            for (int c = 0; c < nc; ++c) mx = fmaxf(mx, __ldcg(a.part_ml + (base + c) * 2));
            float l = 0.f, o = 0.f;
#pragma unroll 4
            for (int c = 0; c < nc; ++c) {
                const float2 ml = __ldcg(reinterpret_cast<const float2*>(a.part_ml + (base + c) * 2));
                const float pa = __ldcg(a.part_acc + (base + c) * DH + el);
                const float f = expf(ml.x - mx);
                l = fmaf(ml.y, f, l);
                o = fmaf(pa, f, o);
            }
            og[(size_t)(row0 + qi) * a.ldo + h * DH + el] = from_float<T>(o / l);
        }
    }
}

// ---------------------------------------------------------------------------------------------------
// Decode attention, bf16, built for short dependent chains and for streaming: a cluster of CL CTAs (1, 2, 4 or 8,
// fixed per launch configuration) serves one (sequence, head).  CTA `rank` takes the 128-position chunks rank,
// rank + CL, ... (anchored at absolute position 0); inside a chunk warp w owns positions 16w .. 16w+15.  Every warp
// runs on its own: it fetches its rows through a private cp.async ring, keeps the online-softmax state of all the
// block's queries (up to 16) in registers and never waits for another warp until the end, where the CTA folds its
// warps' states in warp order, sends the result to the CTA that finishes the query (remote shared-memory stores),
// and that CTA merges the CL states in rank order.  No global scratch, no second kernel.
//
// The two small products of a 16-position tile run on the tensor cores as warp-level m16n8k16 MMAs, transposed: S^T = K Q^T with
// the 16 keys as the MMA's rows and eight queries as its columns, O^T += V^T P^T with 16 elements of the head as rows.  (With
// the queries as the 16 rows a block of up to eight of them left half of every MMA to absent rows: 32 sequences x 16 heads x 64
// x 8194 positions took 187-190 us a call, now 169 us, 6.3 TB/s.)  K and V fragments come straight from the ring
// with ldmatrix (V transposed on the way), the queries stay in registers, the softmax works on the accumulator fragments (a
// query's 16 scores sit in eight lanes), and the probabilities become the second product's B fragments by an 8 x 8 register
// transpose, each as two bf16 numbers (value and remainder).  A query's column depends on its own query only, so a block
// pass and a one-row pass give the same bits.  The probabilities use the fast exponential
// (2^x hardware approximation), well inside the bf16 tolerance.
// ---------------------------------------------------------------------------------------------------
constexpr int ATD_THREADS = 256;
constexpr int ATD_WARPS = ATD_THREADS / 32;
constexpr int ATD_ERR_EXCHANGE = 5;                                 // error code: the wait for the cluster's states gave up
constexpr int ATD_CLUSTER = 8;                                      // largest cluster; launches use 1, 2, 4 or 8
constexpr int ATD_SLOTS = ATT_NQ;                                   // inbox states per CTA: cluster size x queries it finishes <= 16
constexpr int ATD_WROWS = ATT_CH / ATD_WARPS;                       // positions of a chunk per warp (16)
static_assert(ATD_WROWS == 16, "one m16n8k16 tile per warp and chunk");

template <int DH> struct AtdCfg {
    static constexpr int TPK = DH / 8;               // 16-byte units per key
    static constexpr int STAGES = DH <= 64 ? 3 : 2;
    static constexpr int TILE_ELEMS = ATD_WROWS * DH;   // a warp's keys (or values) of one chunk
    static constexpr int STAGE_ELEMS = 2 * TILE_ELEMS;
    static constexpr int UNITS = ATD_WROWS * TPK / 32;  // 16-byte units per lane per tile
    static constexpr int KSTEPS = DH / 16;           // MMAs along the head dimension for S, 16-row tiles of O^T
};
template <int DH>
constexpr size_t attn_decode_smem_bytes() {
    // the warps' rings (reused for the warps' final states) + the inbox of states sent by the cluster's CTAs
    return (size_t)ATD_WARPS * AtdCfg<DH>::STAGES * AtdCfg<DH>::STAGE_ELEMS * sizeof(bf16) + sizeof(float) * (size_t)ATD_SLOTS * (DH + 2);
}
static_assert((size_t)ATT_NQ * (128 + 2) * sizeof(float) <= (size_t)AtdCfg<128>::STAGES * AtdCfg<128>::STAGE_ELEMS * sizeof(bf16) &&
              (size_t)ATT_NQ * (64 + 2) * sizeof(float) <= (size_t)AtdCfg<64>::STAGES * AtdCfg<64>::STAGE_ELEMS * sizeof(bf16) &&
              (size_t)ATT_NQ * (32 + 2) * sizeof(float) <= (size_t)AtdCfg<32>::STAGES * AtdCfg<32>::STAGE_ELEMS * sizeof(bf16),
              "a warp's states fit in its ring");

// Where the 16-byte unit u of ring row r lives within the row: XOR-swizzled so that the eight row addresses of
// one ldmatrix fall into different banks (rows are DH * 2 bytes apart).
template <int DH>
__device__ __forceinline__ int atd_swz(int r, int u) { return u ^ (DH >= 64 ? (r & 7) : ((r >> 1) & 3)); }

__device__ __forceinline__ void ldmatrix_x4(uint32_t addr, uint32_t (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t addr, uint32_t (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
// D (16x8, fp32) += A (16x16, bf16, row) * B (16x8, bf16, col)
__device__ __forceinline__ void mma_bf16_16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// Transpose of an 8 x 8 matrix of 16-bit elements held as a fragment.
__device__ __forceinline__ uint32_t movmatrix_trans(uint32_t a) {
    uint32_t d;
    asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(d) : "r"(a));
    return d;
}
__device__ __forceinline__ uint32_t atd_pack_bf16x2(float lo, float hi) {
    const __nv_bfloat162 p = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&p);
}

// grid: (CL, heads, sequences or groups) with the CL CTAs along x forming one cluster, CL in {1, 2, 4, 8}; block: ATD_THREADS.
// NT: groups of eight query columns in use (1 up to eight rows per CTA, 2 up to 16).
// MODE: ATD_CLUSTERED, CL in {2, 4, 8}; ATD_ALONE, CL = 1, results straight from the fold of the warps' states (32 x 16 x 64 x 8194:
// 171 -> 165 us, without the trip through the inbox); ATD_PASS, a teacher-forced pass: groups of unequal length, the second segment of a block's own keys,
// and a warp on its own per group and head, since there are hundreds of them over short contexts, or two or four that deal its tiles and merge
// their states through shared memory where fewer units leave the chip a long chain each (grid: warps in all / 8; one warp each: 49 groups x 16
// heads x 64 over up to 257 positions: 25 -> 20 us under ncu, 193 blocks of four rows x 8 heads 26 -> 17 us).  (The same code with these choices made at run time costs the stand-alone call on 1 x 16 x 64 x 1028 3.5 %: 5.58 -> 5.78 us.)
enum { ATD_CLUSTERED = 0, ATD_ALONE = 1, ATD_PASS = 2 };
template <int DH, int NT, int MODE>
__global__ void __launch_bounds__(ATD_THREADS) attn_decode_kernel(AttnArgs a) {
    using C = AtdCfg<DH>;
    constexpr int NW = ATD_WARPS;
    constexpr int SW = DH + 2;                     // a state: DH output sums, the running maximum, the running sum
    extern __shared__ __align__(128) unsigned char smem_raw[];
    bf16* ring_all = reinterpret_cast<bf16*>(smem_raw);
    constexpr int WST = C::STAGES * C::STAGE_ELEMS / 2;      // floats between two warps' states: each where the warp's ring was
    float* wst = reinterpret_cast<float*>(smem_raw);         // [NW][16][SW], after the main loop
    float* inbox = reinterpret_cast<float*>(ring_all + (size_t)NW * C::STAGES * C::STAGE_ELEMS);   // [CL][QPC][SW]

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int rank = MODE == ATD_PASS ? 0 : blockIdx.x;
    // Grouped-query attention: the tile's 16 rows hold the block's queries of `gpc` query heads that share one
    // key/value head (row = head * nq + block row), so their keys and values are streamed once for all of them.
    const int gpc = a.heads_per_cta > 0 ? a.heads_per_cta : 1;
    const int log_parts = MODE == ATD_PASS ? a.log_parts : 0, part = warp & ((1 << log_parts) - 1);   // ATD_PASS: this warp's share of its unit's tiles
    const int head_groups = a.n_heads / gpc, unit = MODE == ATD_PASS ? (blockIdx.x * NW + warp) >> log_parts : 0;
    if (MODE == ATD_PASS && unit >= a.units) return;
    const int g = MODE == ATD_PASS ? unit / head_groups : blockIdx.z;
    const int h = (MODE == ATD_PASS ? unit - g * head_groups : blockIdx.y) * gpc;   // first query head of this CTA (warp)
    const int CL = MODE == ATD_CLUSTERED ? gridDim.x : 1;   // cluster size
    const int log_cl = MODE == ATD_CLUSTERED ? __ffs(CL) - 1 : 0;   // (a division by a number known at run time costs the chain about 0.05 us)
    const int QPC = ATT_NQ >> log_cl;              // queries a CTA finishes at most
    __shared__ __align__(8) uint64_t s_inbox_bar;  // counts the bytes of the states sent to this CTA by the cluster's CTAs
    if (CL > 1 && tid == 0) { mbar_init(smem_u32(&s_inbox_bar), 1); mbar_init_fence(); }
    if (CL > 1) cluster_arrive_relaxed();          // opening handshake: waited for just before the first remote store
    bf16* ring = ring_all + (size_t)warp * C::STAGES * C::STAGE_ELEMS;
    const uint32_t ring_s = smem_u32(ring);
    // The row arrays were written at the start of the pass, at least two kernels back in the stream, so they may be
    // read before the wait below: a kernel lets its successor start only after its own wait has returned, that is
    // after its predecessor has finished, hence everything older than the immediate predecessor is complete.
    const int n_kv = a.n_kv_heads > 0 ? a.n_kv_heads : a.n_heads;
    const int kvh = n_kv == a.n_heads ? h : h / (a.n_heads / n_kv);   // grouped-query attention: several query heads share one key/value head
    if (a.wait_first) {   // (a successor has nothing to fetch that would be in this kernel's way)
        pdl_wait();
        pdl_launch_dependents();
    }
    const int pg = MODE == ATD_PASS ? __ldcg(a.pass_grp + g) : 0;
    const int nq = MODE == ATD_PASS ? (pg >> 16) & 15 : a.nq, row0 = MODE == ATD_PASS ? pg & 0xffff : g * nq;
    const int cnt = gpc * nq;                      // rows of the tile in use
    const int b = MODE == ATD_PASS ? pg >> 20 : (a.row_seq ? __ldcg(a.row_seq + row0) : g);          // from L2: nothing an earlier kernel on this SM may have cached
    const int pos_first = MODE == ATD_PASS ? __ldcg(a.pass_pos + g) : (a.row_seq ? __ldcg(a.row_pos + row0) : a.pos_all);
    const int pos_last = pos_first + nq - 1;
    const int n_chunks = pos_last / ATT_CH + 1;
    const int n_mine = MODE == ATD_PASS ? (pos_last / ATD_WROWS + (1 << log_parts) - part) >> log_parts : rank < n_chunks ? (n_chunks - rank + CL - 1) >> log_cl : 0;
    const size_t head_base = ((size_t)b * n_kv + kvh) * a.t_max;
    const size_t head_base2 = MODE == ATD_PASS ? (size_t)kvh * a.t_max2 + row0 - pos_first : ((size_t)b * n_kv + kvh) * a.t_max2;   // (ATD_PASS: to be added to a position)
    const int split = a.k2 ? (MODE == ATD_PASS ? pos_first : a.split) : INT_MAX;
    const int base2 = MODE == ATD_PASS ? 0 : split;    // position of the second segment's first key

    // this warp's rows of its CTA's it-th chunk into stage it % STAGES.  Lane L moves unit L % TPK of rows
    // L / TPK + (32 / TPK) * u; a tile that lies wholly in one cache and before the last query (all but a
    // boundary tile or two) takes the short way: one base address, constant steps.
    constexpr int RSTEP = 32 / C::TPK;             // rows between a lane's consecutive units
    const int i_row = lane / C::TPK, i_unit = lane - i_row * C::TPK;
    auto tile_start = [&](int it) { return MODE == ATD_PASS ? ((it << log_parts) + part) * ATD_WROWS : (rank + it * CL) * ATT_CH + warp * ATD_WROWS; };
    auto issue = [&](int it) {
        const int t0 = tile_start(it);
        bf16* ks = ring + (size_t)(it % C::STAGES) * C::STAGE_ELEMS;
        bf16* vs = ks + C::TILE_ELEMS;
        const bool first = t0 + ATD_WROWS <= split, second = t0 >= split;
        if (t0 + ATD_WROWS - 1 <= pos_last && (first || second)) {
            const size_t src = first ? (head_base + t0 + i_row) * DH : (head_base2 + (t0 - base2) + i_row) * DH;
            const bf16* kg = static_cast<const bf16*>(first ? a.kcache : a.k2) + src + i_unit * 8;
            const bf16* vg = static_cast<const bf16*>(first ? a.vcache : a.v2) + src + i_unit * 8;
#pragma unroll
            for (int u = 0; u < C::UNITS; ++u) {
                const int t = i_row + RSTEP * u;
                const int dst = t * DH + atd_swz<DH>(t, i_unit) * 8;
                cp_async16(ks + dst, kg + (size_t)u * RSTEP * DH);
                cp_async16(vs + dst, vg + (size_t)u * RSTEP * DH);
            }
            return;
        }
#pragma unroll
        for (int u = 0; u < C::UNITS; ++u) {
            const int t = i_row + RSTEP * u, v = i_unit;
            const int ta = t0 + t;
            const int dst = t * DH + atd_swz<DH>(t, v) * 8;
            if (ta <= pos_last) {
                const bf16 *kg, *vg;
                if (ta < split) {
                    kg = static_cast<const bf16*>(a.kcache) + (head_base + ta) * DH;
                    vg = static_cast<const bf16*>(a.vcache) + (head_base + ta) * DH;
                } else {
                    kg = static_cast<const bf16*>(a.k2) + (head_base2 + (ta - base2)) * DH;
                    vg = static_cast<const bf16*>(a.v2) + (head_base2 + (ta - base2)) * DH;
                }
                cp_async16(ks + dst, kg + v * 8);
                cp_async16(vs + dst, vg + v * 8);
            } else {   // past the last query: zeros, so that a zero weight times them stays zero
                *reinterpret_cast<uint4*>(ks + dst) = make_uint4(0u, 0u, 0u, 0u);
                *reinterpret_cast<uint4*>(vs + dst) = make_uint4(0u, 0u, 0u, 0u);
            }
        }
    };
    // Tiles that end before the block's first position hold committed keys and values from earlier iterations (or
    // earlier steps of this one): they are fetched before the wait; what the predecessor may have written, after it.
    int pre = 0;
#pragma unroll 1   // (less code to fetch)
    for (int it = 0; it < C::STAGES - 1; ++it) {
        if (it == pre && it < n_mine && tile_start(it) + ATD_WROWS <= pos_first) {
            issue(it);
            cp_async_commit();
            ++pre;
        }
    }
    pdl_wait();   // queries and the newest keys/values come from the kernel before this one
#pragma unroll 1
    for (int it = 0; it < C::STAGES - 1; ++it) {
        if (it >= pre) {
            if (it < n_mine) issue(it);
            cp_async_commit();
        }
    }

    // The queries as B fragments: this lane holds query 8 nt + lane/4, elements 2*(lane%4) (+1) (+8) of each 16-wide step along
    // the head dimension; queries beyond cnt are absent (zero, never stored)
    const int kc = 2 * (lane & 3);
    uint32_t qf[NT][C::KSTEPS][2];
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
        const int rr = nt * 8 + (lane >> 2);
        const int hq = gpc > 1 && rr < cnt ? rr / nq : 0, ib = rr < cnt ? rr - hq * nq : 0;      // query head within the CTA, block row
        const bf16* qp = static_cast<const bf16*>(a.q) + (size_t)(row0 + ib) * a.ldq + (h + hq) * DH + kc;
#pragma unroll
        for (int ks = 0; ks < C::KSTEPS; ++ks) {
            qf[nt][ks][0] = rr < cnt ? *reinterpret_cast<const uint32_t*>(qp + ks * 16) : 0u;
            qf[nt][ks][1] = rr < cnt ? *reinterpret_cast<const uint32_t*>(qp + ks * 16 + 8) : 0u;
        }
    }
    // Accumulators: this lane's columns are queries 8 nt + kc + e, e = 0, 1; last position that each of them attends (-1: absent)
    int q_last[NT][2];
    float o[NT][C::KSTEPS][4];
    float m[NT][2], l[NT][2];                            // l: this lane's keys only until the end
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int rr = nt * 8 + kc + e;
            q_last[nt][e] = rr < cnt ? pos_first + (gpc > 1 ? rr % nq : rr) : -1;
            m[nt][e] = -INFINITY;
            l[nt][e] = 0.f;
        }
#pragma unroll
        for (int mt = 0; mt < C::KSTEPS; ++mt) { o[nt][mt][0] = 0.f; o[nt][mt][1] = 0.f; o[nt][mt][2] = 0.f; o[nt][mt][3] = 0.f; }
    }

    // ldmatrix row addresses of this lane (matrix lane/8, row lane%8), relative to the K (or V) tile of a stage
    const int lm_m = lane >> 3, lm_r = lane & 7;
    const uint32_t k_row = (uint32_t)((((lm_m & 1) << 3) + lm_r) * DH * 2);     // K: key = 8 * (matrix & 1) + row, unit = 2 * ks + matrix / 2
    const uint32_t v_row = (uint32_t)((((lm_m >> 1) << 3) + lm_r) * DH * 2);    // V: key = 8 * (matrix / 2) + row, unit = 2 * mt + matrix & 1
    const int k_sw = atd_swz<DH>(((lm_m & 1) << 3) + lm_r, 0), v_sw = atd_swz<DH>(((lm_m >> 1) << 3) + lm_r, 0);

    for (int it = 0; it < n_mine; ++it) {
        if (it + C::STAGES - 1 < n_mine) issue(it + C::STAGES - 1);
        cp_async_commit();
        asm volatile("cp.async.wait_group %0;" ::"n"(C::STAGES - 1) : "memory");
        __syncwarp();
        const int t0 = tile_start(it);
        const uint32_t ks_s = ring_s + (uint32_t)((it % C::STAGES) * C::STAGE_ELEMS * 2);
        const uint32_t vs_s = ks_s + (uint32_t)(C::TILE_ELEMS * 2);

        // S^T = K Q^T for the tile's 16 keys; even and odd steps in two accumulators (half the dependent chain)
        float sc[NT][2][4];
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
            for (int b2 = 0; b2 < 2; ++b2) { sc[nt][b2][0] = 0.f; sc[nt][b2][1] = 0.f; sc[nt][b2][2] = 0.f; sc[nt][b2][3] = 0.f; }
#pragma unroll
        for (int ks = 0; ks < C::KSTEPS; ++ks) {
            uint32_t kf[4];
            ldmatrix_x4(ks_s + k_row + (uint32_t)(((ks * 2 + (lm_m >> 1)) ^ k_sw) << 4), kf);
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) mma_bf16_16816(sc[nt][ks & 1], kf, qf[nt][ks][0], qf[nt][ks][1]);
        }
        // scale, causal mask, running maxima, probabilities: element (hh, e) is key t0 + lane/4 + 8 hh, query 8 nt + kc + e
        uint32_t pf[NT][2], pr[NT][2];
        float f[NT][2];
        bool moved = false;
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
            float p[2][2];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int key = t0 + (lane >> 2);
                float x0 = (sc[nt][0][e] + sc[nt][1][e]) * a.scale, x1 = (sc[nt][0][2 + e] + sc[nt][1][2 + e]) * a.scale;
                x0 = key <= q_last[nt][e] ? x0 : -INFINITY;
                x1 = key + 8 <= q_last[nt][e] ? x1 : -INFINITY;
                float mc = fmaxf(x0, x1);
                mc = fmaxf(mc, __shfl_xor_sync(0xffffffffu, mc, 4));
                mc = fmaxf(mc, __shfl_xor_sync(0xffffffffu, mc, 8));
                mc = fmaxf(mc, __shfl_xor_sync(0xffffffffu, mc, 16));
                const float mn = fmaxf(m[nt][e], mc);
                f[nt][e] = m[nt][e] > -INFINITY ? __expf(m[nt][e] - mn) : (mn > -INFINITY ? 0.f : 1.f);
                m[nt][e] = mn;
                moved = moved || f[nt][e] != 1.f;
                p[0][e] = mn > -INFINITY ? __expf(x0 - mn) : 0.f;
                p[1][e] = mn > -INFINITY ? __expf(x1 - mn) : 0.f;
                l[nt][e] = l[nt][e] * f[nt][e] + (p[0][e] + p[1][e]);
            }
            // each probability as the sum of two bf16 numbers (the rounded value and the rounded remainder): the second product
            // then sees them to about 16 significant bits instead of 8, at the price of a second MMA
#pragma unroll
            for (int hh = 0; hh < 2; ++hh) {
                const __nv_bfloat162 hi = __floats2bfloat162_rn(p[hh][0], p[hh][1]);
                pf[nt][hh] = movmatrix_trans(*reinterpret_cast<const uint32_t*>(&hi));
                pr[nt][hh] = movmatrix_trans(atd_pack_bf16x2(p[hh][0] - __low2float(hi), p[hh][1] - __high2float(hi)));
            }
        }
        // O^T = O^T * f + V^T P^T; the rescaling is skipped while no query of the warp has a new maximum (a factor of exactly 1)
        const bool rescale = __any_sync(0xffffffffu, moved);
#pragma unroll
        for (int mt = 0; mt < C::KSTEPS; ++mt) {
            uint32_t vf[4];
            ldmatrix_x4_trans(vs_s + v_row + (uint32_t)(((2 * mt + (lm_m & 1)) ^ v_sw) << 4), vf);
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) {
                float (&acc)[4] = o[nt][mt];
                if (rescale) { acc[0] *= f[nt][0]; acc[1] *= f[nt][1]; acc[2] *= f[nt][0]; acc[3] *= f[nt][1]; }
                mma_bf16_16816(acc, vf, pf[nt][0], pf[nt][1]);
                mma_bf16_16816(acc, vf, pr[nt][0], pr[nt][1]);
            }
        }
        __syncwarp();   // the stage may be refilled by this warp's next issue
    }
    pdl_launch_dependents();   // the successor starts behind the merge, not behind this kernel's loads (measured: a little faster)
    auto store = [&](int qi, int e, float res) {   // tile row qi = query head hq of this CTA (warp), block row qi - hq * nq
        const int hq = gpc > 1 ? qi / nq : 0;
        const size_t oi = (size_t)(row0 + qi - hq * nq) * a.ldo + (h + hq) * DH + e;
        if (a.out_lo) {
            const bf16 hi = __float2bfloat16_rn(res);
            static_cast<bf16*>(a.out)[oi] = hi;
            static_cast<bf16*>(a.out_lo)[oi] = __float2bfloat16_rn(res - __bfloat162float(hi));
        } else {
            static_cast<bf16*>(a.out)[oi] = __float2bfloat16_rn(res);
        }
    };
    if (MODE == ATD_PASS && log_parts == 0) {   // the warp has met all keys: results straight from its registers
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                float lr = l[nt][e];
                lr += __shfl_xor_sync(0xffffffffu, lr, 4);
                lr += __shfl_xor_sync(0xffffffffu, lr, 8);
                lr += __shfl_xor_sync(0xffffffffu, lr, 16);
                const int rr = nt * 8 + kc + e;
                if (rr >= cnt) continue;
#pragma unroll
                for (int mt = 0; mt < C::KSTEPS; ++mt) {
                    store(rr, mt * 16 + (lane >> 2), o[nt][mt][e] / lr);
                    store(rr, mt * 16 + 8 + (lane >> 2), o[nt][mt][2 + e] / lr);
                }
            }
        return;
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncwarp();   // this warp is done with its ring: its states go there
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            float lr = l[nt][e];                       // a query's sum: add the eight lanes that share its column
            lr += __shfl_xor_sync(0xffffffffu, lr, 4);
            lr += __shfl_xor_sync(0xffffffffu, lr, 8);
            lr += __shfl_xor_sync(0xffffffffu, lr, 16);
            const int rr = nt * 8 + kc + e;
            if (rr >= cnt) continue;
            float* st = wst + warp * WST + rr * SW + (lane >> 2);
#pragma unroll
            for (int mt = 0; mt < C::KSTEPS; ++mt) { st[mt * 16] = o[nt][mt][e]; st[mt * 16 + 8] = o[nt][mt][2 + e]; }
            if (lane < 4) { st[DH] = m[nt][e]; st[DH + 1] = lr; }
        }
    if constexpr (MODE == ATD_PASS) {   // the unit's warps fold their states (all of them are here: units end with their last warp)
        asm volatile("bar.sync %0, %1;" ::"r"(1 + (warp >> log_parts)), "r"(32 << log_parts) : "memory");
        const float* st = wst + (warp - part) * WST;
        for (int i = part * 32 + lane; i < cnt * DH; i += 32 << log_parts) {
            const int qa = i / DH, e = i - qa * DH;
            float mx = -INFINITY, val = 0.f, lsum = 0.f;
            for (int w = 0; w < 1 << log_parts; ++w) mx = fmaxf(mx, st[w * WST + qa * SW + DH]);
            for (int w = 0; w < 1 << log_parts; ++w) {
                const float* sw = st + w * WST + qa * SW;
                const float f = sw[DH] > -INFINITY ? __expf(sw[DH] - mx) : 0.f;
                val = fmaf(sw[e], f, val);
                lsum = fmaf(sw[DH + 1], f, lsum);
            }
            store(qa, e, val / lsum);
        }
        return;
    }
    __syncthreads();
    // fold the warps' states in warp order and send the CTA's state of query qa to CTA qa & (CL - 1)
    if (CL > 1) cluster_wait();   // closes the opening handshake: every CTA of the cluster is running
    // One thread per (query, output element); the thread of element 0 also folds the query's running sum and sends its
    // maximum (with 4 queries of 64 elements that is one pass over the block's 256 threads).  A CTA on its own has the result
    // right here (every thread folds the sum then).
    for (int i = tid; i < cnt * DH; i += ATD_THREADS) {
        const int qa = i / DH, e = i - qa * DH;
        float mx = -INFINITY;
#pragma unroll
        for (int w = 0; w < NW; ++w) mx = fmaxf(mx, wst[w * WST + qa * SW + DH]);
        float val = 0.f, lsum = 0.f;
#pragma unroll
        for (int w = 0; w < NW; ++w) {
            const float* st = wst + w * WST + qa * SW;
            const float f = st[DH] > -INFINITY ? __expf(st[DH] - mx) : 0.f;
            val = fmaf(st[e], f, val);
            if (e == 0 || MODE == ATD_ALONE) lsum = fmaf(st[DH + 1], f, lsum);
        }
        if (MODE == ATD_ALONE) { store(qa, e, val / lsum); continue; }
        float* slot = inbox + ((size_t)rank * QPC + (qa >> log_cl)) * SW;
        st_async_dsmem_f32(smem_u32(slot + e), smem_u32(&s_inbox_bar), qa & (CL - 1), val);   // counted on the receiver's barrier
        if (e == 0) {
            st_async_dsmem_f32(smem_u32(slot + DH), smem_u32(&s_inbox_bar), qa & (CL - 1), mx);
            st_async_dsmem_f32(smem_u32(slot + DH + 1), smem_u32(&s_inbox_bar), qa & (CL - 1), lsum);
        }
    }
    if (MODE == ATD_ALONE) return;
    {
        // This CTA finishes queries rank, rank + CL, ...: it waits (bounded) until every CTA's state of each of them
        // has arrived.  No cluster-wide barrier: a CTA without queries of its own leaves right after sending.
        const int n_fin = rank < cnt ? (cnt - rank + CL - 1) >> log_cl : 0;
        if (n_fin > 0) {
            if (tid == 0) mbar_arrive_expect_tx(smem_u32(&s_inbox_bar), (uint32_t)(CL * n_fin * SW * 4));
            if (!mbar_wait(smem_u32(&s_inbox_bar), 0) && a.err_flag) atomicExch(a.err_flag, ATD_ERR_EXCHANGE);
        }
    }
    for (int u = 0; u < QPC; ++u) {
        const int qi = rank + u * CL;
        if (qi < cnt && tid < DH) {
            // the CTAs' states in rank order; all loads and exponentials first, then the two sums (same order as a plain loop)
            float mr[ATD_CLUSTER], lr[ATD_CLUSTER], orr[ATD_CLUSTER];
            float mx = -INFINITY;
#pragma unroll
            for (int r = 0; r < ATD_CLUSTER; ++r) {
                const float* st = inbox + ((size_t)r * QPC + u) * SW;
                mr[r] = r < CL ? st[DH] : -INFINITY;
                lr[r] = r < CL ? st[DH + 1] : 0.f;
                orr[r] = r < CL ? st[tid] : 0.f;
                mx = fmaxf(mx, mr[r]);
            }
            float l = 0.f, ov = 0.f;
#pragma unroll
            for (int r = 0; r < ATD_CLUSTER; ++r) {
                if (r < CL) {
                    const float f = mr[r] > -INFINITY ? __expf(mr[r] - mx) : 0.f;
                    l = fmaf(lr[r], f, l);
                    ov = fmaf(orr[r], f, ov);
                }
            }
            store(qi, tid, ov / l);
        }
    }
}

}  // namespace tandem
