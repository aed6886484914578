// Causal prompt attention (Eq. 1 over the prompt) on the tcgen05 tensor cores, bf16, head size 64 or 128.
//
// One CTA serves one head and up to 256 consecutive queries of one sequence, as two tiles of 128.  The context is swept in
// chunks of KC keys (128 at 128-wide heads, else 64) anchored at position 0, each tile up to its own last query; per tile and chunk:
//     S  = Q K^T        M = 128 queries on the TMEM lanes, N = KC keys, K = head size; one or two S buffers per tile, 128 columns
//     P  = softmax step thread i of the tile's four warps owns query i: reads its row of S from TMEM, masks keys after its
//                       position, writes bf16 probabilities back into TMEM where S was
//     O += P V          M = 128 queries, N = head size, K = KC keys; P is the A operand straight from TMEM, V is used as it
//                       lies in the cache ([key][element], i.e. MN-major for the B operand), O accumulates in TMEM
// The S that takes the place of a chunk's P is issued right behind the product that reads P (a CTA's products run in issue
// order), and one tile's softmax runs beside the other's products.  TMEM holds S / P and O of both tiles: all 512 columns.
// Nothing but Q, K and V goes through shared memory, and a chunk of K and V serves 256 queries.
// What bounds it (128-wide heads): per 128 queries and keys 128 x 128 exponentials, products whose A operand comes from TMEM for
// half of them, and the softmax warps' own chain from S to P with its barriers; under ncu the tensor pipe and the
// exponential unit are both 63 % busy.  Chunks of 128 keys halve the chain's fixed parts and the products' share of reading Q;
// with 64-wide heads, whose prompts are short, the coarser diagonal costs as much.  The longest tiles start first (a causal
// tile costs what its position says).  8191 rows x 32 heads x 128: 448 us = 1228 TFLOP/s at full clocks, 488 us with chunks of
// 64 keys in two buffers.  Taking the chunk's maximum beside the exponentials instead of before them was slower (470 us).
// The running maximum is lazy: probabilities are taken relative to a reference m that moves only when a chunk's
// maximum exceeds it by more than ATC_LAZY (so they stay below e^ATC_LAZY); only then is O, in TMEM, rescaled
// (tcgen05.ld, multiply, tcgen05.st) - rare after the first chunks.  The row sum adds the fp32 probabilities (their
// bf16 roundings, which the tensor core multiplies with V, differ from them by 2^-9 each with random signs).
// Warps 0-3 / 4-7: softmax and epilogue of tile 0 / 1; warp 8 streams K and V (256 keys each in flight) by TMA; warp 9 allocates
// TMEM and issues the MMAs.  Every wait is bounded.
#pragma once
#include "common.cuh"
#include "gemm_tc.cuh"
#include "tc_common.cuh"

namespace tandem {

struct AttnTcArgs {
    void* out; int ldo;                   // bf16 [M][ldo]; head h at columns h*DH..
    const int* row_seq; const int* row_pos;
    const int* grp_row0; const int* grp_cnt;
    int n_heads, t_max;
    int n_kv_heads;                       // key/value heads of the cache (<= n_heads, divides it)
    float scale;
    int* err_flag;
};

constexpr int ATC_THREADS = 320;
constexpr int ATC_TILE = 128;             // queries per tile
constexpr int ATC_Q = 2 * ATC_TILE;       // queries per CTA
constexpr int ATC_SUB = 128 * 128;        // bytes of one 128-row x 64-element bf16 sub-tile (queries)
constexpr float ATC_LAZY = 5.0f;          // how far a chunk's maximum may exceed the reference before O is rescaled
template <int DH> struct AtcCfg {
    static constexpr int NSUB = DH / 64;                       // 64-element sub-tiles along the head dimension
    static constexpr int KC = DH == 128 ? 128 : 64;            // keys per chunk
    static constexpr int BUFS = 128 / KC;                      // S / P buffers per tile
    static constexpr int STAGES = 256 / KC;                    // chunks of keys, and of values, in flight
    static constexpr int KSUB = KC * 128;                      // bytes of one KC-key x 64-element sub-tile (keys, values)
    static constexpr int Q_BYTES = NSUB * ATC_SUB;             // a tile of queries
    static constexpr int K_BYTES = NSUB * KSUB;            // a chunk of keys, a chunk of values
    static constexpr int SMEM_BYTES = 2 * Q_BYTES + 2 * STAGES * K_BYTES + 1024;
    static constexpr int TMEM_COLS = 512;                      // S / P of tile t, buffer b: columns 128 t + KC b ..; O of tile t: 256 + 128 t ..
};
static_assert(AtcCfg<128>::SMEM_BYTES + 1024 <= 227 * 1024, "one CTA per SM");

// Instruction descriptor: bf16 A (K-major) and B, fp32 accumulation; b_mn = 1 when B is MN-major.
__host__ __device__ constexpr uint32_t umma_idesc_bf16_b(int M, int N, int b_mn) {
    return umma_idesc_bf16(M, N) | (static_cast<uint32_t>(b_mn) << 16);
}
// Shared-memory descriptor of an MN-major bf16 operand with the 128-byte swizzle: rows of 64 MN-elements (128 bytes),
// one row per K index, 8-row groups 1024 bytes apart; further 64-element MN blocks `mn_block_bytes` apart.
__device__ __forceinline__ uint64_t umma_desc_mn_sw128(uint32_t smem_addr, uint32_t mn_block_bytes) {
    uint64_t d = 0;
    d |= static_cast<uint64_t>((smem_addr & 0x3FFFFu) >> 4);
    d |= static_cast<uint64_t>((mn_block_bytes >> 4) & 0x3FFFu) << 16;   // leading-dimension offset: next MN block
    d |= static_cast<uint64_t>(1024 >> 4) << 32;                          // stride offset: next group of 8 K rows
    d |= static_cast<uint64_t>(1) << 46;
    d |= static_cast<uint64_t>(2) << 61;
    return d;
}
// 16 consecutive fp32 columns of this thread's TMEM lane, written back (the counterpart of tmem_ld16).
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const float (&v)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"
        ::"r"(taddr), "r"(__float_as_uint(v[0])), "r"(__float_as_uint(v[1])), "r"(__float_as_uint(v[2])), "r"(__float_as_uint(v[3])),
          "r"(__float_as_uint(v[4])), "r"(__float_as_uint(v[5])), "r"(__float_as_uint(v[6])), "r"(__float_as_uint(v[7])),
          "r"(__float_as_uint(v[8])), "r"(__float_as_uint(v[9])), "r"(__float_as_uint(v[10])), "r"(__float_as_uint(v[11])),
          "r"(__float_as_uint(v[12])), "r"(__float_as_uint(v[13])), "r"(__float_as_uint(v[14])), "r"(__float_as_uint(v[15]))
        : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
// 64 consecutive fp32 columns of this thread's TMEM lane in one load (load and wait in one statement: the registers
// are not read before the load has landed).
__device__ __forceinline__ void tmem_ld64(uint32_t taddr, float (&v)[64]) {
    uint32_t r[64];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x64.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32,%33,%34,%35,%36,%37,%38,%39,%40,%41,%42,%43,%44,%45,%46,%47,%48,%49,%50,%51,%52,%53,%54,%55,%56,%57,%58,%59,%60,%61,%62,%63}, [%64];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
              "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
              "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
              "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31]),
              "=r"(r[32]), "=r"(r[33]), "=r"(r[34]), "=r"(r[35]), "=r"(r[36]), "=r"(r[37]), "=r"(r[38]), "=r"(r[39]),
              "=r"(r[40]), "=r"(r[41]), "=r"(r[42]), "=r"(r[43]), "=r"(r[44]), "=r"(r[45]), "=r"(r[46]), "=r"(r[47]),
              "=r"(r[48]), "=r"(r[49]), "=r"(r[50]), "=r"(r[51]), "=r"(r[52]), "=r"(r[53]), "=r"(r[54]), "=r"(r[55]),
              "=r"(r[56]), "=r"(r[57]), "=r"(r[58]), "=r"(r[59]), "=r"(r[60]), "=r"(r[61]), "=r"(r[62]), "=r"(r[63])
        : "r"(taddr) : "memory");
#pragma unroll
    for (int i = 0; i < 64; ++i) v[i] = __uint_as_float(r[i]);
}
// ... and 128.
__device__ __forceinline__ void tmem_ld128(uint32_t taddr, float (&v)[128]) {
    uint32_t r[128];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x128.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32,%33,%34,%35,%36,%37,%38,%39,%40,%41,%42,%43,%44,%45,%46,%47,%48,%49,%50,%51,%52,%53,%54,%55,%56,%57,%58,%59,%60,%61,%62,%63,%64,%65,%66,%67,%68,%69,%70,%71,%72,%73,%74,%75,%76,%77,%78,%79,%80,%81,%82,%83,%84,%85,%86,%87,%88,%89,%90,%91,%92,%93,%94,%95,%96,%97,%98,%99,%100,%101,%102,%103,%104,%105,%106,%107,%108,%109,%110,%111,%112,%113,%114,%115,%116,%117,%118,%119,%120,%121,%122,%123,%124,%125,%126,%127}, [%128];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31]),
          "=r"(r[32]), "=r"(r[33]), "=r"(r[34]), "=r"(r[35]), "=r"(r[36]), "=r"(r[37]), "=r"(r[38]), "=r"(r[39]),
          "=r"(r[40]), "=r"(r[41]), "=r"(r[42]), "=r"(r[43]), "=r"(r[44]), "=r"(r[45]), "=r"(r[46]), "=r"(r[47]),
          "=r"(r[48]), "=r"(r[49]), "=r"(r[50]), "=r"(r[51]), "=r"(r[52]), "=r"(r[53]), "=r"(r[54]), "=r"(r[55]),
          "=r"(r[56]), "=r"(r[57]), "=r"(r[58]), "=r"(r[59]), "=r"(r[60]), "=r"(r[61]), "=r"(r[62]), "=r"(r[63]),
          "=r"(r[64]), "=r"(r[65]), "=r"(r[66]), "=r"(r[67]), "=r"(r[68]), "=r"(r[69]), "=r"(r[70]), "=r"(r[71]),
          "=r"(r[72]), "=r"(r[73]), "=r"(r[74]), "=r"(r[75]), "=r"(r[76]), "=r"(r[77]), "=r"(r[78]), "=r"(r[79]),
          "=r"(r[80]), "=r"(r[81]), "=r"(r[82]), "=r"(r[83]), "=r"(r[84]), "=r"(r[85]), "=r"(r[86]), "=r"(r[87]),
          "=r"(r[88]), "=r"(r[89]), "=r"(r[90]), "=r"(r[91]), "=r"(r[92]), "=r"(r[93]), "=r"(r[94]), "=r"(r[95]),
          "=r"(r[96]), "=r"(r[97]), "=r"(r[98]), "=r"(r[99]), "=r"(r[100]), "=r"(r[101]), "=r"(r[102]), "=r"(r[103]),
          "=r"(r[104]), "=r"(r[105]), "=r"(r[106]), "=r"(r[107]), "=r"(r[108]), "=r"(r[109]), "=r"(r[110]), "=r"(r[111]),
          "=r"(r[112]), "=r"(r[113]), "=r"(r[114]), "=r"(r[115]), "=r"(r[116]), "=r"(r[117]), "=r"(r[118]), "=r"(r[119]),
          "=r"(r[120]), "=r"(r[121]), "=r"(r[122]), "=r"(r[123]), "=r"(r[124]), "=r"(r[125]), "=r"(r[126]), "=r"(r[127])
        : "r"(taddr) : "memory");
#pragma unroll
    for (int i = 0; i < 128; ++i) v[i] = __uint_as_float(r[i]);
}
// 16 consecutive columns of this thread's TMEM lane, as they are (the probabilities of 32 keys, two to a column).
__device__ __forceinline__ void tmem_st16_u32(uint32_t taddr, const uint32_t (&v)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"
        ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]), "r"(v[9]),
          "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]) : "memory");
}
// D[tmem] (+)= A[tmem] * B[smem]: A's rows are the TMEM lanes, two bf16 of K per 32-bit column (16 of K: eight columns).
// 64 elements of K, issued by one lane of a converged warp (see umma_bf16_k64).
__device__ __forceinline__ void umma_bf16_ts_k64(uint32_t tmem_d, uint32_t tmem_a, uint64_t desc_b, uint64_t step_b, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred e, p, t;\n\t"
        "elect.sync _|e, 0xffffffff;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "setp.eq.b32 t, 0, 0;\n\t"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], [%5], %6, %3, t;\n\t"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], [%7], %8, %3, t;\n\t"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], [%9], %10, %3, t;\n\t}"
        ::"r"(tmem_d), "r"(tmem_a), "l"(desc_b), "r"(idesc), "r"(accumulate), "r"(tmem_a + 8), "l"(desc_b + step_b),
          "r"(tmem_a + 16), "l"(desc_b + 2 * step_b), "r"(tmem_a + 24), "l"(desc_b + 3 * step_b) : "memory");
}
// Two fp32 operations in one instruction: a * b + c, and a + b, on pairs.
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
    float2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(reinterpret_cast<uint64_t&>(d))
        : "l"(reinterpret_cast<const uint64_t&>(a)), "l"(reinterpret_cast<const uint64_t&>(b)), "l"(reinterpret_cast<const uint64_t&>(c)));
    return d;
}
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
    float2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(reinterpret_cast<uint64_t&>(d))
        : "l"(reinterpret_cast<const uint64_t&>(a)), "l"(reinterpret_cast<const uint64_t&>(b)));
    return d;
}
// 2^x by the hardware approximation (relative error about 2^-22; 2^-inf = 0), one instruction.
__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// grid: (heads, groups), the last group first; dynamic smem AtcCfg<DH>::SMEM_BYTES.
// tmq: queries [M][d_model] (box 64 x 128); tmk / tmv: one layer's cache seen as [(seq, kv head, position)][DH] (box 64 x 64).
template <int DH>
__global__ void __launch_bounds__(ATC_THREADS, 1)
attn_prefill_tc_kernel(const AttnTcArgs a, const __grid_constant__ CUtensorMap tmq, const __grid_constant__ CUtensorMap tmk,
                       const __grid_constant__ CUtensorMap tmv) {
    using C = AtcCfg<DH>;
    extern __shared__ __align__(1024) unsigned char smem_dyn[];
    __shared__ __align__(8) uint64_t s_qfull, s_kfull[C::STAGES], s_kfree[C::STAGES], s_vfull[C::STAGES], s_vfree[C::STAGES];
    __shared__ __align__(8) uint64_t s_sfull[2][C::BUFS], s_pready[2][C::BUFS], s_odone[2], s_ofinal[2];   // [tile][buffer]; odone[tile]: one phase per chunk but the last, ofinal[tile]: the last
    __shared__ uint32_t s_tmem;

    const int tid = threadIdx.x, warp = warp_uniform(tid >> 5), lane = tid & 31;
    const uint32_t q0 = (smem_u32(smem_dyn) + 1023u) & ~1023u, k0 = q0 + 2 * C::Q_BYTES, v0 = k0 + C::STAGES * C::K_BYTES;

    if (warp == 9) {
        if (lane == 0) {
            mbar_init(smem_u32(&s_qfull), 1);
            for (int s = 0; s < C::STAGES; ++s) {
                mbar_init(smem_u32(&s_kfull[s]), 1); mbar_init(smem_u32(&s_kfree[s]), 1);
                mbar_init(smem_u32(&s_vfull[s]), 1); mbar_init(smem_u32(&s_vfree[s]), 1);
            }
            for (int t = 0; t < 2; ++t) {
                mbar_init(smem_u32(&s_odone[t]), 1); mbar_init(smem_u32(&s_ofinal[t]), 1);
                for (int u = 0; u < C::BUFS; ++u) {
                    mbar_init(smem_u32(&s_sfull[t][u]), 1);
                    mbar_init(smem_u32(&s_pready[t][u]), 4);   // one arrive per softmax warp of the tile
                }
            }
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
    pdl_wait();                // queries, keys and values come from the kernel before this one

    const int h = blockIdx.x, g = gridDim.y - 1 - blockIdx.y;
    const int row0 = a.grp_row0[g], cnt = a.grp_cnt[g];
    const int b = a.row_seq[row0];
    const int pos_first = a.row_pos[row0];
    // chunks of each tile: up to the tile's last query (0: the group ends before the tile)
    const int n0 = (pos_first + min(cnt, ATC_TILE) - 1) / C::KC + 1;
    const int n1 = cnt > ATC_TILE ? (pos_first + cnt - 1) / C::KC + 1 : 0;
    const int n_max = max(n0, n1);
    const int kv_row0 = (b * a.n_kv_heads + h / (a.n_heads / a.n_kv_heads)) * a.t_max;   // row of position 0 of this head's key/value head in the cache's 2-D view

    if (warp == 8) {
        // ---- TMA: Q once, then K and V of every chunk as their stages come free ----
        {
            const bool leader = elect_one();
            if (leader) { tma_prefetch_desc(&tmq); tma_prefetch_desc(&tmk); tma_prefetch_desc(&tmv); }
            const int tiles = n1 > 0 ? 2 : 1;
            if (leader) mbar_arrive_expect_tx(smem_u32(&s_qfull), tiles * C::Q_BYTES);
            for (int t = 0; t < tiles && leader; ++t)
                for (int sb = 0; sb < C::NSUB; ++sb)
                    tma_load_2d_nohint(q0 + t * C::Q_BYTES + sb * ATC_SUB, &tmq, h * DH + sb * 64, row0 + t * ATC_TILE, smem_u32(&s_qfull));
            for (int c = 0; c < n_max; ++c) {
                const int st = c % C::STAGES;
                const uint32_t old = ((c / C::STAGES) - 1) & 1;
                if (c >= C::STAGES && !mbar_wait_warp(smem_u32(&s_kfree[st]), old)) { tc_report(a.err_flag, TC_ERR_SLOT); break; }
                if (elect_one()) {
                    mbar_arrive_expect_tx(smem_u32(&s_kfull[st]), C::K_BYTES);
                    for (int sb = 0; sb < C::NSUB; ++sb)
                        tma_load_2d_nohint(k0 + st * C::K_BYTES + sb * C::KSUB, &tmk, sb * 64, kv_row0 + c * C::KC, smem_u32(&s_kfull[st]));
                }
                if (c >= C::STAGES && !mbar_wait_warp(smem_u32(&s_vfree[st]), old)) { tc_report(a.err_flag, TC_ERR_SLOT); break; }
                if (elect_one()) {
                    mbar_arrive_expect_tx(smem_u32(&s_vfull[st]), C::K_BYTES);
                    for (int sb = 0; sb < C::NSUB; ++sb)
                        tma_load_2d_nohint(v0 + st * C::K_BYTES + sb * C::KSUB, &tmv, sb * 64, kv_row0 + c * C::KC, smem_u32(&s_vfull[st]));
                }
            }
            pdl_launch_dependents();
        }
        __syncwarp();
    } else if (warp == 9) {
        // ---- MMA issue: one lane of a converged warp ----
        constexpr uint32_t idesc_s = umma_idesc_bf16_b(128, C::KC, 0);
        constexpr uint32_t idesc_o = umma_idesc_bf16_b(128, DH, 1);
        // S = Q K^T of chunk c into buffer c % BUFS: both operands K-major, 64 elements of the head dimension at a time
        auto issue_s = [&](int t, int c) {
            const uint32_t qaddr = q0 + t * C::Q_BYTES, kaddr = k0 + (c % C::STAGES) * C::K_BYTES;
#pragma unroll
            for (int sb = 0; sb < C::NSUB; ++sb)
                umma_bf16_k64(tmem + t * 128 + (c % C::BUFS) * C::KC, umma_desc_k_sw128(qaddr + sb * ATC_SUB), umma_desc_k_sw128(kaddr + sb * C::KSUB), idesc_s, sb != 0 ? 1u : 0u);
            umma_commit_one(smem_u32(&s_sfull[t][c % C::BUFS]));
        };
        auto keys = [&](int c) {   // chunk c's keys are there
            const bool there = mbar_wait_warp(smem_u32(&s_kfull[c % C::STAGES]), (c / C::STAGES) & 1);
            if (!there) tc_report(a.err_flag, TC_ERR_OPERANDS);
            tc_fence_after_sync();
            return there;
        };
        bool ok = mbar_wait_warp(smem_u32(&s_qfull), 0);
        if (!ok) tc_report(a.err_flag, TC_ERR_OPERANDS);
        for (int c = 0; c < min(n_max, C::BUFS) && ok; ++c) {
            if (!(ok = keys(c))) break;
            for (int t = 0; t < 2; ++t)
                if (c < (t == 0 ? n0 : n1)) issue_s(t, c);
            umma_commit_one(smem_u32(&s_kfree[c]));
        }
        for (int c = 0; c < n_max && ok; ++c) {
            const int st = c % C::STAGES, buf = c % C::BUFS, next = c + C::BUFS;
            ok = mbar_wait_warp(smem_u32(&s_vfull[st]), (c / C::STAGES) & 1);
            if (!ok) { tc_report(a.err_flag, TC_ERR_OPERANDS); break; }
            if (next < n_max && !keys(next)) break;
            for (int t = 0; t < 2; ++t) {
                const int n = t == 0 ? n0 : n1;
                if (c >= n) continue;
                if (!mbar_wait_warp(smem_u32(&s_pready[t][buf]), (c / C::BUFS) & 1)) { tc_report(a.err_flag, TC_ERR_ACCUM); ok = false; break; }
                tc_fence_after_sync();
                // O += P V: P from TMEM, V MN-major; then the S that takes P's place, behind it in the pipe
#pragma unroll
                for (int ks = 0; ks < C::KC / 64; ++ks)
                    umma_bf16_ts_k64(tmem + 256 + t * 128, tmem + t * 128 + buf * C::KC + ks * 32, umma_desc_mn_sw128(v0 + st * C::K_BYTES + ks * 8192, C::KSUB),
                                     2048 >> 4, idesc_o, (c | ks) != 0 ? 1u : 0u);
                umma_commit_one(smem_u32(c + 1 < n ? &s_odone[t] : &s_ofinal[t]));   // O of tile t holds chunks 0 .. c
                if (next < n) issue_s(t, next);
            }
            umma_commit_one(smem_u32(&s_vfree[st]));
            if (next < n_max) umma_commit_one(smem_u32(&s_kfree[next % C::STAGES]));
        }
        __syncwarp();
    } else {
        // ---- softmax warps: thread = query = TMEM lane ----
        const int t = warp >> 2, wl = warp & 3;
        const int qi = t * ATC_TILE + wl * 32 + lane;
        const int n = t == 0 ? n0 : n1;
        const int tile_pos = pos_first + t * ATC_TILE;
        const int qpos = pos_first + qi;                 // (rows past cnt compute on whatever the tile holds; never stored)
        const uint32_t lane_addr = tmem + (static_cast<uint32_t>(wl * 32) << 16);
        const uint32_t o_addr = lane_addr + 256 + t * 128;
        // Everything runs in the base-2 domain: with sc2 = scale * log2(e), a probability is 2^(s * sc2 - m) (half a
        // paired multiply-add and one ex2 per element); m is the reference maximum in that domain.
        const float sc2 = a.scale * 1.4426950408889634f;
        constexpr float LAZY2 = ATC_LAZY * 1.4426950408889634f;
        float m = -INFINITY, l = 0.f;                    // reference maximum of the exponentials, running sum
        bool ok = true;
        for (int c = 0; c < n; ++c) {
            if (!mbar_wait(smem_u32(&s_sfull[t][c % C::BUFS]), (c / C::BUFS) & 1)) { tc_report(a.err_flag, TC_ERR_ACCUM); ok = false; break; }
            tc_fence_after_sync();
            const uint32_t s_addr = lane_addr + t * 128 + (c % C::BUFS) * C::KC;
            float s[C::KC];
            if constexpr (C::KC == 128) tmem_ld128(s_addr, s); else tmem_ld64(s_addr, s);                       // this row of S, raw
            // keys after the query's position become -inf (every chunk but the tile's last ones lies wholly before its first query)
            if (c * C::KC + C::KC - 1 > tile_pos) {
#pragma unroll
                for (int i = 0; i < C::KC; ++i) s[i] = (c * C::KC + i <= qpos) ? s[i] : -INFINITY;
            }
            float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
            for (int i = 0; i < C::KC; i += 8)
#pragma unroll
                for (int u = 0; u < 4; ++u) mx[u] = fmaxf(mx[u], fmaxf(s[i + u], s[i + 4 + u]));
            const float mc = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])) * sc2;   // the chunk's maximum in the base-2 domain (the scale is positive)
            // lazy reference: it moves only when this chunk's maximum exceeds it by more than the margin
            const bool move = mc > m + LAZY2;            // (first chunk: m = -inf, every row with a visible key moves)
            if (c > 0 && __any_sync(0xffffffffu, move)) {   // O is touched only when P V of the previous chunk is complete
                // (phase c - 1 or c is current: S of chunk c lies behind product c - BUFS, and product c needs this warp's P)
                if (!mbar_wait(smem_u32(&s_odone[t]), (c - 1) & 1)) { tc_report(a.err_flag, TC_ERR_ACCUM); ok = false; break; }
                tc_fence_after_sync();
                const float f = (move && m > -INFINITY) ? ex2_approx(m - mc) : 1.0f;   // rows that keep their reference: exactly 1
#pragma unroll 1
                for (int e0 = 0; e0 < DH; e0 += 16) {
                    float o[16];
                    tmem_ld16(o_addr + e0, o);
#pragma unroll
                    for (int i = 0; i < 16; ++i) o[i] *= f;
                    tmem_st16(o_addr + e0, o);
                }
                l *= f;
            }
            if (move) m = mc;
            // probabilities relative to the reference (2^(-inf) = 0 for masked keys), their sum, and the row of P where S was
            const float2 sc22 = make_float2(sc2, sc2), nm2 = make_float2(-m, -m);
            float2 ls0 = make_float2(0.f, 0.f), ls1 = make_float2(0.f, 0.f);
#pragma unroll
            for (int c0 = 0; c0 < C::KC; c0 += 32) {
                uint32_t pk[16];
#pragma unroll
                for (int i = 0; i < 32; i += 4) {
                    const float* sp = &s[c0 + i];
                    const float2 x0 = fma2(make_float2(sp[0], sp[1]), sc22, nm2), x1 = fma2(make_float2(sp[2], sp[3]), sc22, nm2);
                    const float2 p0 = make_float2(ex2_approx(x0.x), ex2_approx(x0.y)), p1 = make_float2(ex2_approx(x1.x), ex2_approx(x1.y));
                    ls0 = add2(ls0, p0);
                    ls1 = add2(ls1, p1);
                    pk[i >> 1] = pack_bf16x2(p0.x, p0.y);
                    pk[(i >> 1) + 1] = pack_bf16x2(p1.x, p1.y);
                }
                tmem_st16_u32(s_addr + (c0 >> 1), pk);
            }
            ls0 = add2(ls0, ls1);
            l += ls0.x + ls0.y;
            tmem_wait_st();
            tc_fence_before_sync();      // P and a rescaled O are in TMEM before the next product reads them
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&s_pready[t][c % C::BUFS]));
        }
        if (ok && n > 0) {   // all chunks accumulated
            // (a barrier of its own: this S being there says no more than that the product BUFS chunks back is done, and a wait for a
            // parity cannot tell a phase from the one two before it)
            if (!mbar_wait(smem_u32(&s_ofinal[t]), 0)) { tc_report(a.err_flag, TC_ERR_ACCUM); ok = false; }
            tc_fence_after_sync();
            const float inv = 1.0f / l;
            bf16* dst = static_cast<bf16*>(a.out) + (size_t)(row0 + qi) * a.ldo + h * DH;
#pragma unroll 2
            for (int e0 = 0; e0 < DH; e0 += 16) {
                float o[16];
                tmem_ld16(o_addr + e0, o);   // warp-wide: every lane takes part
                if (ok && qi < cnt) {
                    uint4 lo, hi;
                    lo.x = pack_bf16x2(o[0] * inv, o[1] * inv); lo.y = pack_bf16x2(o[2] * inv, o[3] * inv);
                    lo.z = pack_bf16x2(o[4] * inv, o[5] * inv); lo.w = pack_bf16x2(o[6] * inv, o[7] * inv);
                    hi.x = pack_bf16x2(o[8] * inv, o[9] * inv); hi.y = pack_bf16x2(o[10] * inv, o[11] * inv);
                    hi.z = pack_bf16x2(o[12] * inv, o[13] * inv); hi.w = pack_bf16x2(o[14] * inv, o[15] * inv);
                    *reinterpret_cast<uint4*>(dst + e0) = lo;
                    *reinterpret_cast<uint4*>(dst + e0 + 8) = hi;
                }
            }
            tc_fence_before_sync();
        }
    }
    tc_fence_before_sync();
    __syncthreads();
    if (warp == 9) tmem_dealloc(tmem, C::TMEM_COLS);
}

}  // namespace tandem
