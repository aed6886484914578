// Host side of the C boundary: context, arena layout, pass scheduling, and the exported entry points.
#include <cuda_runtime.h>
#include <limits.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>
#include <time.h>

#include <algorithm>
#include <atomic>
#include <mutex>
#include <new>
#include <type_traits>
#include <vector>

#include "../../include/tandem.h"
#include "attention.cuh"
#include "attention_tc.cuh"
#include "common.cuh"
#include "gemm_simt.cuh"
#include "gemm_tc.cuh"
#include "misc_kernels.cuh"
#include "router.cuh"
#include "sampling.cuh"

using namespace tandem;

namespace {

thread_local char g_cuda_err[256] = "";

#define CK(call)                                                                                  \
    do {                                                                                          \
        cudaError_t err__ = (call);                                                               \
        if (err__ != cudaSuccess) {                                                               \
            snprintf(g_cuda_err, sizeof(g_cuda_err), "%s at %s:%d", cudaGetErrorString(err__), __FILE__, __LINE__); \
            return TANDEM_ERR_CUDA;                                                               \
        }                                                                                         \
    } while (0)
#define TRY(expr)                             \
    do {                                      \
        tandem_status st__ = (expr);          \
        if (st__ != TANDEM_OK) return st__;   \
    } while (0)

size_t align_up(size_t v, size_t a = 256) { return (v + a - 1) / a * a; }
int cdiv(int a, int b) { return (a + b - 1) / b; }

// Queries per attention group of the large model in a teacher-forced pass: one group of the MMA's eight columns (a warp meets all
// keys of its group on its own, so more and lighter warps: 20.5 -> 17.5 us a layer for 772 rows x 16 heads x 64 under ncu).
constexpr int PASS_GROUP = 8;
// Most rows of a prompt or teacher-forced pass whose projections run beside the large model's layers, see prompt_project_forked.
constexpr int PROMPT_FORK_ROWS = 2048;

struct Layout {   // byte offsets into the arena
    size_t kv_large, kv_small;
    size_t st_n, st_pending, st_drafts, st_targets, st_accept, st_emitted, st_done, st_out, st_counters, st_hist;
    size_t st_block_len, st_drafting, st_confidence;
    size_t forced_ids, forced_len, forced_nll, forced_top;   // teacher-forced forward: given tokens [B][T], lengths [B], scores [B][T]
    // ... in one pass (bf16), see place_pass: rows in front of the products, GELU outputs, queries and the projections' buffers of the
    // large model's part; stream, rows, own keys / values, GELU outputs, queries of the small model's; the head's per-tile results
    size_t fr_x, fr_f, fr_q, fr_raw, fr_yhat, fr_a, fr_t1, fr_hs, fr_xs, fr_kv, fr_fs, fr_tiles;
    size_t fa_yhat, fa_a, fa_t1;            // ... the projections' buffers apart from what the large model's layers write
    size_t fr_start, fr_truth;              // ... the sequences' first rows, the rows' next tokens (where a prompt pass has its staged inputs)
    size_t row_tok, row_seq, row_pos, grp_row0, grp_cnt;
    size_t stage;                                   // a prompt pass's lengths, offsets and token ids as the host staged them
    size_t attn_counters;   // inside the zero-filled state block
    size_t h_large, h_small, a, q, o, f, xb, t1, yhat, a_s, logits_large, logits_small, part_ml, part_acc, dbg;
    size_t smp_large, smp_small;                     // sampled SPEED: (maximum, sum of weights) of every row of logits
    size_t amax_val_large, amax_idx_large, amax_val_small, amax_idx_small;
    size_t a32, o32, f32;                           // value / remainder planes between the bf16 decode kernels: LayerNorm inputs ((x - c).g) / attention / GELU outputs
    size_t ln_src, ln_rows_large, ln_rows_small, ln_stats, ln_ref;   // LayerNorms behind the GEMMs (bf16 decode): sources, their rows, the token rows' statistics, reference values (see ln_ref_of)
    size_t proj_snap, proj_yhat, proj_a, proj_t1;   // per small layer: the decode projection's own buffers (it runs beside the large pass)
    size_t total;
    int max_rows, dec_rows, max_groups, n_chunks_max, vocab_tiles, score_tiles;
    int fr_apart;                            // whether there is a second set of the projections' buffers
    int fr_rows, fr_head_rows;               // most rows of a teacher-forced pass, and of one run of its output head
    size_t kv_large_layer, kv_small_layer;   // elements per (layer, k-or-v)
};

struct Model {
    tandem_dims d;
    int kv_heads, d_kv;     // key/value heads and the width of a position's keys (kv_heads * d_head)
    int wbase;
    size_t kv_off;          // arena offset of this model's KV cache
    size_t kv_layer_elems;  // elements per (layer, K or V): B * kv_heads * T * dh
};

}  // namespace

enum { PC_GEMM_SMALLM = 0, PC_GEMM_TILED, PC_ATTN_SPLIT, PC_ATTN_MERGE, PC_ATTN_PROMPT, PC_LAYERNORM, PC_ROWS, PC_ARGMAX,
       PC_VERIFY, PC_GEMM_TC_DECODE, PC_GEMM_TC_TILED, PC_COUNT };

struct Prof {   // optional per-launch timing with CUDA events (measurement hook)
    bool on = false;
    std::vector<cudaEvent_t> ev;
    std::vector<int> cls;
    std::vector<double> bytes;
    size_t used = 0;   // events used (two per launch)
};

struct tandem_ctx {
    Prof prof;
    tandem_config cfg;
    std::vector<int32_t> layer_map;
    std::vector<const void*> w;
    Layout lay;
    Model large, small;
    int tbase;          // first FF_Tandem weight index
    int hidden;
    unsigned char* arena;
    cudaStream_t stream;
    size_t esz;         // storage element size
    // host trackers
    int batch;          // sequences of the current prefill (0 = none)
    int n_ub;           // upper bound on max_b n_b (exact after every synchronising call)
    long long n_sum;    // sum_b n_b at the last synchronisation (accounting only)
    int32_t* pinned;    // staging for prefill row arrays and small read-backs
    size_t pinned_ints;
    int64_t launches = 0;
    int last_gamma = 0;
    size_t hidden_at = 0;                // where the large model's final residual stream of the last decode rows lies
    LoopState st{};
    // CUDA graphs of one iteration, keyed by everything baked into the captured launches
    struct GraphEntry {
        int kind, gamma, mode, max_new, batch, chunks;
        uint64_t seed;
        bool warm;
        cudaGraphExec_t exec;
        int64_t kernels;
    };
    std::vector<GraphEntry> graphs;
    cudaStream_t cap_stream = nullptr;   // capture happens here (the caller's stream may be the legacy default stream)
    bool use_graphs = true;
    int chunks_launch = 1;               // attention grid size along the context for the current iteration
    int32_t* hflags = nullptr;           // mapped pinned host memory the verify kernel publishes to
    int64_t ticket = 0;                  // verify kernels enqueued since creation (the device counts them too)
    // tensor-core path (bf16 only)
    int n_lns = 0;                       // LayerNorms of both models (bf16), see Layout::ln_src
    bool use_pdl = true;                 // programmatic dependent launch between the decode kernels
    int amax_tiles = 0;                  // tiles of the output heads' arg-max results per row
    int n_sms = 0;                       // multiprocessors of the context's device: split-K decode GEMMs aim for about one CTA each
    std::vector<CUtensorMap> wmap;       // one per weight pointer (matrices only), box 128 rows x 64 columns
    std::vector<CUtensorMap> wpart;      // the same in boxes of 32 rows
    // Decode activations as two bf16 planes (values, then remainders, dec_rows rows each) that the consuming GEMM loads by
    // TMA: maps of the residual stream (less c, times the next LayerNorm's gain: see NextLn) / attention / GELU buffers, [buffer 0..2][0 large,
    // 1 small], boxes of 16 rows of both planes.
    CUtensorMap xmap[3][2];
    CUtensorMap lnmap[2];                // the LayerNorms' own rows, four per LayerNorm (2 l, 2 l + 1 of layer l, then the final one)
    std::vector<CUtensorMap> kmap, vmap; // the large model's key / value cache of each layer as [(seq, head, position)][d_head]
    cudaStream_t side = nullptr;         // the decode-time FF_Tandem projections run here, beside the large model's later layers
    std::vector<cudaEvent_t> ev_fork;    // one per small layer
    cudaEvent_t ev_join = nullptr;
    cudaEvent_t ev_staged = nullptr;     // the last prompt pass's copy out of the pinned staging buffer
    bool next_launch_plain = false;      // the next launch follows a cross-stream wait: no programmatic dependency on a kernel
    bool setup_failed = false;           // a launch helper could not encode a tensor map: reported by the enclosing call
    bool tc_prompt_attn = false;         // prompt attention on the tensor cores (head size 64 or 128)
    int prompt_group = ATT_NQ;           // queries per attention group of the prompt pass
    float temp_large = 1.0f, temp_small = 1.0f;   // sampled SPEED (accept mode 4): temperatures of the two models
    RouterArgs router{};                 // adaptive block length: the router's weights (caller-owned, DEVICE) and threshold
    bool has_router = false;
    int64_t router_ticket = 0;           // router launches since creation
    double prompt_sq_sum = 0.0;          // sum over the sequences of the current prompt pass of (rows)^2 (accounting of the attention's work)
};

namespace {
// Brackets one launch with two events when profiling is on.
struct ProfScope {
    tandem_ctx& c;
    bool active;
    ProfScope(tandem_ctx& ctx, int cls, double bytes) : c(ctx), active(false) {
        Prof& p = c.prof;
        if (p.on && p.used + 2 <= p.ev.size()) {
            active = true;
            p.cls.push_back(cls);
            p.bytes.push_back(bytes);
            cudaEventRecord(p.ev[p.used], c.stream);
        }
    }
    ~ProfScope() {
        if (active) { cudaEventRecord(c.prof.ev[c.prof.used + 1], c.stream); c.prof.used += 2; }
    }
};
}  // namespace

namespace {

int dims_ok(const tandem_dims& d) {
    if (d.n_layers < 1 || d.d_model < 8 || d.n_heads < 1 || d.d_ff < 8 || d.vocab < 1 || d.max_pos < 1) return 0;
    if (d.d_model % d.n_heads) return 0;
    const int dh = d.d_model / d.n_heads;
    if (dh != 32 && dh != 64 && dh != 128) return 0;
    if (d.d_model % 8 || d.d_ff % 8) return 0;
    if (d.n_kv_heads < 0 || (d.n_kv_heads > 0 && d.n_heads % d.n_kv_heads)) return 0;
    return 1;
}
int kv_heads_of(const tandem_dims& d) { return d.n_kv_heads > 0 ? d.n_kv_heads : d.n_heads; }
int d_kv_of(const tandem_dims& d) { return kv_heads_of(d) * (d.d_model / d.n_heads); }

tandem_status validate(const tandem_config* c) {
    if (!c || !c->layer_map) return TANDEM_ERR_INVALID_ARG;
    if (c->dtype != TANDEM_DTYPE_FP32 && c->dtype != TANDEM_DTYPE_BF16) return TANDEM_ERR_INVALID_ARG;
    if (c->ff_tandem_kind != TANDEM_FF_LINEAR && c->ff_tandem_kind != TANDEM_FF_MLP) return TANDEM_ERR_INVALID_ARG;
    if (c->max_batch < 1 || c->max_seq < 2 || c->gamma_max < 0 || c->gamma_max > TANDEM_GAMMA_LIMIT) return TANDEM_ERR_INVALID_ARG;
    if (c->max_prefill_rows < 0 || c->ff_tandem_hidden < 0 || c->device < 0) return TANDEM_ERR_INVALID_ARG;
    if (!dims_ok(c->large) || !dims_ok(c->small)) return TANDEM_ERR_SHAPE;
    if (c->large.vocab != c->small.vocab) return TANDEM_ERR_SHAPE;
    if (c->ff_tandem_hidden % 8) return TANDEM_ERR_SHAPE;
    if ((long long)c->max_batch * (c->gamma_max + 1) > 256) return TANDEM_ERR_SHAPE;
    for (int j = 0; j < c->small.n_layers; ++j)
        if (c->layer_map[j] < 0 || c->layer_map[j] > c->large.n_layers) return TANDEM_ERR_INVALID_ARG;
    return TANDEM_OK;
}

// A teacher-forced pass of `rows` rows in the prompt pass's space from `at` on, as fp32 rows or two bf16 planes; returns where it ends.
// What two steps of a layer never hold together shares a place: the large model's attention writes where the rows of its QKV map
// were, and the GELU outputs lie over the queries and the projections' buffers (the projections are done before the
// FFN's first product).  The small model's part begins when the large model's is over.
size_t place_pass(const tandem_config& c, Layout& L, size_t at, size_t rows) {
    const size_t dL = c.large.d_model, dS = c.small.d_model;
    const size_t hidden = c.ff_tandem_kind == TANDEM_FF_LINEAR ? 0 : (c.ff_tandem_hidden > 0 ? c.ff_tandem_hidden : c.small.d_model);
    size_t off = at;
    auto take = [&](size_t bytes) { size_t o = off; off = align_up(off + bytes); return o; };
    L.fr_x = take(rows * dL * 4);
    L.fr_f = off;
    L.fr_raw = take(rows * dL * 4); L.fr_t1 = take(rows * hidden * 4); L.fr_yhat = take(rows * dS * 4); L.fr_a = take(rows * dS * 4);
    L.fr_q = take(rows * dL * 2);
    size_t end = std::max(off, align_up(L.fr_f + rows * c.large.d_ff * 4));
    off = at;
    L.fr_hs = take(rows * dS * 4); L.fr_xs = take(rows * dS * 4);
    L.fr_tiles = off;                       // (the layers behind it)
    L.fr_kv = take(2 * rows * d_kv_of(c.small) * 2);
    L.fr_fs = take(rows * std::max<size_t>(c.small.d_ff * 4, dS * 2));   // GELU outputs, queries
    return std::max(end, off);
}

// Columns per warp of the fp32 few-row kernel: one until that is two CTAs on each of 148 multiprocessors, then four (the staged rows are
// read once for them).  The output head's arg-max results are laid out by it.
int rows_columns(int N) { return N > 2 * GS_WARPS * 148 ? 4 : 1; }

Layout make_layout(const tandem_config& c) {
    Layout L;
    memset(&L, 0, sizeof(L));
    const size_t esz = c.dtype == TANDEM_DTYPE_BF16 ? 2 : 4;
    const size_t B = c.max_batch, T = c.max_seq, GL = TANDEM_GAMMA_LIMIT;
    const int hidden = c.ff_tandem_hidden > 0 ? c.ff_tandem_hidden : c.small.d_model;
    L.dec_rows = c.max_batch * (c.gamma_max + 1);
    const long long pre = c.max_prefill_rows > 0 ? c.max_prefill_rows : (long long)c.max_batch * c.max_seq;
    L.max_rows = (int)std::max<long long>(pre, L.dec_rows);
    L.max_groups = L.max_rows / ATT_NQ + c.max_batch + 1;
    L.n_chunks_max = cdiv(c.max_seq, ATT_CH);
    const size_t dmax = std::max(std::max(c.large.d_model, c.small.d_model), hidden);
    const size_t fmax = std::max(c.large.d_ff, c.small.d_ff);
    const size_t hmax = std::max(c.large.n_heads, c.small.n_heads);
    const bool bf = c.dtype == TANDEM_DTYPE_BF16;
    const size_t R = L.max_rows, RD = L.dec_rows, V = c.large.vocab;
    size_t off = 0;
    auto take = [&](size_t bytes) { size_t o = off; off = align_up(off + bytes); return o; };
    L.kv_large_layer = B * T * d_kv_of(c.large);
    L.kv_small_layer = B * T * d_kv_of(c.small);
    L.kv_large = take((size_t)c.large.n_layers * 2 * L.kv_large_layer * esz);
    L.kv_small = take((size_t)c.small.n_layers * 2 * L.kv_small_layer * esz);
    L.st_n = take(B * 4); L.st_pending = take(B * 4); L.st_drafts = take(B * GL * 4);
    L.st_targets = take(B * (GL + 1) * 4); L.st_accept = take(B * 4);
    L.st_done = take(B * 4); L.st_out = take(B * T * 4);
    L.st_counters = take(16 * 4); L.st_hist = take((GL + 1) * 8); L.st_emitted = take(B * 4);   // adjacent: read back together
    L.st_block_len = take(B * 4); L.st_drafting = take(B * 4); L.st_confidence = take(B * GL * 4);
    L.row_tok = take(R * 4); L.row_seq = take(R * 4); L.row_pos = take(R * 4);
    L.grp_row0 = take((size_t)L.max_groups * 4); L.grp_cnt = take((size_t)L.max_groups * 4);
    L.stage = take((4 * B + R + B) * 4);
    L.fr_start = L.stage; L.fr_truth = L.stage + 5 * B * 4;   // (B + 1, R)
    L.attn_counters = take(B * hmax * 4);
    L.h_large = take(R * c.large.d_model * 4);
    L.h_small = take(B * c.small.d_model * 4);
    const size_t ws = off;
    L.a = take(R * dmax * esz); L.q = take(R * dmax * esz); L.o = take(R * dmax * esz);
    L.f = take(R * fmax * esz);
    L.xb = take(R * c.large.d_model * esz); L.t1 = take(R * hidden * esz);
    L.yhat = take(R * c.small.d_model * 4); L.a_s = take(R * c.small.d_model * esz);
    L.part_ml = take(RD * hmax * L.n_chunks_max * 2 * 4);
    L.part_acc = take(RD * dmax * L.n_chunks_max * 4);
    if (bf) {
        // A teacher-forced pass takes what it finds here (the attention's parts are fp32 contexts' only): a context asks for no more memory
        // than its prompt pass needs, and a forward over more rows goes in several passes.  Where feed-forward layers are four times
        // as wide as the models (or less), a pass has room for a prompt pass's rows.  Only a work space that cannot hold one
        // block, or sixteen rows' results of the head, grows.
        const size_t ws_end = off, least = std::min<size_t>(R, std::max(1, c.gamma_max));
        size_t rows = std::min<size_t>(R, 32768);
        while (rows > least && place_pass(c, L, ws, rows) > ws_end) {
            const size_t fit = (size_t)((double)rows * (double)(ws_end - ws) / (double)(place_pass(c, L, ws, rows) - ws));
            rows = std::max(least, std::min(rows - 1, fit));
        }
        const size_t pass_end = std::max(ws_end, place_pass(c, L, ws, rows));
        L.fr_rows = (int)rows;
        L.score_tiles = cdiv(c.large.vocab, SCORE_TILE);
        const size_t tile_bytes = (size_t)L.score_tiles * 12, few = std::min<size_t>(rows, 16);
        L.fr_head_rows = (int)std::max(few, std::min(std::min<size_t>(rows, 1024), (pass_end - L.fr_tiles) / tile_bytes));
        off = std::max(pass_end, align_up(L.fr_tiles + few * tile_bytes));
    }
    L.dbg = take(T * dmax * 4);
    L.logits_small = take((size_t)std::max(1, c.gamma_max) * B * V * 4);
    if (bf) {
        // Behind the large model's part, up to the end of the logits that only its successor writes: the projections' buffers once more, if
        // they fit (see Rows::apart).
        const size_t end = off, rows = L.fr_rows, t1 = c.ff_tandem_kind == TANDEM_FF_LINEAR ? 0 : rows * hidden * 4, y = rows * c.small.d_model * 4;
        off = std::max(L.fr_q + rows * c.large.d_model * 2, L.fr_f + rows * c.large.d_ff * 4);
        off = align_up(off);
        if (off + align_up(t1) + 2 * align_up(y) <= end) { L.fa_t1 = take(t1); L.fa_yhat = take(y); L.fa_a = take(y); L.fr_apart = 1; }
        off = end;
    }
    L.logits_large = take(RD * V * 4);
    L.forced_ids = take(B * T * 4); L.forced_len = take(B * 4); L.forced_nll = take(B * T * 4); L.forced_top = take(B * T * 4);
    L.smp_large = take(RD * 8); L.smp_small = take((size_t)std::max(1, c.gamma_max) * B * 8);
    auto take_amax = [&](int columns) {
        L.vocab_tiles = cdiv(c.large.vocab, columns);
        L.amax_val_large = take(RD * L.vocab_tiles * 4); L.amax_idx_large = take(RD * L.vocab_tiles * 4);
        L.amax_val_small = take(B * L.vocab_tiles * 4); L.amax_idx_small = take(B * L.vocab_tiles * 4);
    };
    const size_t amax = off;
    take_amax(128);
    const size_t nS = c.small.n_layers;
    L.a32 = take(RD * dmax * 4); L.o32 = take(RD * dmax * 4); L.f32 = take(RD * fmax * 4);
    if (!bf) {   // blocks of fewer columns, which reach over the planes that fp32 contexts have no use for
        const size_t end = off;
        off = amax;
        take_amax(GS_WARPS * rows_columns(c.large.vocab));
        off = std::max(off, end);
    }
    L.proj_snap = take(nS * RD * c.large.d_model * 4);
    L.proj_yhat = take(nS * RD * c.small.d_model * 4);
    L.proj_a = take(nS * RD * c.small.d_model * 4);
    L.proj_t1 = take(nS * RD * hidden * 4);
    L.ln_src = take((size_t)(2 * c.large.n_layers + 1 + 2 * c.small.n_layers + 1) * sizeof(LnSource));
    L.ln_rows_large = take((size_t)(2 * c.large.n_layers + 1) * 4 * c.large.d_model * 2);
    L.ln_rows_small = take((size_t)(2 * c.small.n_layers + 1) * 4 * c.small.d_model * 2);
    L.ln_stats = take(RD * ((std::max(c.large.d_model, c.small.d_model) + 31) / 32) * 8);
    L.ln_ref = take(2 * RD * 4);
    L.total = off;
    return L;
}

int n_weight_ptrs(const tandem_config& c) {
    const int per_t = c.ff_tandem_kind == TANDEM_FF_LINEAR ? 1 : 2;
    return (5 + 10 * c.large.n_layers) + (5 + 10 * c.small.n_layers) + per_t * c.small.n_layers;
}

enum { W_LN1G = 0, W_LN1B, W_WQ, W_WK, W_WV, W_WO, W_LN2G, W_LN2B, W_W1, W_W2 };
inline const void* w_emb(const tandem_ctx& c, const Model& m) { return c.w[m.wbase]; }
inline const void* w_pos(const tandem_ctx& c, const Model& m) { return c.w[m.wbase + 1]; }
inline const void* w_layer(const tandem_ctx& c, const Model& m, int l, int k) { return c.w[m.wbase + 2 + 10 * l + k]; }
inline const void* w_tail(const tandem_ctx& c, const Model& m, int k) { return c.w[m.wbase + 2 + 10 * m.d.n_layers + k]; }

inline int wi_layer(const Model& m, int l, int k) { return m.wbase + 2 + 10 * l + k; }
inline int wi_tail(const Model& m, int k) { return m.wbase + 2 + 10 * m.d.n_layers + k; }
inline int wi_tandem(const tandem_ctx& c, int j, int k) { return c.tbase + (c.cfg.ff_tandem_kind == TANDEM_FF_LINEAR ? j : 2 * j + k); }

// A linear map given by the indices of up to three weight matrices stacked along the output features.
// (the first matrix has seg_rows0 rows, the others seg_rows each: queries next to narrower keys / values)
struct Lin { int i0, i1, i2, seg_rows0, seg_rows, K; };
inline Lin lin1(int i0, int rows, int K) { Lin l = {i0, -1, -1, rows, rows, K}; return l; }
inline Lin lin3(int i0, int i1, int i2, int rows0, int rows, int K) { Lin l = {i0, i1, i2, rows0, rows, K}; return l; }
inline int lin_n(const Lin& l) { return l.seg_rows0 + ((l.i1 >= 0) + (l.i2 >= 0)) * l.seg_rows; }

template <typename P> P* at(tandem_ctx& c, size_t off) { return reinterpret_cast<P*>(c.arena + off); }

constexpr int MAX_DEVICES = 64;
int cur_dev() {   // opt-in shared-memory sizes are per device
    int d = 0;
    cudaGetDevice(&d);
    return (d >= 0 && d < MAX_DEVICES) ? d : 0;
}

// ---------------------------------------------------------------------------------------------------
// launch helpers
// ---------------------------------------------------------------------------------------------------

// Opt-in dynamic shared memory of a kernel, requested once per device (`done`: one bit per device, one word per
// kernel instantiation).  The attribute call is idempotent, so two threads racing to be first is harmless.
template <typename K>
void ensure_dyn_smem(K kernel, size_t bytes, std::atomic<unsigned long long>& done) {
    const unsigned long long bit = 1ull << cur_dev();
    if (done.load(std::memory_order_acquire) & bit) return;
    cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    done.fetch_or(bit, std::memory_order_release);
}

// Multiprocessors of the current device (asked once per device).
int sm_count() {
    static std::atomic<int> cache[MAX_DEVICES];
    const int dev = cur_dev();
    int n = cache[dev].load(std::memory_order_relaxed);
    if (n > 0) return n;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1) n = 1;
    cache[dev].store(n, std::memory_order_relaxed);
    return n;
}

// ---------------------------------------------------------------------------------------------------
// tensor-core GEMMs: tensor maps and launches
// ---------------------------------------------------------------------------------------------------

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// The driver's tensor-map encoder, looked up through the runtime (the library does not link libcuda).
EncodeTiledFn tmap_encoder() {
    static EncodeTiledFn fn = []() -> EncodeTiledFn {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) != cudaSuccess) return nullptr;
        return q == cudaDriverEntryPointSuccess ? reinterpret_cast<EncodeTiledFn>(p) : nullptr;
    }();
    return fn;
}

// bf16 matrix [rows][cols] with leading dimension ld (elements), tiles of box_rows (128 by default) rows x 64 columns,
// 128-byte swizzle.  base 16-byte aligned, ld a multiple of 8.
bool make_tmap_bf16(CUtensorMap* tm, const void* base, uint64_t rows, uint64_t cols, uint64_t ld, uint32_t box_rows = 128) {
    EncodeTiledFn enc = tmap_encoder();
    if (!enc) return false;
    const cuuint64_t dims[2] = {cols, rows};
    const cuuint64_t strides[1] = {ld * 2};
    const cuuint32_t box[2] = {64, box_rows};
    const cuuint32_t estr[2] = {1, 1};
    return enc(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Two planes [rows][cols], one behind the other, tiles of 16 rows x 64 columns of both.
bool make_tmap_planes(CUtensorMap* tm, const void* base, uint64_t rows, uint64_t cols) {
    EncodeTiledFn enc = tmap_encoder();
    if (!enc) return false;
    const cuuint64_t dims[3] = {cols, rows, 2};
    const cuuint64_t strides[2] = {cols * 2, rows * cols * 2};
    const cuuint32_t box[3] = {64, 16, 2};
    const cuuint32_t estr[3] = {1, 1, 1};
    return enc(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// make_tmap_bf16, remembered: a tensor map depends on nothing but its arguments, and the stand-alone calls get the same weight matrices again
// and again (an encoding costs the host about 0.4 us, which the first call on a matrix pays).  128 maps per thread, 24 KB, the last one to hash to a place stays.
bool cached_tmap_bf16(CUtensorMap* tm, const void* base, uint64_t rows, uint64_t cols) {
    struct Entry { const void* base; uint64_t rows, cols; CUtensorMap tm; };
    static thread_local std::vector<Entry> cache;
    if (cache.empty()) cache.resize(128, Entry{nullptr, 0, 0, {}});
    const uint64_t h = splitmix64(reinterpret_cast<uintptr_t>(base) ^ (rows << 40) ^ (cols << 20));
    Entry& e = cache[h & 127];
    if (e.base != base || e.rows != rows || e.cols != cols) {
        e.base = nullptr;
        if (!make_tmap_bf16(&e.tm, base, rows, cols, cols)) return false;
        e.base = base; e.rows = rows; e.cols = cols;
    }
    *tm = e.tm;
    return true;
}

struct TcW {              // up to three weight matrices stacked along the output features
    CUtensorMap tm[3];
    CUtensorMap part[3];  // the same in boxes of 32 rows (prompt pass)
    int n_segs, seg_rows0, seg_rows, K;   // rows of the first segment, rows of every further one
};
inline int tcw_n(const TcW& w) { return w.seg_rows0 + (w.n_segs - 1) * w.seg_rows; }
struct TcScratch {
    int* err;                  // where a bounded wait that ran out records its code (nullable)
    unsigned poll_limit = 0;   // 0: the kernels' default
    int withhold_weights = 0;  // test hook, see TcDecodeArgs
    int wait_first = 0;        // the launch may follow kernels that write its weights, see TcDecodeArgs
    int rows_early = 0;        // the row arrays are older than the preceding kernel, see TcDecodeArgs
};

TcW tcw3(const tandem_ctx& c, int i0, int i1, int i2, int seg_rows0, int seg_rows, int K) {
    TcW w;
    w.tm[0] = c.wmap[i0];
    w.tm[1] = c.wmap[i1 >= 0 ? i1 : i0];
    w.tm[2] = c.wmap[i2 >= 0 ? i2 : i0];
    w.part[0] = c.wpart[i0];
    w.part[1] = c.wpart[i1 >= 0 ? i1 : i0];
    w.part[2] = c.wpart[i2 >= 0 ? i2 : i0];
    w.n_segs = 1 + (i1 >= 0) + (i2 >= 0);
    w.seg_rows0 = seg_rows0; w.seg_rows = seg_rows; w.K = K;
    return w;
}
TcW tcw(const tandem_ctx& c, int i0, int i1, int i2, int seg_rows, int K) { return tcw3(c, i0, i1, i2, seg_rows, seg_rows, K); }

TcScratch tc_scratch(tandem_ctx& c) {
    TcScratch s;
    s.err = c.st.counters ? c.st.counters + 2 : nullptr;
    return s;
}

template <typename... KArgs, typename... Args>
void launch_ex(tandem_ctx& c, bool pdl, int cluster, void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, Args&&... args) {
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = c.stream;
    cudaLaunchAttribute attr[2];
    int n = 0;
    const bool plain = c.next_launch_plain;
    c.next_launch_plain = false;
    if (pdl && c.use_pdl && !plain) {
        attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[n].val.programmaticStreamSerializationAllowed = 1;
        ++n;
    }
    if (cluster > 1) {   // consecutive blocks along x form a thread-block cluster
        attr[n].id = cudaLaunchAttributeClusterDimension;
        attr[n].val.clusterDim.x = (unsigned)cluster; attr[n].val.clusterDim.y = 1; attr[n].val.clusterDim.z = 1;
        ++n;
    }
    cfg.attrs = attr;
    cfg.numAttrs = n;
    cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
    c.launches++;
}

// Token rows that lie in two bf16 planes (PRO_TMA), and the LayerNorm that is applied to them (PRO_LNT).
struct TcRows {
    const CUtensorMap* map = nullptr;
    const CUtensorMap* ln_map = nullptr;
    int ln_row = 0;                        // the LayerNorm's first row there
    const float2* ln_stats = nullptr;      // [rows][ln_groups]
    int ln_groups = 0;
    const float* ln_ref = nullptr;         // [rows] each
    float* ln_mean = nullptr;
};

template <int NB, int PRO, int EPI>
void launch_tc_decode_nb(tandem_ctx& c, const TcDecodeArgs& a, const TcW& w, int units, const TcRows& x) {
    using C = TcdCfg<NB, PRO == PRO_LNT>;
    static std::atomic<unsigned long long> attr_done{0};
    ensure_dyn_smem(gemm_tc_decode_kernel<NB, PRO, EPI>, C::SMEM_BYTES, attr_done);
    launch_ex(c, true, a.splits, gemm_tc_decode_kernel<NB, PRO, EPI>, dim3(units), dim3(TCD_THREADS), (size_t)C::SMEM_BYTES, a, w.tm[0], w.tm[1], w.tm[2],
              x.map ? *x.map : w.tm[0], x.ln_map ? *x.ln_map : w.tm[0]);
}

// y = prologue(x) W^T for few rows on the tensor cores, streaming W once per group of up to 64 rows (one group in
// every benchmark configuration; more rows than that re-read the weights per group, with unchanged arithmetic).
template <int PRO, int EPI>
void launch_tc_decode(tandem_ctx& c, const TcScratch& sc, const void* x, int ldx, const void* ln_g, const void* ln_b, int rows,
                      const TcW& w, bool stream_weights, const EpiArgs& e, float* amax_val = nullptr, int* amax_idx = nullptr,
                      int amax_stride = 0, const TcRows& xr = TcRows()) {
    if (rows <= 0) return;
    TcDecodeArgs a;
    memset(&a, 0, sizeof(a));
    a.x = x; a.ldx = ldx; a.ln_g = static_cast<const float*>(ln_g); a.ln_b = static_cast<const float*>(ln_b);
    a.rows = rows;
    a.ln_row = xr.ln_row; a.ln_groups = xr.ln_groups; a.ln_stats = xr.ln_stats; a.ln_ref = xr.ln_ref; a.ln_mean = xr.ln_mean;
    a.K = w.K; a.N = tcw_n(w); a.seg_rows0 = w.seg_rows0; a.tiles0 = cdiv(w.seg_rows0, 128);
    a.seg_rows = w.seg_rows; a.tiles_per_seg = cdiv(w.seg_rows, 128);
    const int tiles = a.tiles0 + (w.n_segs - 1) * a.tiles_per_seg, KB = cdiv(w.K, 64);
    // K-slices per tile = cluster size: the smallest power of two that puts tiles * S CTAs at or above one per
    // multiprocessor, at most 8 and at most one per 64-element K-block; four instead of eight where those already reach a
    // quarter of the multiprocessors with slices of four K-blocks or fewer (they fit the ring, and only 15 clusters of
    // eight run beside each other before two CTAs share a multiprocessor, but 33 of four).  A layer's four GEMMs with four
    // slices in both wide ones against eight: 1024 wide, one row 12.5 -> 11.9 us, eight rows 13.9 -> 13.1; 512 wide 9.9 -> 9.5 and
    // 11.8 -> 11.4.  The residual GEMMs (a quarter of the tiles or a slice beyond the ring) are 2 to 10 % slower with four.
    // The head GEMM keeps whole tiles.
    int S = 1;
    if (EPI != EPI_ARGMAX)
        while (S < 8 && 2 * S <= KB && tiles * S < c.n_sms && !(S == 4 && KB <= 16 && 16 * tiles >= c.n_sms)) S *= 2;
    a.splits = S;
    a.stream_weights = stream_weights ? 1 : 0;
    a.err_flag = sc.err;
    a.poll_limit = sc.poll_limit;
    a.withhold_weights = sc.withhold_weights;
    a.wait_first = sc.wait_first;
    a.rows_early = sc.rows_early && e.row_seq ? 1 : 0;
    a.release_early = (size_t)a.N * (size_t)w.K * 2 <= ((size_t)16 << 20) ? 1 : 0;
    a.amax_val = amax_val; a.amax_idx = amax_idx; a.amax_stride = amax_stride;
    a.e = e;
    const double xsz = PRO == PRO_BF16 ? 2 : 4, osz = EPI == EPI_QKV || EPI == EPI_KV || EPI == EPI_STORE ? 2.0 : 4.0;
    const int units = tiles * S;
    for (int r0 = 0; r0 < rows; r0 += 64) {
        const int nr = std::min(64, rows - r0);
        TcDecodeArgs g = a;
        tcd_shift_rows<PRO, EPI>(g, r0, nr);
        if (r0 > 0) g.wait_first = 0;
        ProfScope ps(c, PC_GEMM_TC_DECODE, 2.0 * a.N * w.K + nr * (w.K * xsz + a.N * osz));
        if (nr <= 16) launch_tc_decode_nb<16, PRO, EPI>(c, g, w, units, xr);
        else if (nr <= 32) launch_tc_decode_nb<32, PRO, EPI>(c, g, w, units, xr);
        else if (nr <= 48) launch_tc_decode_nb<48, PRO, EPI>(c, g, w, units, xr);
        else launch_tc_decode_nb<64, PRO, EPI>(c, g, w, units, xr);
    }
}

// Which kernel the product of a prompt or teacher-forced pass takes, from estimated times in us.  Both are bound by their operands' way
// from L2 into the multiprocessors, so the estimates are a start-up time, plus per K-block what a CTA's share of it takes, plus what an
// epilogue leaves uncovered.  They are there to choose by: single estimates are off by up to a half (residual adds of many rows), the choice is
// within a tenth of the best kernel but for a few.  us measured, split kernel with 1 / 2 / 4 K-slices | pair kernel, * the choice:
//   one plane
//    511 x 3072 x 1024          7.8*  8.3  16.1 |  8.1       511 x 1024 x 4096, residual  32.1  17.5  11.3* | 17.4
//   1023 x 1024 x 1024, resid. 17.5  10.3  11.8 |  7.2*     1500 x 1024 x 4096, residual  37.3  32.1  27.7  | 20.5*
//   1023 x 4096 x 1024, GELU   12.3* 20.0   -   | 16.5       511 x 4096 x 4096, residual  42.4  38.9  33.1  | 20.2*
//    255 x 12288 x 4096        32.3  37.0   -   | 28.3*     2047 x 2048 x 2048, residual  40.9  56.1   -    | 18.9*
//   two planes (of 120 sizes, 64-3000 rows of the small and the medium pair, seven are more than a tenth off, the worst ones at the end; kernels one
//   by one under the profiler, caches warm)
//    256 x 3072 x 1024         13.7  11.4* 14.0 | 11.4       769 x 1024 x 4096, residual  56.3  33.5  23.4* | 26.8
//   1500 x 4096 x 1024, GELU   39.3  43.7  69.2 | 31.3*     1023 x 1024 x 1024, residual  28.1  17.6  15.6  | 12.2*
//   3000 x 8192 x 2048, GELU  183.4 213.7 304.1 | 132.1*     769 x 2048 x 8192, residual 108.1  83.4  67.4  | 56.9*
//   2047 x 4096 x 1024, GELU   41.9* 57.1  88.4 | 36.2      1500 x 768 x 3072, residual   49.2  28.8  29.6* | 21.8
struct TiledPlan { bool pair; int slices, whole, parts; };
TiledPlan tiled_plan(int n_sms, int epi, bool planes, int tiles128, int tiles256, int KB) {
    TiledPlan best = {false, 1, 0, 1};
    double least = 0.0;
    // Split kernel: the K range of a tile dealt to S CTAs (four K-blocks each at least: fewer would not pay for the exchange); one CTA per
    // multiprocessor waits for its operands' latency, two share the bandwidth, and slices that do not all run at the same time
    // wait for each other.
    for (int S = 1; S <= 4; S *= 2) {
        const int n = tiles128 * S;
        if (S > 1 && (epi == EPI_SCORE || KB < 4 * S)) break;
        const double per_kb = n <= n_sms ? (planes ? 0.60 : 0.33) : (planes ? 0.85 : 0.46) * cdiv(n, 2 * n_sms);
        double us = 3.0 + per_kb * cdiv(KB, S);
        if (S > 1) us += 1.2 + (n > 2 * n_sms ? 12.0 : (n > n_sms ? 4.0 : 0.0));
        if (epi == EPI_RESID) us += S == 1 ? 7.0 : (S == 2 ? 4.0 : 1.5);   // (the stream's old values, a row per thread: more columns to a CTA)
        if (epi == EPI_GELU) us += 2.0;
        if (S == 1 || us < least) { least = us; best.slices = S; }
    }
    // Pair kernel: full rounds of all pairs, then the rest in parts (1, 2 or 4) as far as one round holds them.
    const int n_pairs = n_sms / 2;
    if (n_pairs > 0) {
        const int rest = tiles256 % n_pairs, rounds = tiles256 / n_pairs;
        const int parts = epi == EPI_SCORE ? 1 : (rest * 4 <= n_pairs ? 4 : (rest * 2 <= n_pairs ? 2 : 1));
        const double whole_kb = planes ? 0.75 : 0.42, part_kb = parts == 4 ? (planes ? 0.32 : 0.24) : (parts == 2 ? (planes ? 0.42 : 0.27) : whole_kb);
        double us = 4.2 + KB * (rounds * whole_kb + (rest > 0 ? part_kb : 0.0));
        if (epi == EPI_RESID) us += 0.5;
        if (epi == EPI_GELU) us += 5.0;
        if (us < least || tiles256 >= 2 * n_pairs) { best.pair = true; best.whole = tiles256 - rest; best.parts = parts; }
    }
    return best;
}

// What the output head of a teacher-forced pass leaves per row and SCORE_TILE features instead of the logits.
struct TcScore { float* val; int* idx; float* sum; int stride; const int* truth; float* truth_val; const int* keep; float* kept; };

// y = x W^T for many rows on the tensor cores; x bf16 [M][ldx].  PL: x as two planes, the remainders lo_row rows behind the values.
template <int EPI, bool PL>
tandem_status launch_tc_tiled(tandem_ctx& c, const bf16* x, int ldx, int M, const TcW& w, const EpiArgs& e, int* err, int lo_row = 0, const TcScore& sc = TcScore()) {
    if (M <= 0) return TANDEM_OK;
    CUtensorMap tmx;
    if (!make_tmap_bf16(&tmx, x, PL ? (uint64_t)lo_row + M : (uint64_t)M, (uint64_t)w.K, (uint64_t)ldx)) {
        snprintf(g_cuda_err, sizeof(g_cuda_err), "cuTensorMapEncodeTiled failed for an activation buffer");
        return TANDEM_ERR_CUDA;
    }
    TcTiledArgs a;
    memset(&a, 0, sizeof(a));
    a.M = M; a.K = w.K; a.N = tcw_n(w); a.seg_rows0 = w.seg_rows0; a.seg_rows = w.seg_rows;
    a.err_flag = err; a.e = e; a.lo_row = lo_row;
    if (EPI == EPI_SCORE) { a.tile_max = sc.val; a.tile_idx = sc.idx; a.tile_sum = sc.sum; a.tile_stride = sc.stride; a.truth = sc.truth; a.truth_val = sc.truth_val; a.keep = sc.keep; a.kept = sc.kept; }
    const int n_sms = std::max(1, c.n_sms);
    auto feature_tiles = [&](int width) {
        a.tiles0 = cdiv(w.seg_rows0, width);
        a.tiles_per_seg = cdiv(w.seg_rows, width);
        a.tiles_n = a.tiles0 + (w.n_segs - 1) * a.tiles_per_seg;
        return (long long)a.tiles_n * a.tiles_m;
    };
    ProfScope ps(c, PC_GEMM_TC_TILED, 2.0 * M * (double)a.N * w.K);   // flops
    a.tiles_m = cdiv(M, 128);
    const int tiles128 = (int)feature_tiles(TCS_BN);
    a.tiles_m = cdiv(M, 256);
    const int tiles256 = (int)feature_tiles(TCP_BN);
    const TiledPlan plan = tiled_plan(n_sms, EPI, PL, tiles128, tiles256, cdiv(w.K, 64));
    if (plan.pair) {
        a.whole = plan.whole; a.parts = plan.parts;
        static std::atomic<unsigned long long> attr_done{0};
        ensure_dyn_smem(gemm_tc_pair_kernel<EPI, PL>, TcpCfg<PL>::SMEM_BYTES, attr_done);
        const int items = plan.whole + (tiles256 - plan.whole) * plan.parts;
        launch_ex(c, true, 2, gemm_tc_pair_kernel<EPI, PL>, dim3(2 * std::min(items, n_sms / 2)), dim3(TCP_THREADS), (size_t)TcpCfg<PL>::SMEM_BYTES, a, tmx, w.tm[0], w.tm[1], w.tm[2],
                  w.part[0], w.part[1], w.part[2]);
        return TANDEM_OK;
    }
    a.tiles_m = cdiv(M, 128);
    feature_tiles(TCS_BN);
    a.splits = plan.slices;
    static std::atomic<unsigned long long> attr_done{0};
    ensure_dyn_smem(gemm_tc_split_kernel<EPI, PL>, TcsCfg<PL>::SMEM_BYTES, attr_done);
    launch_ex(c, true, plan.slices, gemm_tc_split_kernel<EPI, PL>, dim3(tiles128 * plan.slices), dim3(TCS_THREADS), (size_t)TcsCfg<PL>::SMEM_BYTES, a, tmx, w.tm[0], w.tm[1], w.tm[2]);
    return TANDEM_OK;
}

WSegs segs_of(const tandem_ctx& c, const Lin& l) {
    WSegs s;
    s.w[0] = c.w[l.i0];
    s.w[1] = l.i1 >= 0 ? c.w[l.i1] : nullptr;
    s.w[2] = l.i2 >= 0 ? c.w[l.i2] : nullptr;
    s.seg_rows0 = l.seg_rows0;
    s.seg_rows = l.seg_rows;
    return s;
}

// fp32, few rows.  ln_g / ln_b non-null: LayerNorm of the rows first (fused; K <= GS_KC, see fp32_few_rows).
template <int MT, int NC, int FORM, int EPI>
void launch_rows_as(tandem_ctx& c, const float* x, int ldx, int M, int K, const WSegs& ws, int N, const float* ln_g, const float* ln_b, const EpiArgs& e,
                    float* amax_val, int* amax_idx) {
    static std::atomic<unsigned long long> attr_done{0};
    ensure_dyn_smem(gemm_rows_kernel<MT, NC, FORM, EPI>, (size_t)MT * GS_KC * sizeof(float), attr_done);
    launch_ex(c, true, 1, gemm_rows_kernel<MT, NC, FORM, EPI>, dim3(cdiv(N, GS_WARPS * NC), cdiv(M, MT)), dim3(GS_THREADS),
              (size_t)MT * std::min(K, GS_KC) * sizeof(float), x, ldx, M, K, ws, N, ln_g, ln_b, e, amax_val, amax_idx, c.amax_tiles);
}
template <bool LN, int EPI>
void launch_rows(tandem_ctx& c, const float* x, int ldx, int M, const Lin& l, const EpiArgs& e, const void* ln_g = nullptr, const void* ln_b = nullptr,
                 float* av = nullptr, int* ai = nullptr) {
    if (M <= 0) return;
    const WSegs ws = segs_of(c, l);
    const int N = lin_n(l), K = l.K;
    const float *g = static_cast<const float*>(ln_g), *b = static_cast<const float*>(ln_b);
    ProfScope ps(c, PC_GEMM_SMALLM, ((double)N * K + (double)M * K + (double)M * N) * sizeof(float));
    const bool wide = rows_columns(N) == 4;
    auto go = [&](auto mt, auto nc) {
        constexpr int MT = decltype(mt)::value, NC = decltype(nc)::value;
        if constexpr (!LN) launch_rows_as<MT, NC, ROWS_PLAIN, EPI>(c, x, ldx, M, K, ws, N, g, b, e, av, ai);
        else if (K <= rows_ln_regs_max(NC)) launch_rows_as<MT, NC, ROWS_LN_REGS, EPI>(c, x, ldx, M, K, ws, N, g, b, e, av, ai);
        else launch_rows_as<MT, NC, ROWS_LN_SMEM, EPI>(c, x, ldx, M, K, ws, N, g, b, e, av, ai);
    };
    auto columns = [&](auto mt) { if (wide) go(mt, std::integral_constant<int, 4>()); else go(mt, std::integral_constant<int, 1>()); };
    if (M <= 1) columns(std::integral_constant<int, 1>());
    else if (M <= 4) columns(std::integral_constant<int, 4>());
    else columns(std::integral_constant<int, 8>());
}

// y = x W^T with a fused epilogue for many rows: the prompt-pass kernels (tensor cores for bf16).
template <typename T, int EPI>
void launch_gemm(tandem_ctx& c, const T* x, int ldx, int M, const Lin& l, const EpiArgs& e) {
    if (M <= 0) return;
    if constexpr (sizeof(T) == 2) {
        if (launch_tc_tiled<EPI, false>(c, x, ldx, M, tcw3(c, l.i0, l.i1, l.i2, l.seg_rows0, l.seg_rows, l.K), e, c.st.counters + 2) != TANDEM_OK)
            c.setup_failed = true;
    } else {
        const int N = lin_n(l), K = l.K;
        dim3 grid(cdiv(N, GT_BN), cdiv(M, GT_BM));
        ProfScope ps(c, PC_GEMM_TILED, 2.0 * M * (double)N * K);   // flops, not bytes: this one is compute-bound
        gemm_tiled_kernel<T, EPI><<<grid, GT_THREADS, 0, c.stream>>>(x, ldx, M, K, segs_of(c, l), N, e);
        c.launches++;
    }
}

template <typename T, int DH>
void launch_attn_dh(tandem_ctx& c, const AttnArgs& a, int groups, bool loop, int n_chunks, double kv_bytes) {
    static std::atomic<unsigned long long> attr_done_loop{0};
    if (loop) {
        ensure_dyn_smem(attn_kernel<T, DH, true>, attn_smem_bytes<T, DH>(), attr_done_loop);
        ProfScope ps(c, PC_ATTN_PROMPT, kv_bytes);
        launch_ex(c, true, 1, attn_kernel<T, DH, true>, dim3(1, a.n_heads, groups), dim3(ATT_THREADS), attn_smem_bytes<T, DH>(), a);
        return;
    }
    if constexpr (sizeof(T) == 4) {   // (the bf16 decode passes have their own kernel)
        static std::atomic<unsigned long long> attr_done_split{0};
        ensure_dyn_smem(attn_kernel<T, DH, false>, attn_smem_bytes<T, DH>(), attr_done_split);
        ProfScope ps(c, PC_ATTN_SPLIT, kv_bytes);
        launch_ex(c, true, 1, attn_kernel<T, DH, false>, dim3(n_chunks, a.n_heads, groups), dim3(ATT_THREADS), attn_smem_bytes<T, DH>(), a);
    }
}

template <typename T>
void launch_attn(tandem_ctx& c, int d_head, const AttnArgs& a, int groups, bool loop, int n_chunks, double kv_bytes) {
    if (d_head == 32) launch_attn_dh<T, 32>(c, a, groups, loop, n_chunks, kv_bytes);
    else if (d_head == 64) launch_attn_dh<T, 64>(c, a, groups, loop, n_chunks, kv_bytes);
    else launch_attn_dh<T, 128>(c, a, groups, loop, n_chunks, kv_bytes);
}

// bf16 decode attention: one cluster of `cl` CTAs per (sequence, group of query heads); no scratch.
template <int DH, int NT, int MODE>
void launch_attn_decode_as(tandem_ctx& c, const AttnArgs& a, dim3 grid, int cl) {
    static std::atomic<unsigned long long> attr_done{0};
    ensure_dyn_smem(attn_decode_kernel<DH, NT, MODE>, attn_decode_smem_bytes<DH>(), attr_done);
    launch_ex(c, true, cl, attn_decode_kernel<DH, NT, MODE>, grid, dim3(ATD_THREADS), attn_decode_smem_bytes<DH>(), a);
}
template <int DH>
void launch_attn_decode_dq(tandem_ctx& c, const AttnArgs& a, int groups, int cl, bool pass, double kv_bytes) {
    const int gpc = std::max(1, a.heads_per_cta);
    const bool narrow = gpc * a.nq <= 8;
    const dim3 grid(cl, a.n_heads / gpc, groups);
    ProfScope ps(c, PC_ATTN_SPLIT, kv_bytes);
    if (pass) {
        AttnArgs w = a;
        w.units = groups * (a.n_heads / gpc);
        // Up to four warps share a unit's keys as long as all warps run at the same time with two CTAs per multiprocessor: one sequence of 257 tokens
        // through the small pair 1226 -> 1165 us with four (1185 with two), of 64 tokens 988 -> 967.  Beyond that the merge only
        // adds work: eight of 400 tokens 3325 us with one, 3530 with two, 3655 with four.  (128-wide heads with sixteen columns fit once: 400 / 512 rows
        // of 8 heads a launch 36.1 / 40.0 us with two, 35.9 / 39.5 with four in two rounds, so the line is the same.)
        while (w.log_parts < 2 && w.units * 2 << w.log_parts <= 2 * ATD_WARPS * c.n_sms) ++w.log_parts;
        const dim3 warps(cdiv(w.units << w.log_parts, ATD_WARPS));
        if (narrow) launch_attn_decode_as<DH, 1, ATD_PASS>(c, w, warps, 1); else launch_attn_decode_as<DH, 2, ATD_PASS>(c, w, warps, 1);
    }
    else if (cl == 1) { if (narrow) launch_attn_decode_as<DH, 1, ATD_ALONE>(c, a, grid, cl); else launch_attn_decode_as<DH, 2, ATD_ALONE>(c, a, grid, cl); }
    else if (narrow) launch_attn_decode_as<DH, 1, ATD_CLUSTERED>(c, a, grid, cl);
    else launch_attn_decode_as<DH, 2, ATD_CLUSTERED>(c, a, grid, cl);
}
// Clusters of `cl` decode-attention CTAs that the device can run at the same time (asked once per device and size).  It is
// less than the multiprocessors would suggest, because a cluster has to fit into one GPC: with 148 multiprocessors and one
// 128-wide CTA on each, 33 clusters of four and 15 of eight (64-wide, two CTAs each: 71 and 33).
template <int DH>
int attn_max_clusters(int cl) {
    static std::atomic<int> cache[MAX_DEVICES][4];
    std::atomic<int>& slot = cache[cur_dev()][cl == 8 ? 3 : (cl == 4 ? 2 : (cl == 2 ? 1 : 0))];
    int n = slot.load(std::memory_order_relaxed);
    if (n > 0) return n;
    static std::atomic<unsigned long long> attr_done{0};
    ensure_dyn_smem(attn_decode_kernel<DH, 2, ATD_CLUSTERED>, attn_decode_smem_bytes<DH>(), attr_done);
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3(cl); cfg.blockDim = dim3(ATD_THREADS); cfg.dynamicSmemBytes = attn_decode_smem_bytes<DH>();
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = (unsigned)cl; attr.val.clusterDim.y = 1; attr.val.clusterDim.z = 1;
    cfg.attrs = &attr; cfg.numAttrs = 1;
    if (cudaOccupancyMaxActiveClusters(&n, attn_decode_kernel<DH, 2, ATD_CLUSTERED>, &cfg) != cudaSuccess || n < 1) n = 1;
    slot.store(n, std::memory_order_relaxed);
    return n;
}
// Cluster size, 1, 2, 4 or 8: the one with the least rounds of resident clusters x (a CTA's share of the context + what a CTA
// costs apart from it, about two and a half chunks).  It depends on the number of sequences and key/value heads only (the
// share is taken of 24 chunks, 3072 positions), so every pass of a run (block or one-row) cuts the context the same way.  The
// stand-alone call takes the same rule; its length is not looked at.
// Two sequences x 8 key/value heads x 128, blocks of six rows: 35-41 us with eight (16 clusters where 15 fit), 18.6 us with
// four.  20 sequences x 16 heads x 64 x 3000 positions, 320 clusters where 296 CTAs fit: 61 us with one, 52 with two, 49 with
// four; 32 x 16 x 64 x 8194: 160 us with one, 166 with two.  (Sizes in between measured 3 % slower per iteration at batch 8: a
// cluster of three merges more states than its extra CTAs save.)
// In a decode pass (beside others) a cluster of eight, which needs eight places in one GPC, finds about half of them taken by
// the kernels before and behind it: four sequences x 8 heads x 64, 32 clusters where 33 fit on an empty GPU, a layer of the 512-wide model 14.5 us with eight, 13.1 with four.
int attn_cluster_size(long long clusters, int d_head, bool alone) {
    int best = 1;
    double least = 0.0;
    for (int cl = 1; cl <= ATD_CLUSTER; cl *= 2) {
        int fit = d_head == 32 ? attn_max_clusters<32>(cl) : (d_head == 64 ? attn_max_clusters<64>(cl) : attn_max_clusters<128>(cl));
        if (cl == 8 && !alone) fit = std::max(1, fit / 2);
        const double cost = (double)((clusters + fit - 1) / fit) * (24.0 / cl + 2.5);
        if (cl == 1 || cost < least) { least = cost; best = cl; }
    }
    return best;
}
// pass: a teacher-forced pass, which has a warp per group of rows and head.
void launch_attn_decode(tandem_ctx& c, int d_head, const AttnArgs& a0, int groups, double kv_bytes, bool pass = false) {
    AttnArgs a = a0;
    // Grouped-query attention: the query heads of one key/value head ride in one CTA as far as the 16-row tile has
    // room (heads * queries per block <= 16; a power of two that divides the group).  The cluster size is taken
    // from the key/value heads, which do not depend on the number of queries: a block pass and a one-row pass cut
    // the context the same way.
    const int n_kv = a.n_kv_heads > 0 ? a.n_kv_heads : a.n_heads;
    const int group = a.n_heads / n_kv;
    int gpc = 1;
    while (gpc * 2 <= group && group % (gpc * 2) == 0 && gpc * 2 * a.nq <= ATT_NQ) gpc *= 2;
    a.heads_per_cta = gpc;
    const int cl = pass ? 1 : attn_cluster_size((long long)groups * n_kv, d_head, a.wait_first != 0);
    if (d_head == 32) launch_attn_decode_dq<32>(c, a, groups, cl, pass, kv_bytes);
    else if (d_head == 64) launch_attn_decode_dq<64>(c, a, groups, cl, pass, kv_bytes);
    else launch_attn_decode_dq<128>(c, a, groups, cl, pass, kv_bytes);
}

// raw (bf16 only, nullable): also leaves a bf16 copy of the rows as they are.  PL: both as two planes, the remainders `lo` elements behind.
template <typename T, bool PL = false>
void launch_layernorm(tandem_ctx& c, int M, const float* x, const void* gain, const void* bias, T* out, int d, bf16* raw = nullptr, size_t lo = 0) {
    ProfScope ps(c, PC_LAYERNORM, (double)M * d * (4.0 + (PL ? 2 : 1) * (sizeof(T) + (raw ? 2.0 : 0.0))));
    const float *g = static_cast<const float*>(gain), *b = static_cast<const float*>(bias);
    // A warp per row beyond 256 rows, which no decode pass has (those keep one order of the sums whatever their rows); for a few rows
    // a block each is the shorter chain (40 rows of 768 between the two products of a stand-alone projection 11.7 us, 11.9 with a warp each).
    auto by_warps = [&](auto kernel) { launch_ex(c, true, 1, kernel, dim3(std::min(cdiv(M, 4), 4 * c.n_sms)), dim3(128), 0, x, g, b, out, d, M, raw, lo); };
    if (M > 256 && d <= 1024) by_warps(layernorm_warp_kernel<T, PL, 8>);
    else if (M > 256 && d <= LNW_MAX) by_warps(layernorm_warp_kernel<T, PL, 16>);
    else
        launch_ex(c, true, 1, layernorm_rows_kernel<T, PL>, dim3(std::min(M, 4 * std::max(1, c.n_sms))), dim3(128), 0, x, g, b, out, d, M, raw, lo);
}

// Describes the rows of one pass.
struct Rows {
    int M;            // rows
    int groups;       // attention groups
    int nq;           // rows per group when group arrays are not used (decode)
    bool decode;      // decode kernels (split attention, streaming GEMM) or prompt kernels
    int n_chunks;     // split attention grid size along the context
    double kv_positions;   // context positions read by one attention launch, summed over sequences (accounting only)
    bool whole_pass = false;            // a teacher-forced pass (see forced_pass)
    int plane = 0;                      // ... rows between its planes of values and of remainders
    bool apart = false;                 // ... whose projections' buffers (but their input) lie apart from what the large model's layers write
    const int *grp = nullptr, *grp_pos = nullptr;        // ... its attention groups, see AttnArgs::pass_grp
    bf16 *own_k = nullptr, *own_v = nullptr;             // ... the small model's keys / values of its own [kv head][row of the pass][d_head], beside the large-derived ones in the cache
};

template <typename T>
T* kv_ptr(tandem_ctx& c, const Model& m, int layer, int which) {
    return at<T>(c, m.kv_off) + ((size_t)layer * 2 + which) * m.kv_layer_elems;
}

EpiArgs epi_plain(void* out, int ldo) {
    EpiArgs e; memset(&e, 0, sizeof(e)); e.out = out; e.ldo = ldo; return e;
}

template <typename T>
EpiArgs epi_cache(tandem_ctx& c, const Model& m, int layer, void* q_out) {
    EpiArgs e; memset(&e, 0, sizeof(e));
    e.out = q_out; e.ldo = m.d.d_model;
    e.kcache = kv_ptr<T>(c, m, layer, 0); e.vcache = kv_ptr<T>(c, m, layer, 1);
    e.row_seq = at<int>(c, c.lay.row_seq); e.row_pos = at<int>(c, c.lay.row_pos);
    e.n_heads = m.kv_heads; e.d_head = m.d.d_model / m.d.n_heads; e.t_max = c.cfg.max_seq;
    e.seg0 = q_out ? m.d.d_model : m.d_kv; e.seg = m.d_kv;   // with queries: [d_model | d_kv | d_kv]; keys / values alone: [d_kv | d_kv]
    return e;
}

// Prompt attention of the large model's layer l on the tensor cores; groups of up to 128 queries.
template <int DH>
void launch_attn_prompt_tc_dh(tandem_ctx& c, const AttnTcArgs& a, const CUtensorMap& tmq, int l, int groups) {
    static std::atomic<unsigned long long> attr_done{0};
    ensure_dyn_smem(attn_prefill_tc_kernel<DH>, AtcCfg<DH>::SMEM_BYTES, attr_done);
    launch_ex(c, true, 1, attn_prefill_tc_kernel<DH>, dim3(a.n_heads, groups), dim3(ATC_THREADS), (size_t)AtcCfg<DH>::SMEM_BYTES, a, tmq,
              c.kmap[l], c.vmap[l]);
}
void launch_attn_prompt_tc(tandem_ctx& c, int l, const bf16* q, bf16* o, const Rows& r) {
    const int d = c.large.d.d_model, H = c.large.d.n_heads, dh = d / H;
    CUtensorMap tmq;
    if (!make_tmap_bf16(&tmq, q, (uint64_t)r.M, (uint64_t)d, (uint64_t)d)) {
        snprintf(g_cuda_err, sizeof(g_cuda_err), "cuTensorMapEncodeTiled failed for the query buffer");
        c.setup_failed = true;
        return;
    }
    AttnTcArgs a;
    memset(&a, 0, sizeof(a));
    a.out = o; a.ldo = d; a.row_seq = at<int>(c, c.lay.row_seq); a.row_pos = at<int>(c, c.lay.row_pos);
    a.grp_row0 = at<int>(c, c.lay.grp_row0); a.grp_cnt = at<int>(c, c.lay.grp_cnt);
    a.n_heads = H; a.n_kv_heads = c.large.kv_heads; a.t_max = c.cfg.max_seq; a.scale = 1.0f / sqrtf((float)dh); a.err_flag = c.st.counters + 2;
    // causal attention: Q K^T and P V over the lower triangle, 2 * d_head * T^2 flops per head and sequence
    ProfScope ps(c, PC_ATTN_PROMPT, 2.0 * dh * H * c.prompt_sq_sum);
    if (dh == 64) launch_attn_prompt_tc_dh<64>(c, a, tmq, l, r.groups);
    else launch_attn_prompt_tc_dh<128>(c, a, tmq, l, r.groups);
}

template <typename T>
void attention(tandem_ctx& c, const Model& m, int l, const T* q, T* o, const Rows& r) {
    const int d = m.d.d_model, H = m.d.n_heads, dh = d / H;
    AttnArgs aa; memset(&aa, 0, sizeof(aa));
    aa.q = q; aa.ldq = d; aa.kcache = kv_ptr<T>(c, m, l, 0); aa.vcache = kv_ptr<T>(c, m, l, 1);
    aa.out = o; aa.ldo = d; aa.row_seq = at<int>(c, c.lay.row_seq); aa.row_pos = at<int>(c, c.lay.row_pos);
    if (!r.decode) { aa.grp_row0 = at<int>(c, c.lay.grp_row0); aa.grp_cnt = at<int>(c, c.lay.grp_cnt); }
    aa.nq = r.nq; aa.n_heads = H; aa.n_kv_heads = m.kv_heads; aa.t_max = c.cfg.max_seq;
    aa.part_ml = at<float>(c, c.lay.part_ml); aa.part_acc = at<float>(c, c.lay.part_acc);
    aa.n_chunks_max = c.lay.n_chunks_max; aa.scale = 1.0f / sqrtf((float)dh);
    aa.merge_counters = at<int>(c, c.lay.attn_counters);
    if (!r.decode && sizeof(T) == 2 && c.tc_prompt_attn && &m == &c.large) {
        launch_attn_prompt_tc(c, l, reinterpret_cast<const bf16*>(q), reinterpret_cast<bf16*>(o), r);
        return;
    }
    launch_attn<T>(c, dh, aa, r.groups, !r.decode, r.n_chunks, r.kv_positions * 2.0 * d * sizeof(T));
}

// bf16 decode / block attention over the cache of layer l: bf16 queries, output rows as a value and a remainder plane.
void attention_decode(tandem_ctx& c, const Model& m, int l, const bf16* q, bf16* o, bf16* o_lo, const Rows& r) {
    const int d = m.d.d_model, H = m.d.n_heads, dh = d / H;
    AttnArgs aa; memset(&aa, 0, sizeof(aa));
    aa.q = q; aa.ldq = d; aa.kcache = kv_ptr<bf16>(c, m, l, 0); aa.vcache = kv_ptr<bf16>(c, m, l, 1);
    aa.out = o; aa.out_lo = o_lo; aa.ldo = d; aa.row_seq = at<int>(c, c.lay.row_seq); aa.row_pos = at<int>(c, c.lay.row_pos);
    aa.nq = r.nq; aa.n_heads = H; aa.n_kv_heads = m.kv_heads; aa.t_max = c.cfg.max_seq; aa.scale = 1.0f / sqrtf((float)dh);
    aa.err_flag = tc_scratch(c).err;
    aa.pass_grp = r.grp; aa.pass_pos = r.grp_pos;
    if (r.own_k) { aa.k2 = r.own_k; aa.v2 = r.own_v; aa.t_max2 = c.lay.fr_rows; }
    else if (r.whole_pass) aa.wait_first = 1;   // (a group's earlier positions may be rows of this very pass)
    launch_attn_decode(c, dh, aa, r.groups, r.kv_positions * 2.0 * d * 2.0, r.whole_pass);
}

// The fp32 passes whose maps run on the few-row kernel with LayerNorm fused into it: decode passes and short prompts.
bool fp32_few_rows(const tandem_ctx& c, const Rows& r) {
    return c.cfg.dtype == TANDEM_DTYPE_FP32 && (r.decode || r.M <= 64);
}
// LayerNorm, then y = a W^T (few rows, fp32): one kernel up to GS_KC elements per row, two beyond.
template <int EPI>
void ln_rows(tandem_ctx& c, const float* h, int M, const void* g, const void* b, const Lin& l, const EpiArgs& e, float* av = nullptr, int* ai = nullptr) {
    if (l.K <= GS_KC) { launch_rows<true, EPI>(c, h, l.K, M, l, e, g, b, av, ai); return; }
    float* a = at<float>(c, c.lay.a);
    launch_layernorm<float>(c, M, h, g, b, a, l.K);
    launch_rows<false, EPI>(c, a, l.K, M, l, e, nullptr, nullptr, av, ai);
}

// Eq. 2, first line, for small layer j, then that layer's LayerNorm and key/value maps: writes the
// small model's large-derived keys/values for the rows' positions.
template <typename T>
void project_layer(tandem_ctx& c, int j, const Rows& r) {
    const int dL = c.large.d.d_model, dS = c.small.d.d_model;
    const Lin t0 = lin1(wi_tandem(c, j, 0), c.cfg.ff_tandem_kind == TANDEM_FF_LINEAR ? dS : c.hidden, dL);
    const Lin kv = lin3(wi_layer(c.small, j, W_WK), wi_layer(c.small, j, W_WV), -1, c.small.d_kv, c.small.d_kv, dS);
    float* yhat = at<float>(c, c.lay.yhat);
    T* t1 = at<T>(c, c.lay.t1);
    const EpiArgs ekv = epi_cache<T>(c, c.small, j, nullptr);
    const void *lg = w_layer(c, c.small, j, W_LN1G), *lb = w_layer(c, c.small, j, W_LN1B);
    if constexpr (sizeof(T) == 4) {
        const float* x = at<float>(c, c.lay.h_large);   // fp32: the residual stream itself is the input
        if (fp32_few_rows(c, r)) {
            if (c.cfg.ff_tandem_kind == TANDEM_FF_LINEAR) {
                launch_rows<false, EPI_STORE_F32>(c, x, dL, r.M, t0, epi_plain(yhat, dS));
            } else {
                launch_rows<false, EPI_GELU>(c, x, dL, r.M, t0, epi_plain(t1, c.hidden));
                launch_rows<false, EPI_STORE_F32>(c, t1, c.hidden, r.M, lin1(wi_tandem(c, j, 1), dS, c.hidden), epi_plain(yhat, dS));
            }
            ln_rows<EPI_KV>(c, yhat, r.M, lg, lb, kv, ekv);
            return;
        }
    }
    const T* x = sizeof(T) == 4 ? reinterpret_cast<const T*>(at<float>(c, c.lay.h_large)) : at<T>(c, c.lay.xb);
    T* a_s = at<T>(c, c.lay.a_s);
    if (c.cfg.ff_tandem_kind == TANDEM_FF_LINEAR) {
        launch_gemm<T, EPI_STORE_F32>(c, x, dL, r.M, t0, epi_plain(yhat, dS));
    } else {
        launch_gemm<T, EPI_GELU>(c, x, dL, r.M, t0, epi_plain(t1, c.hidden));
        launch_gemm<T, EPI_STORE_F32>(c, t1, c.hidden, r.M, lin1(wi_tandem(c, j, 1), dS, c.hidden), epi_plain(yhat, dS));
    }
    launch_layernorm<T>(c, r.M, yhat, lg, lb, a_s, dS);
    launch_gemm<T, EPI_KV>(c, a_s, dS, r.M, kv, ekv);
}

bool projects_from(const tandem_ctx& c, int n_large_layers_done) {
    for (int j = 0; j < c.small.d.n_layers; ++j)
        if (c.layer_map[j] == n_large_layers_done) return true;
    return false;
}
template <typename T>
void project_after(tandem_ctx& c, int n_large_layers_done, const Rows& r) {
    for (int j = 0; j < c.small.d.n_layers; ++j)
        if (c.layer_map[j] == n_large_layers_done) project_layer<T>(c, j, r);
}

// bf16 prompt passes of few rows leave multiprocessors idle: their projections run on the side stream, beside the large model's next
// layers.  They share the buffers of one projection (and the copy of the residual stream that they read), so the main stream
// waits for the last ones before the next copy is made, and for all of them at the end of the pass.  (Small pair, 99 / 511 / 1499 rows: 602 -> 567, 759 -> 731, 1279 -> 1235 us;
// large pair, 899 rows: 1 %.)
template <typename P>
void prompt_project_forked(tandem_ctx& c, P project, bool join_all = true) {
    cudaStream_t main_stream = c.stream;
    cudaEvent_t fork = c.ev_fork[0];
    cudaEventRecord(fork, main_stream);
    cudaStreamWaitEvent(c.side, fork, 0);
    c.stream = c.side;
    c.next_launch_plain = true;   // first kernel after a cross-stream wait
    project();
    if (join_all) cudaEventRecord(c.ev_join, c.side);   // (else by `project`)
    c.stream = main_stream;
}
void prompt_project_join(tandem_ctx& c) {
    cudaStreamWaitEvent(c.stream, c.ev_join, 0);
    c.next_launch_plain = true;
}

// One decoder layer (Eq. 1; the same form serves the small model's layers in Eq. 2) on residual stream h.  project: the
// FF_Tandem projections that read h as it enters the layer (they run behind the first LayerNorm, which leaves them a bf16
// copy of h on its way).  snap (fp32 decode passes): copy of x^(l+1) when an FF_Tandem projection reads it.
template <typename T>
void decoder_layer(tandem_ctx& c, const Model& m, int l, float* h, const Rows& r, bool project = false, float* snap = nullptr, bool fork = false) {
    const int d = m.d.d_model, dff = m.d.d_ff;
    T* a = at<T>(c, c.lay.a);
    T* q = at<T>(c, c.lay.q);
    T* o = at<T>(c, c.lay.o);
    T* f = at<T>(c, c.lay.f);
    const Lin qkv = lin3(wi_layer(m, l, W_WQ), wi_layer(m, l, W_WK), wi_layer(m, l, W_WV), d, m.d_kv, d);
    const Lin wo = lin1(wi_layer(m, l, W_WO), d, d), w1 = lin1(wi_layer(m, l, W_W1), dff, d), w2 = lin1(wi_layer(m, l, W_W2), d, dff);
    const void *g1 = w_layer(c, m, l, W_LN1G), *b1 = w_layer(c, m, l, W_LN1B), *g2 = w_layer(c, m, l, W_LN2G), *b2 = w_layer(c, m, l, W_LN2B);
    if constexpr (sizeof(T) == 4) {
        if (fp32_few_rows(c, r)) {
            if (project) project_after<T>(c, l, r);
            ln_rows<EPI_QKV>(c, h, r.M, g1, b1, qkv, epi_cache<T>(c, m, l, q));
            attention<T>(c, m, l, q, o, r);
            launch_rows<false, EPI_RESID>(c, o, d, r.M, wo, epi_plain(h, d));
            ln_rows<EPI_GELU>(c, h, r.M, g2, b2, w1, epi_plain(f, dff));
            EpiArgs e2 = epi_plain(h, d);
            e2.snap = snap; e2.snap_ld = d;
            launch_rows<false, EPI_RESID>(c, f, dff, r.M, w2, e2);
            return;
        }
    }
    launch_layernorm<T>(c, r.M, h, g1, b1, a, d, project && sizeof(T) == 2 ? at<bf16>(c, c.lay.xb) : nullptr);
    if (project) { if (fork) prompt_project_forked(c, [&] { project_after<T>(c, l, r); }); else project_after<T>(c, l, r); }
    launch_gemm<T, EPI_QKV>(c, a, d, r.M, qkv, epi_cache<T>(c, m, l, q));
    attention<T>(c, m, l, q, o, r);
    launch_gemm<T, EPI_RESID>(c, o, d, r.M, wo, epi_plain(h, d));
    launch_layernorm<T>(c, r.M, h, g2, b2, a, d);
    launch_gemm<T, EPI_GELU>(c, a, d, r.M, w1, epi_plain(f, dff));
    launch_gemm<T, EPI_RESID>(c, f, dff, r.M, w2, epi_plain(h, d));
}

// Final LayerNorm, output head of a decode pass (fp32): logits, and (argmax) the blocks' maxima that the next pass's row set-up or the
// verify kernel turns into token ids.
void fp32_head(tandem_ctx& c, const Model& m, float* h, const Rows& r, float* logits, size_t amax_val_off, size_t amax_idx_off, bool argmax = true) {
    const Lin w = lin1(wi_tail(m, 2), m.d.vocab, m.d.d_model);
    if (argmax) ln_rows<EPI_ARGMAX>(c, h, r.M, w_tail(c, m, 0), w_tail(c, m, 1), w, epi_plain(logits, m.d.vocab), at<float>(c, amax_val_off), at<int>(c, amax_idx_off));
    else ln_rows<EPI_STORE_F32>(c, h, r.M, w_tail(c, m, 0), w_tail(c, m, 1), w, epi_plain(logits, m.d.vocab));
}

// The large model's layers over the current rows, whose embeddings are in the residual stream (block mode in decode,
// whole prompt otherwise).
template <typename T>
void large_layers(tandem_ctx& c, const Rows& r, bool project) {
    float* h = at<float>(c, c.lay.h_large);
    const int n = c.large.d.n_layers;
    const bool fork = sizeof(T) == 2 && project && r.M <= PROMPT_FORK_ROWS;
    bool forked = false;
    for (int l = 0; l < n; ++l) {
        const bool here = project && projects_from(c, l);
        if (here && forked) prompt_project_join(c);
        decoder_layer<T>(c, c.large, l, h, r, here, nullptr, fork);
        forked = forked || (here && fork);
    }
    if (forked) prompt_project_join(c);
    if (!project || !projects_from(c, n)) return;
    if constexpr (sizeof(T) == 2) {   // after the last layer no LayerNorm of the large model follows
        const size_t elems = (size_t)r.M * c.large.d.d_model;
        ProfScope ps(c, PC_ROWS, (double)elems * 6.0);
        launch_ex(c, true, 1, cast_rows_kernel<false>, dim3((unsigned)((elems / 8 + 255) / 256)), dim3(256), 0, (const float*)h, at<bf16>(c, c.lay.xb), elems, (size_t)0);
    }
    project_after<T>(c, n, r);
}

Rows decode_rows(tandem_ctx& c, int r_last, int nq) {
    Rows r;
    r.M = c.batch * nq; r.groups = c.batch; r.nq = nq; r.decode = true;
    r.n_chunks = c.chunks_launch;
    r.kv_positions = (double)c.n_sum + (double)c.batch * r_last;
    return r;
}

// Row set-up + embedding for block rows r0 .. r0+nq-1 of every sequence; fin_r: block row whose token is the
// arg-max the small model's last head GEMM left as per-tile results (-1: none).
template <typename T>
void begin_rows(tandem_ctx& c, const Model& m, float* h, int r0, int nq, int fin_r, float* snap = nullptr, const NextLn& ln = NextLn{}) {
    ProfScope ps(c, PC_ROWS, (double)c.batch * nq * m.d.d_model * 8.0);
    launch_ex(c, true, 1, step_begin_kernel<T>, dim3(c.batch * nq), dim3(128), 0, c.st, r0, nq, fin_r,
              (const float*)at<float>(c, c.lay.amax_val_small), (const int*)at<int>(c, c.lay.amax_idx_small), c.amax_tiles,
              c.amax_tiles, at<int>(c, c.lay.row_tok), at<int>(c, c.lay.row_seq), at<int>(c, c.lay.row_pos),
              (const T*)w_emb(c, m), (const T*)w_pos(c, m), h, m.d.d_model, snap, ln);
}

// fp32 draft step s: one token per sequence through the small model over the mixed context (Eq. 2, lines 2-3).  drafts_known: the
// previous draft is in the loop state (drawn, or given), not left as the blocks' maxima.
void fp32_small_step(tandem_ctx& c, int s, bool drafts_known, bool argmax = true) {
    float* y = at<float>(c, c.lay.h_small);
    begin_rows<float>(c, c.small, y, s, 1, (s > 0 && !drafts_known) ? s : -1);
    const Rows r = decode_rows(c, s, 1);
    for (int j = 0; j < c.small.d.n_layers; ++j) decoder_layer<float>(c, c.small, j, y, r);
    fp32_head(c, c.small, y, r, at<float>(c, c.lay.logits_small) + (size_t)s * c.batch * c.small.d.vocab, c.lay.amax_val_small, c.lay.amax_idx_small, argmax);
}

// FF_Tandem of the block's rows x (the residual stream after layer_map[j] large layers) for small layer j, as in the bf16 decode passes.
void fp32_project(tandem_ctx& c, int j, const float* x, const Rows& r, float* yhat, float* t1) {
    const int dL = c.large.d.d_model, dS = c.small.d.d_model;
    if (c.cfg.ff_tandem_kind == TANDEM_FF_LINEAR) {
        launch_rows<false, EPI_STORE_F32>(c, x, dL, r.M, lin1(wi_tandem(c, j, 0), dS, dL), epi_plain(yhat, dS));
    } else {
        launch_rows<false, EPI_GELU>(c, x, dL, r.M, lin1(wi_tandem(c, j, 0), c.hidden, dL), epi_plain(t1, c.hidden));
        launch_rows<false, EPI_STORE_F32>(c, t1, c.hidden, r.M, lin1(wi_tandem(c, j, 1), dS, c.hidden), epi_plain(yhat, dS));
    }
    const Lin kv = lin3(wi_layer(c.small, j, W_WK), wi_layer(c.small, j, W_WV), -1, c.small.d_kv, c.small.d_kv, dS);
    ln_rows<EPI_KV>(c, yhat, r.M, w_layer(c, c.small, j, W_LN1G), w_layer(c, c.small, j, W_LN1B), kv, epi_cache<float>(c, c.small, j, nullptr), nullptr, nullptr);
}

// The projections of a decode pass after n large layers.  They run on the side stream,
// from the copy of x^(l(j)) that the producing kernel left: they depend on nothing the large model does
// afterwards (and nothing in the iteration depends on them before the next draft), so they run beside the large model's
// later layers instead of in their chain.  (fp32, small layers wider than GS_KC: LayerNorm kernel and maps share the large pass's
// buffer, so those stay in its chain.)
template <typename P>
void project_forked(tandem_ctx& c, int n_large_layers_done, int slot, P project) {
    const size_t RD = (size_t)c.lay.dec_rows, dS = c.small.d.d_model;
    const float* snap = at<float>(c, c.lay.proj_snap) + (size_t)slot * RD * c.large.d.d_model;
    cudaStream_t main_stream = c.stream;
    cudaEventRecord(c.ev_fork[slot], main_stream);
    cudaStreamWaitEvent(c.side, c.ev_fork[slot], 0);
    c.stream = c.side;
    c.next_launch_plain = true;   // first kernel after a cross-stream wait
    for (int j = 0; j < c.small.d.n_layers; ++j)
        if (c.layer_map[j] == n_large_layers_done)
            project(j, snap, at<float>(c, c.lay.proj_yhat) + (size_t)j * RD * dS, at<float>(c, c.lay.proj_a) + (size_t)j * RD * dS,
                    at<float>(c, c.lay.proj_t1) + (size_t)j * RD * c.hidden);
    c.stream = main_stream;
}
// They join the main stream before the verify kernel.
void project_join(tandem_ctx& c) {
    cudaEventRecord(c.ev_join, c.side);
    cudaStreamWaitEvent(c.stream, c.ev_join, 0);
    c.next_launch_plain = true;
}

// Slot of the projection buffers for the residual stream after `n` large layers: the first small layer fed from there, or -1.
int project_slot(const tandem_ctx& c, int n) {
    for (int j = 0; j < c.small.d.n_layers; ++j)
        if (c.layer_map[j] == n) return j;
    return -1;
}

// fp32 block pass of the large model over nq rows per sequence; fin_r: see begin_rows; head: final LayerNorm + output head.
void fp32_large_block(tandem_ctx& c, int nq, int fin_r, bool project, bool head) {
    float* h = at<float>(c, c.lay.h_large);
    const size_t snap_elems = (size_t)c.lay.dec_rows * c.large.d.d_model;
    const bool fork = project && c.small.d.d_model <= GS_KC;
    auto snap_of = [&](int n) -> float* {
        const int slot = fork ? project_slot(c, n) : -1;
        return slot >= 0 ? at<float>(c, c.lay.proj_snap) + (size_t)slot * snap_elems : nullptr;
    };
    begin_rows<float>(c, c.large, h, 0, nq, fin_r, snap_of(0));
    const Rows r = decode_rows(c, nq - 1, nq);
    auto run = [&](int j, const float* snap, float* yhat, float*, float* t1) { fp32_project(c, j, snap, r, yhat, t1); };
    if (!fork) {
        large_layers<float>(c, r, project);
    } else {
        for (int l = 0; l <= c.large.d.n_layers; ++l) {
            if (project_slot(c, l) >= 0) project_forked(c, l, project_slot(c, l), run);
            if (l < c.large.d.n_layers) decoder_layer<float>(c, c.large, l, h, r, false, snap_of(l + 1));
        }
    }
    if (head) fp32_head(c, c.large, h, r, at<float>(c, c.lay.logits_large), c.lay.amax_val_large, c.lay.amax_idx_large);
    if (fork) project_join(c);   // (every small layer is fed from somewhere)
}

// Teacher-forced round (accept mode 5, fp32): the given tokens become the round's drafts; after the draft steps their
// logits are scored against the given next tokens.
void launch_forced_fill(tandem_ctx& c, int gamma) {
    ProfScope ps(c, PC_ROWS, (double)c.batch * gamma * 8.0);
    launch_ex(c, true, 1, forced_fill_kernel, dim3(1), dim3(256), 0, c.st, c.batch, gamma, (const int*)at<int>(c, c.lay.forced_ids),
              (const int*)at<int>(c, c.lay.forced_len), (int)c.cfg.max_seq);
}
void launch_score_rows(tandem_ctx& c, int gamma) {
    ProfScope ps(c, PC_ARGMAX, (double)c.batch * gamma * c.small.d.vocab * 8.0);
    launch_ex(c, true, SCR_CLUSTER, score_rows_kernel, dim3(SCR_CLUSTER, gamma, c.batch), dim3(SCR_THREADS), 0, c.st, c.batch, (const float*)at<float>(c, c.lay.logits_small),
              (int)c.small.d.vocab, (const int*)at<int>(c, c.lay.forced_ids), (const int*)at<int>(c, c.lay.forced_len), (int)c.cfg.max_seq,
              at<float>(c, c.lay.forced_nll), at<int>(c, c.lay.forced_top));
}

void launch_verify(tandem_ctx& c, int gamma, int mode, uint64_t seed, int max_new, bool from_tiles, bool adaptive = false) {
    ProfScope ps(c, PC_VERIFY, (double)c.batch * (2 * gamma + 8) * 4.0);
    launch_ex(c, true, 1, verify_kernel, dim3(1), dim3(VERIFY_THREADS), 0, c.st, c.batch, gamma, mode, (unsigned long long)seed, max_new,
              from_tiles ? (const float*)at<float>(c, c.lay.amax_val_large) : (const float*)nullptr,
              from_tiles ? (const int*)at<int>(c, c.lay.amax_idx_large) : (const int*)nullptr, c.amax_tiles, c.amax_tiles,
              from_tiles ? (const float*)at<float>(c, c.lay.amax_val_small) : (const float*)nullptr,
              from_tiles ? (const int*)at<int>(c, c.lay.amax_idx_small) : (const int*)nullptr,
              adaptive ? (const int*)c.st.block_len : (const int*)nullptr);
}

// Adaptive block length: the router's decision after draft step s, for every sequence that is still drafting.
void launch_router(tandem_ctx& c, int s, int gamma_max) {
    const float* logits = at<float>(c, c.lay.logits_small) + (size_t)s * c.batch * c.small.d.vocab;
    ProfScope ps(c, PC_ARGMAX, (double)c.batch * c.small.d.vocab * 8.0);
    const size_t feat_bytes = sizeof(float) * (size_t)(1 + c.router.k + c.router.k * c.small.d.d_model);   // <= 48 KB, checked by tandem_set_router
    static std::atomic<unsigned long long> attr_bf16{0}, attr_fp32{0};
    if (c.cfg.dtype == TANDEM_DTYPE_BF16) ensure_dyn_smem(router_kernel<bf16>, 48 * 1024, attr_bf16);
    else ensure_dyn_smem(router_kernel<float>, 48 * 1024, attr_fp32);   // (48 KB and the static part are more than the default limit)
    if (c.cfg.dtype == TANDEM_DTYPE_BF16)
        launch_ex(c, true, RT_CLUSTER, router_kernel<bf16>, dim3(RT_CLUSTER, c.batch), dim3(RT_THREADS), feat_bytes, c.st, c.batch, logits, (int)c.small.d.vocab, s, gamma_max,
                  (const bf16*)w_emb(c, c.small), (int)c.small.d.d_model, c.router);
    else
        launch_ex(c, true, RT_CLUSTER, router_kernel<float>, dim3(RT_CLUSTER, c.batch), dim3(RT_THREADS), feat_bytes, c.st, c.batch, logits, (int)c.small.d.vocab, s, gamma_max,
                  (const float*)w_emb(c, c.small), (int)c.small.d.d_model, c.router);
}
void launch_adaptive_begin(tandem_ctx& c) {
    ProfScope ps(c, PC_ROWS, (double)c.batch * 8.0);
    launch_ex(c, true, 1, adaptive_begin_kernel, dim3(1), dim3(256), 0, c.st, c.batch);
}

// Sampled SPEED: draft s of every sequence drawn from the small model's logits of step s.
void launch_sample_draft(tandem_ctx& c, int s, uint64_t seed) {
    const float* logits = at<float>(c, c.lay.logits_small) + (size_t)s * c.batch * c.small.d.vocab;
    ProfScope ps(c, PC_ARGMAX, (double)c.batch * c.small.d.vocab * 4.0);
    launch_ex(c, true, SMC_CLUSTER, sample_draft_kernel, dim3(SMC_CLUSTER, c.batch), dim3(SMC_THREADS), 0, c.st, logits, (int)c.small.d.vocab, s,
              c.temp_small, (unsigned long long)seed, at<float2>(c, c.lay.smp_small) + (size_t)s * c.batch);
}
// Sampled SPEED: accept / redraw decisions of the iteration, ahead of the verify kernel's bookkeeping.
void launch_sample_verify(tandem_ctx& c, int gamma, uint64_t seed) {
    const int rows = c.batch * (gamma + 1), V = c.large.d.vocab;
    const float* logits = at<float>(c, c.lay.logits_large);
    ProfScope ps(c, PC_ARGMAX, (double)(rows + 2 * c.batch) * V * 4.0);
    launch_ex(c, true, SMC_CLUSTER, sample_stats_kernel, dim3(SMC_CLUSTER, rows), dim3(SMC_THREADS), 0, logits, V, c.temp_large, at<float2>(c, c.lay.smp_large));
    launch_ex(c, true, SMC_CLUSTER, sample_verify_kernel, dim3(SMC_CLUSTER, c.batch), dim3(SMC_THREADS), 0, c.st, c.batch, gamma, logits,
              (const float*)at<float>(c, c.lay.logits_small), V, c.temp_large, c.temp_small, (unsigned long long)seed,
              (const float2*)at<float2>(c, c.lay.smp_large), (const float2*)at<float2>(c, c.lay.smp_small));
}

void fp32_iteration(tandem_ctx& c, int gamma, int mode, uint64_t seed, int max_new) {
    const bool known = mode == 4 || mode == 5;        // drafts drawn, or given
    if (mode == 5) launch_forced_fill(c, gamma);
    for (int s = 0; s < gamma; ++s) {
        fp32_small_step(c, s, known, !known);
        if (mode == 4) launch_sample_draft(c, s, seed);
    }
    if (mode == 5) launch_score_rows(c, gamma);
    if (mode == 3 || mode == 5) fp32_large_block(c, gamma, -1, true, false);   // stand-alone Tandem without the free token: gamma rows, no output head
    else fp32_large_block(c, gamma + 1, (gamma > 0 && !known) ? gamma : -1, true, true);
    if (mode == 4) launch_sample_verify(c, gamma, seed);
    launch_verify(c, gamma, mode == 5 ? 3 : mode, seed, max_new, mode != 5);
    c.last_gamma = gamma;
}

void fp32_greedy_iteration(tandem_ctx& c, int max_new) {
    fp32_large_block(c, 1, -1, false, true);
    launch_verify(c, 0, 0, 0ull, max_new, true);
    c.last_gamma = 0;
}

// ---------------------------------------------------------------------------------------------------
// bf16 decode on the tensor cores: five kernels per decoder layer, chained by programmatic dependent launch
// ---------------------------------------------------------------------------------------------------

// The decode activations' value / remainder planes (see tandem_ctx::xmap): buffer 0 = residual stream, less c, times the next
// LayerNorm's gain, 1 = attention output, 2 = GELU output; K = the row length in use (the model's width, or its FFN width
// for buffer 2).
struct XPlanes { bf16* hi; bf16* lo; TcRows rows; };
XPlanes x_planes(tandem_ctx& c, int buf, const Model& m) {
    const size_t off = buf == 0 ? c.lay.a32 : (buf == 1 ? c.lay.o32 : c.lay.f32);
    const size_t K = buf == 2 ? m.d.d_ff : m.d.d_model;
    XPlanes p;
    p.hi = at<bf16>(c, off);
    p.lo = p.hi + (size_t)c.lay.dec_rows * K;
    p.rows.map = &c.xmap[buf][&m == &c.large ? 0 : 1];
    return p;
}

// LayerNorm number `idx` of a model (2 l, 2 l + 1 of layer l, 2 n_layers the final one): its gain, what the producer of the
// residual stream leaves for it, and the operand of the GEMM behind it.
const void* ln_gain(const tandem_ctx& c, const Model& m, int idx) {
    return idx == 2 * m.d.n_layers ? w_tail(c, m, 0) : w_layer(c, m, idx / 2, idx % 2 ? W_LN2G : W_LN1G);
}
// The value taken off each row before LayerNorm `idx` (NextLn::ref).  Two arrays in turn: the GEMM behind a LayerNorm reads its
// own from one and leaves the rows' means, the next LayerNorm's, in the other.
float* ln_ref_of(tandem_ctx& c, int idx) { return at<float>(c, c.lay.ln_ref) + (size_t)(idx & 1) * c.lay.dec_rows; }
NextLn next_ln(tandem_ctx& c, const Model& m, int idx) {
    const XPlanes p = x_planes(c, 0, m);
    return {static_cast<const float*>(ln_gain(c, m, idx)), p.hi, p.lo, at<float2>(c, c.lay.ln_stats), cdiv(m.d.d_model, 32), ln_ref_of(c, idx)};
}
TcRows ln_rows_of(tandem_ctx& c, const Model& m, int idx) {
    TcRows r = x_planes(c, 0, m).rows;
    r.ln_map = &c.lnmap[&m == &c.large ? 0 : 1];
    r.ln_row = 4 * idx;
    r.ln_stats = at<float2>(c, c.lay.ln_stats);
    r.ln_groups = cdiv(m.d.d_model, 32);
    r.ln_ref = ln_ref_of(c, idx);
    r.ln_mean = ln_ref_of(c, idx + 1);
    return r;
}

// Whether the projection's LayerNorm is fused into its GEMM's operand load.  Fused, every CTA of the GEMM normalises the rows
// it needs itself: right for a couple of sequences and short rows, wasteful beyond.  The choice depends on the batch and the
// model only, never on the number of rows.
bool tc_fused_prologue(const tandem_ctx& c, int K) { return c.batch <= 2 && K <= 1024; }

// One decoder layer of a decode pass.  Between the kernels the activations are fp32 (the residual stream) or pairs of bf16
// planes; only the queries and the cached keys / values are bf16.
void tc_decoder_layer(tandem_ctx& c, const Model& m, int l, float* h, const Rows& r, bool stream_w, float* snap = nullptr) {
    const int d = m.d.d_model, dff = m.d.d_ff;
    bf16* q = at<bf16>(c, c.lay.q);
    TcScratch sc = tc_scratch(c);
    sc.rows_early = l > 0;   // (the first layer's maps follow the kernel that writes them)
    const XPlanes xo = x_planes(c, 1, m), xf = x_planes(c, 2, m);
    launch_tc_decode<PRO_LNT, EPI_QKV>(c, sc, nullptr, d, nullptr, nullptr, r.M,
                                       tcw3(c, wi_layer(m, l, W_WQ), wi_layer(m, l, W_WK), wi_layer(m, l, W_WV), d, m.d_kv, d), stream_w,
                                       epi_cache<bf16>(c, m, l, q), nullptr, nullptr, 0, ln_rows_of(c, m, 2 * l));
    attention_decode(c, m, l, q, xo.hi, xo.lo, r);
    EpiArgs eo = epi_plain(h, d);
    eo.ln = next_ln(c, m, 2 * l + 1);
    launch_tc_decode<PRO_TMA, EPI_RESID>(c, sc, nullptr, d, nullptr, nullptr, r.M, tcw(c, wi_layer(m, l, W_WO), -1, -1, d, d), stream_w, eo,
                                         nullptr, nullptr, 0, xo.rows);
    EpiArgs e1 = epi_plain(xf.hi, dff);
    e1.out_lo = xf.lo;
    launch_tc_decode<PRO_LNT, EPI_GELU>(c, sc, nullptr, d, nullptr, nullptr, r.M, tcw(c, wi_layer(m, l, W_W1), -1, -1, dff, d), stream_w, e1,
                                        nullptr, nullptr, 0, ln_rows_of(c, m, 2 * l + 1));
    EpiArgs e2 = epi_plain(h, d);
    e2.snap = snap; e2.snap_ld = d;   // copy of x^(l+1) when an FF_Tandem projection reads it
    e2.ln = next_ln(c, m, 2 * l + 2);
    launch_tc_decode<PRO_TMA, EPI_RESID>(c, sc, nullptr, dff, nullptr, nullptr, r.M, tcw(c, wi_layer(m, l, W_W2), -1, -1, d, dff), stream_w, e2,
                                         nullptr, nullptr, 0, xf.rows);
}

// Final LayerNorm + output head; leaves fp32 logits and the per-tile (max, index) pairs that the next kernel
// (the next pass's row set-up, or the verify kernel) turns into token ids.
void tc_head(tandem_ctx& c, const Model& m, const Rows& r, float* logits, size_t amax_val_off, size_t amax_idx_off, bool stream_w) {
    launch_tc_decode<PRO_LNT, EPI_ARGMAX>(c, tc_scratch(c), nullptr, m.d.d_model, nullptr, nullptr, r.M, tcw(c, wi_tail(m, 2), -1, -1, m.d.vocab, m.d.d_model),
                                          stream_w, epi_plain(logits, m.d.vocab), at<float>(c, amax_val_off), at<int>(c, amax_idx_off), c.amax_tiles,
                                          ln_rows_of(c, m, 2 * m.d.n_layers));
}

// sampled: the previous draft was drawn by sample_draft_kernel (it is in the loop state already), not left as per-tile
// arg-max results.
enum StepPart { STEP_WHOLE, STEP_HEAD, STEP_TAIL };   // all of a draft step; its row set-up and first layer; the rest
void tc_small_step(tandem_ctx& c, int s, bool sampled, StepPart part = STEP_WHOLE) {
    float* y = at<float>(c, c.lay.h_small);
    if (part != STEP_TAIL) begin_rows<bf16>(c, c.small, y, s, 1, (s > 0 && !sampled) ? s : -1, nullptr, next_ln(c, c.small, 0));
    const Rows r = decode_rows(c, s, 1);
    for (int j = part == STEP_TAIL ? 1 : 0; j < (part == STEP_HEAD ? 1 : c.small.d.n_layers); ++j) tc_decoder_layer(c, c.small, j, y, r, false);
    if (part == STEP_HEAD) return;
    float* logits = at<float>(c, c.lay.logits_small) + (size_t)s * c.batch * c.small.d.vocab;
    tc_head(c, c.small, r, logits, c.lay.amax_val_small, c.lay.amax_idx_small, false);
}

// FF_Tandem of decode rows x (fp32, [r.M][d_large], the residual stream after layer_map[j] large layers; Eq. 2, first line) for small layer
// j, then that layer's LayerNorm and key/value maps with the cache write as the GEMM epilogue.  yhat, a_j, t1: fp32 rows.
void tc_project(tandem_ctx& c, int j, const float* x, const Rows& r, float* yhat, float* a_j, float* t1) {
    const int dL = c.large.d.d_model, dS = c.small.d.d_model;
    const TcScratch sc = tc_scratch(c);
    if (c.cfg.ff_tandem_kind == TANDEM_FF_LINEAR) {
        launch_tc_decode<PRO_F32, EPI_STORE_F32>(c, sc, x, dL, nullptr, nullptr, r.M, tcw(c, wi_tandem(c, j, 0), -1, -1, dS, dL), true,
                                                 epi_plain(yhat, dS));
    } else {
        launch_tc_decode<PRO_F32, EPI_GELU>(c, sc, x, dL, nullptr, nullptr, r.M, tcw(c, wi_tandem(c, j, 0), -1, -1, c.hidden, dL), true,
                                            epi_plain(t1, c.hidden));
        launch_tc_decode<PRO_F32, EPI_STORE_F32>(c, sc, t1, c.hidden, nullptr, nullptr, r.M, tcw(c, wi_tandem(c, j, 1), -1, -1, dS, c.hidden),
                                                 true, epi_plain(yhat, dS));
    }
    const void *lg = w_layer(c, c.small, j, W_LN1G), *lb = w_layer(c, c.small, j, W_LN1B);
    const TcW wkv = tcw(c, wi_layer(c.small, j, W_WK), wi_layer(c.small, j, W_WV), -1, c.small.d_kv, dS);
    const EpiArgs ekv = epi_cache<bf16>(c, c.small, j, nullptr);
    if (tc_fused_prologue(c, dS)) {
        launch_tc_decode<PRO_LN, EPI_KV>(c, sc, yhat, dS, lg, lb, r.M, wkv, true, ekv);
    } else {
        launch_layernorm<float>(c, r.M, yhat, lg, lb, a_j, dS);
        launch_tc_decode<PRO_F32, EPI_KV>(c, sc, a_j, dS, nullptr, nullptr, r.M, wkv, true, ekv);
    }
}

// The large model over nq block rows per sequence (row 0 = pending token, row r = draft r); fin_r: block row whose
// token the small model's last head GEMM left as per-tile results (-1: none); head: final LayerNorm + output head.
void tc_large_block(tandem_ctx& c, int nq, int fin_r, bool project, bool head) {
    float* h = at<float>(c, c.lay.h_large);
    const size_t snap_elems = (size_t)c.lay.dec_rows * c.large.d.d_model;
    auto snap_of = [&](int n) -> float* {
        const int slot = project ? project_slot(c, n) : -1;
        return slot >= 0 ? at<float>(c, c.lay.proj_snap) + (size_t)slot * snap_elems : nullptr;
    };
    bool any_fork = false;
    begin_rows<bf16>(c, c.large, h, 0, nq, fin_r, snap_of(0), next_ln(c, c.large, 0));
    const Rows r = decode_rows(c, nq - 1, nq);
    auto run = [&](int j, const float* snap, float* yhat, float* a_j, float* t1) { tc_project(c, j, snap, r, yhat, a_j, t1); };
    if (project && project_slot(c, 0) >= 0) { project_forked(c, 0, project_slot(c, 0), run); any_fork = true; }
    for (int l = 0; l < c.large.d.n_layers; ++l) {
        tc_decoder_layer(c, c.large, l, h, r, true, snap_of(l + 1));
        if (project && project_slot(c, l + 1) >= 0) { project_forked(c, l + 1, project_slot(c, l + 1), run); any_fork = true; }
    }
    if (head) tc_head(c, c.large, r, at<float>(c, c.lay.logits_large), c.lay.amax_val_large, c.lay.amax_idx_large, true);
    if (any_fork) project_join(c);
}

// ---- teacher-forced pass (bf16): the prompt pass's kernels with activations as two planes ----------------------------

// What a pass's maps read: two planes of `plane` rows of K elements.
template <int EPI>
void pass_gemm(tandem_ctx& c, const bf16* x, int M, int plane, const TcW& w, EpiArgs e, const TcScore& sc = TcScore()) {
    if (EPI == EPI_GELU) e.out_lo = static_cast<bf16*>(e.out) + (size_t)plane * e.ldo;
    if (launch_tc_tiled<EPI, true>(c, x, w.K, M, w, e, c.st.counters + 2, plane, sc) != TANDEM_OK) c.setup_failed = true;
}
void pass_layernorm(tandem_ctx& c, int M, int plane, const float* x, const void* gain, const void* bias, bf16* out, int d, bf16* raw = nullptr) {
    launch_layernorm<bf16, true>(c, M, x, gain, bias, out, d, raw, (size_t)plane * d);
}

// FF_Tandem of a pass's rows (planes x, the large model's residual stream) for small layer j, into the small model's cache.
// read (nullable): recorded when x has been read.
void pass_project(tandem_ctx& c, int j, const bf16* x, const Rows& r, cudaEvent_t read = nullptr) {
    const int dL = c.large.d.d_model, dS = c.small.d.d_model;
    float* yhat = at<float>(c, r.apart ? c.lay.fa_yhat : c.lay.fr_yhat);
    bf16 *a_j = at<bf16>(c, r.apart ? c.lay.fa_a : c.lay.fr_a), *t1 = at<bf16>(c, r.apart ? c.lay.fa_t1 : c.lay.fr_t1);
    if (c.cfg.ff_tandem_kind == TANDEM_FF_LINEAR) {
        pass_gemm<EPI_STORE_F32>(c, x, r.M, r.plane, tcw(c, wi_tandem(c, j, 0), -1, -1, dS, dL), epi_plain(yhat, dS));
        if (read) cudaEventRecord(read, c.stream);
    } else {
        pass_gemm<EPI_GELU>(c, x, r.M, r.plane, tcw(c, wi_tandem(c, j, 0), -1, -1, c.hidden, dL), epi_plain(t1, c.hidden));
        if (read) cudaEventRecord(read, c.stream);
        pass_gemm<EPI_STORE_F32>(c, t1, r.M, r.plane, tcw(c, wi_tandem(c, j, 1), -1, -1, dS, c.hidden), epi_plain(yhat, dS));
    }
    pass_layernorm(c, r.M, r.plane, yhat, w_layer(c, c.small, j, W_LN1G), w_layer(c, c.small, j, W_LN1B), a_j, dS);
    pass_gemm<EPI_KV>(c, a_j, r.M, r.plane, tcw(c, wi_layer(c.small, j, W_WK), wi_layer(c.small, j, W_WV), -1, c.small.d_kv, dS), epi_cache<bf16>(c, c.small, j, nullptr));
}

// One model's layers over a pass's rows in the residual stream h (and the large model's projections between them).
void pass_layers(tandem_ctx& c, const Model& m, float* h, const Rows& r) {
    const int d = m.d.d_model, dff = m.d.d_ff, n = m.d.n_layers;
    const bool large = &m == &c.large, fork = large && r.M <= PROMPT_FORK_ROWS;
    bf16 *x = at<bf16>(c, large ? c.lay.fr_x : c.lay.fr_xs), *f = at<bf16>(c, large ? c.lay.fr_f : c.lay.fr_fs), *q = at<bf16>(c, large ? c.lay.fr_q : c.lay.fr_fs);
    bf16 *o = x, *raw = at<bf16>(c, c.lay.fr_raw);
    // Forked, the large model goes on to its FFN when the layer's projections are done, whose buffers lie under the GELU outputs; or when their
    // input has been read, where the others lie apart.  769 rows of the small pair, projections in the large model's stream 1580 us,
    // forked until the FFN 1548, apart 1533; 256 rows 1180 and 1135 (the first two).
    auto project = [&](int l, bool forked) {
        int last = 0;
        for (int j = 0; j < c.small.d.n_layers; ++j) if (c.layer_map[j] == l) last = j;
        for (int j = 0; j <= last; ++j)
            if (c.layer_map[j] == l) pass_project(c, j, raw, r, forked && r.apart && j == last ? c.ev_join : nullptr);
    };
    bool forked = false;
    for (int l = 0; l < n; ++l) {
        const bool from_here = large && projects_from(c, l);
        pass_layernorm(c, r.M, r.plane, h, w_layer(c, m, l, W_LN1G), w_layer(c, m, l, W_LN1B), x, d, from_here ? raw : nullptr);
        if (from_here) { if (fork) prompt_project_forked(c, [&] { project(l, true); }, !r.apart); else project(l, false); }
        forked = forked || (from_here && fork);
        EpiArgs eq = epi_cache<bf16>(c, m, l, q);
        if (r.own_k) { eq.kcache = r.own_k; eq.vcache = r.own_v; eq.row_seq = eq.row_pos = nullptr; eq.t_max = c.lay.fr_rows; }
        pass_gemm<EPI_QKV>(c, x, r.M, r.plane, tcw3(c, wi_layer(m, l, W_WQ), wi_layer(m, l, W_WK), wi_layer(m, l, W_WV), d, m.d_kv, d), eq);
        attention_decode(c, m, l, q, o, o + (size_t)r.plane * d, r);
        pass_gemm<EPI_RESID>(c, o, r.M, r.plane, tcw(c, wi_layer(m, l, W_WO), -1, -1, d, d), epi_plain(h, d));
        if (from_here && fork) prompt_project_join(c);
        pass_layernorm(c, r.M, r.plane, h, w_layer(c, m, l, W_LN2G), w_layer(c, m, l, W_LN2B), x, d);
        pass_gemm<EPI_GELU>(c, x, r.M, r.plane, tcw(c, wi_layer(m, l, W_W1), -1, -1, dff, d), epi_plain(f, dff));
        pass_gemm<EPI_RESID>(c, f, r.M, r.plane, tcw(c, wi_layer(m, l, W_W2), -1, -1, d, dff), epi_plain(h, d));
    }
    if (forked && r.apart) project_join(c);
    if (!large || !projects_from(c, n)) return;
    const size_t elems = (size_t)r.M * d;   // after the last layer no LayerNorm of the large model follows
    {
        ProfScope ps(c, PC_ROWS, (double)elems * 8.0);
        launch_ex(c, true, 1, cast_rows_kernel<true>, dim3((unsigned)((elems / 8 + 255) / 256)), dim3(256), 0, (const float*)h, raw, elems, (size_t)r.plane * d);
    }
    project(n, false);
}

// The rows f of a teacher-forced forward (whole blocks) through both models.  The large model reads them as one causal pass
// and its projections go to the small model's cache; then the small model reads all blocks at once, since the tokens it would draft
// are given: a row attends the large-derived keys / values of the positions before its block, and its block's own ones, which lie
// row by row in a place of their own for the time of one layer.  Activations keep the decode passes' 16 bits (value + remainder planes), the attention
// is theirs.  Four sequences of 129-257 tokens through the small pair: one round per block, gamma small passes and one large each,
// 36.1 ms; the decode GEMM over groups of 64 rows 1.95 ms (a group fetches every weight tile again); 1.53 ms like this.
void forced_pass(tandem_ctx& c, ForcedRows f, bool only, int groups_large, int groups_small, double kv_positions) {
    const Model &L = c.large, &S = c.small;
    Rows r;
    r.M = f.rows; r.decode = true; r.whole_pass = true; r.plane = c.lay.fr_rows; r.n_chunks = 1; r.kv_positions = kv_positions;
    r.grp = f.grp; r.grp_pos = f.grp_pos;
    r.apart = only && c.lay.fr_apart != 0;   // (of several passes, an earlier one has left logits there)
    auto begin = [&](const Model& m, float* h, int last_rows) {
        ProfScope ps(c, PC_ROWS, (double)f.rows * m.d.d_model * 8.0);
        launch_ex(c, true, 1, forced_rows_kernel, dim3(f.rows + 1 + last_rows), dim3(128), 0, c.st, f, (const bf16*)w_emb(c, m), (const bf16*)w_pos(c, m), h,
                  (int)m.d.d_model, (int)c.ticket, (int)c.router_ticket);
    };
    float *h = at<float>(c, c.lay.h_large), *hs = at<float>(c, c.lay.fr_hs);
    f.group = PASS_GROUP;
    r.nq = PASS_GROUP; r.groups = groups_large;
    begin(L, h, 0);
    pass_layers(c, L, h, r);
    f.group = f.gamma;
    r.nq = f.gamma; r.groups = groups_small;
    r.own_k = at<bf16>(c, c.lay.fr_kv); r.own_v = r.own_k + (size_t)c.lay.fr_rows * S.d_kv;
    begin(S, hs, f.batch * f.gamma);
    pass_layers(c, S, hs, r);
    const int d = S.d.d_model, tiles = c.lay.score_tiles;
    bf16* x = at<bf16>(c, c.lay.fr_xs);
    pass_layernorm(c, f.rows, r.plane, hs, w_tail(c, S, 0), w_tail(c, S, 1), x, d);
    for (int r0 = 0; r0 < f.rows; r0 += c.lay.fr_head_rows) {
        const int rows = std::min(c.lay.fr_head_rows, f.rows - r0);
        float* val = at<float>(c, c.lay.fr_tiles);
        TcScore t;
        t.val = val; t.idx = reinterpret_cast<int*>(val + (size_t)rows * tiles); t.sum = val + (size_t)2 * rows * tiles; t.stride = tiles;
        t.truth = f.truth + r0; t.truth_val = f.nll + f.v0 + r0;
        t.keep = f.keep + r0; t.kept = f.last_logits;
        pass_gemm<EPI_SCORE>(c, x + (size_t)r0 * d, rows, r.plane, tcw(c, wi_tail(S, 2), -1, -1, S.d.vocab, d), epi_plain(nullptr, S.d.vocab), t);
        ProfScope ps(c, PC_ARGMAX, 12.0 * rows * tiles);
        launch_ex(c, true, 1, score_tiles_kernel, dim3(cdiv(rows, 8)), dim3(256), 0, rows, tiles, (const float*)t.val, (const int*)t.idx, (const float*)t.sum,
                  f.nll + f.v0 + r0, f.top + f.v0 + r0);
    }
}

void tc_iteration(tandem_ctx& c, int gamma, int mode, uint64_t seed, int max_new) {
    const bool sampled = mode == 4;
    for (int s = 0; s < gamma; ++s) {
        tc_small_step(c, s, sampled);   // (the sampled drafts are found in the loop state, not in per-tile arg-max results)
        if (sampled) launch_sample_draft(c, s, seed);
    }
    if (mode == 3) tc_large_block(c, gamma, -1, true, false);   // gamma rows, no head: the last draft is finished by the verify kernel
    else tc_large_block(c, gamma + 1, (gamma > 0 && !sampled) ? gamma : -1, true, true);
    if (sampled) launch_sample_verify(c, gamma, seed);
    launch_verify(c, gamma, mode, seed, max_new, true);
    c.last_gamma = gamma;
}

void tc_greedy_iteration(tandem_ctx& c, int max_new) {
    tc_large_block(c, 1, -1, false, true);
    launch_verify(c, 0, 0, 0ull, max_new, true);
    c.last_gamma = 0;
}

tandem_status check_launch() {
    CK(cudaGetLastError());
    return TANDEM_OK;
}
// The same for a context: also reports a launch helper that had to skip its launch.
tandem_status check_launch(tandem_ctx& c) {
    if (c.setup_failed) { c.setup_failed = false; return TANDEM_ERR_CUDA; }
    return check_launch();
}

// kind 0: draft + verify (gamma drafts, accept mode);  1: plain greedy M_L;
// kind 3: one draft step of the adaptive block length (gamma = step index, mode = gamma_max) followed by the router;
// kind 4: the verify half of an adaptive iteration (gamma = longest block of the batch).
// bf16: kind 3 is the step's row set-up and first layer, kind 5 (same arguments) the rest of it and the router.
void enqueue_iteration(tandem_ctx& c, int kind, int gamma, int mode, uint64_t seed, int max_new) {
    const bool bf = c.cfg.dtype == TANDEM_DTYPE_BF16;   // one bf16 path: the tensor-core kernels (a bf16 context always has tensor maps)
    if (kind == 3 || kind == 5) {
        if (kind == 3 && gamma == 0) launch_adaptive_begin(c);
        if (!bf) fp32_small_step(c, gamma, false);
        else tc_small_step(c, gamma, false, kind == 3 ? STEP_HEAD : STEP_TAIL);
        if (!bf || kind == 5) launch_router(c, gamma, mode);
        return;
    }
    if (kind == 4) {
        if (bf) {
            tc_large_block(c, gamma + 1, gamma, true, true);
        } else {
            fp32_large_block(c, gamma + 1, gamma, true, true);
        }
        launch_verify(c, gamma, TANDEM_ACCEPT_NATURAL, 0ull, max_new, true, true);
        c.last_gamma = gamma;
        return;
    }
    if (bf) {
        if (kind == 0) tc_iteration(c, gamma, mode, seed, max_new); else tc_greedy_iteration(c, max_new);
        return;
    }
    if (kind == 0) fp32_iteration(c, gamma, mode, seed, max_new);
    else fp32_greedy_iteration(c, max_new);
}

// Enqueues one iteration on the context's stream: eagerly the first time a launch shape is seen (and whenever
// per-launch profiling is on), as a CUDA graph afterwards.  kind: see enqueue_iteration.
tandem_status launch_iteration(tandem_ctx& c, int kind, int gamma, int mode, uint64_t seed, int max_new) {
    const int need = (c.n_ub - 1 + gamma) / ATT_CH + 1;
    c.chunks_launch = std::min(c.lay.n_chunks_max, (need + 3) / 4 * 4);
    if (c.cfg.dtype == TANDEM_DTYPE_BF16)
        c.chunks_launch = 1;   // the cluster attention's grid does not depend on the context length: one graph serves all
    if (kind == 3) c.router_ticket++; else if (kind != 5) c.ticket++;   // what the host will wait for: the router's or the verify kernel's publication
    if (kind != 3 && kind != 5) { c.last_gamma = kind == 1 ? 0 : gamma; c.hidden_at = c.lay.h_large; }   // (set here, not while enqueueing: a replayed graph enqueues nothing on the host)
    // (A draft step of the adaptive block length starts when the host has seen the router's answer to the one before: a graph of all of
    // it would add its launch's latency to every step, 12.8 ms against 11.5 ms for 48 tokens of the small pair, and launched one by one
    // its kernels come slower than the GPU runs them.  So the first layer's kernels go out by themselves, the rest as a graph
    // behind them: 10.40 -> 10.16 ms.)
    if (c.prof.on || !c.use_graphs || kind == 3) {
        enqueue_iteration(c, kind, gamma, mode, seed, max_new);
        return check_launch();
    }
    tandem_ctx::GraphEntry* g = nullptr;
    for (auto& e : c.graphs)
        if (e.kind == kind && e.gamma == gamma && e.mode == mode && e.max_new == max_new && e.batch == c.batch &&
            e.chunks == c.chunks_launch && e.seed == seed) { g = &e; break; }
    if (!g) {
        c.graphs.push_back({kind, gamma, mode, max_new, c.batch, c.chunks_launch, seed, false, nullptr, 0});
        g = &c.graphs.back();
    }
    if (!g->warm) {   // first use: run eagerly (sets kernel attributes, surfaces launch errors outside a capture)
        g->warm = true;
        enqueue_iteration(c, kind, gamma, mode, seed, max_new);
        return check_launch();
    }
    if (!g->exec) {
        cudaStream_t user = c.stream;
        const int64_t l0 = c.launches;
        CK(cudaStreamBeginCapture(c.cap_stream, cudaStreamCaptureModeThreadLocal));
        c.stream = c.cap_stream;
        enqueue_iteration(c, kind, gamma, mode, seed, max_new);
        c.stream = user;
        cudaGraph_t graph = nullptr;
        cudaError_t e = cudaStreamEndCapture(c.cap_stream, &graph);
        g->kernels = c.launches - l0;
        c.launches = l0;
        if (e == cudaSuccess) e = cudaGraphInstantiate(&g->exec, graph, 0);
        if (graph) cudaGraphDestroy(graph);
        if (e != cudaSuccess) {
            g->exec = nullptr;
            snprintf(g_cuda_err, sizeof(g_cuda_err), "%s while capturing an iteration", cudaGetErrorString(e));
            return TANDEM_ERR_CUDA;
        }
    }
    CK(cudaGraphLaunch(g->exec, c.stream));
    c.launches += g->kernels;
    return TANDEM_OK;
}

// Waits (bounded) until the kernel that publishes into slot `slot` of the host flags (0: verify kernel, 5: router)
// has reached the given ticket.
tandem_status wait_ticket(tandem_ctx& c, int64_t ticket, int slot = 0) {
    volatile int32_t* hf = c.hflags + slot;
    struct timespec t0, t1;
    clock_gettime(CLOCK_MONOTONIC, &t0);
    for (unsigned spin = 0; (int64_t)hf[0] < ticket; ++spin) {
        if ((spin & 1023) == 1023) {
            if (cudaStreamQuery(c.stream) != cudaErrorNotReady && (int64_t)hf[0] < ticket) {
                // the stream drained (or failed) without publishing: report instead of spinning forever
                cudaError_t e = cudaStreamSynchronize(c.stream);
                if ((int64_t)hf[0] >= ticket) break;
                snprintf(g_cuda_err, sizeof(g_cuda_err), "%s while waiting for an iteration", cudaGetErrorString(e));
                return e == cudaSuccess ? TANDEM_ERR_TIMEOUT : TANDEM_ERR_CUDA;
            }
            clock_gettime(CLOCK_MONOTONIC, &t1);
            if (t1.tv_sec - t0.tv_sec > 60) return TANDEM_ERR_TIMEOUT;
        }
    }
    __sync_synchronize();
    return TANDEM_OK;
}

tandem_status begin_call(tandem_ctx* c) {
    if (!c) return TANDEM_ERR_INVALID_ARG;
    CK(cudaSetDevice(c->cfg.device));
    return TANDEM_OK;
}

void launch_call_begin(tandem_ctx& c, bool clear_hist) {
    call_begin_kernel<<<1 + c.n_lns, 256, 0, c.stream>>>(c.st, c.batch, clear_hist, at<LnSource>(c, c.lay.ln_src));
    c.launches++;
}

}  // namespace
// =====================================================================================================
// exported entry points
// =====================================================================================================

extern "C" const char* tandem_status_string(tandem_status s) {
    switch (s) {
        case TANDEM_OK: return "ok";
        case TANDEM_ERR_INVALID_ARG: return "invalid argument";
        case TANDEM_ERR_SHAPE: return "unsupported shape";
        case TANDEM_ERR_ARENA_TOO_SMALL: return "arena too small";
        case TANDEM_ERR_CAPACITY: return "capacity exceeded";
        case TANDEM_ERR_STATE: return "call out of order";
        case TANDEM_ERR_CUDA: return "CUDA error";
        case TANDEM_ERR_TIMEOUT: return "device wait timed out";
        case TANDEM_ERR_UNIMPLEMENTED: return "not implemented";
    }
    return "unknown status";
}

extern "C" const char* tandem_last_cuda_error(void) { return g_cuda_err; }

extern "C" tandem_status tandem_query_arena(const tandem_config* cfg, size_t* bytes) {
    if (!bytes) return TANDEM_ERR_INVALID_ARG;
    TRY(validate(cfg));
    *bytes = make_layout(*cfg).total;
    return TANDEM_OK;
}

namespace {
void release_side(tandem_ctx& c) {
    for (cudaEvent_t ev : c.ev_fork) cudaEventDestroy(ev);
    c.ev_fork.clear();
    if (c.ev_join) { cudaEventDestroy(c.ev_join); c.ev_join = nullptr; }
    if (c.ev_staged) { cudaEventDestroy(c.ev_staged); c.ev_staged = nullptr; }
    if (c.side) { cudaStreamDestroy(c.side); c.side = nullptr; }
}
}  // namespace

extern "C" tandem_status tandem_create(const tandem_config* cfg, const tandem_weights* weights, void* arena,
                                       size_t arena_bytes, tandem_ctx** out) {
    if (!out || !weights || !weights->ptrs || !arena) return TANDEM_ERR_INVALID_ARG;
    TRY(validate(cfg));
    if (weights->n_ptrs != n_weight_ptrs(*cfg)) return TANDEM_ERR_INVALID_ARG;
    for (int i = 0; i < weights->n_ptrs; ++i)
        if (!weights->ptrs[i] || ((uintptr_t)weights->ptrs[i] & 15)) return TANDEM_ERR_INVALID_ARG;
    if ((uintptr_t)arena & 255) return TANDEM_ERR_INVALID_ARG;
    Layout lay = make_layout(*cfg);
    if (arena_bytes < lay.total) return TANDEM_ERR_ARENA_TOO_SMALL;
    CK(cudaSetDevice(cfg->device));

    tandem_ctx* c = new (std::nothrow) tandem_ctx();
    if (!c) return TANDEM_ERR_INVALID_ARG;
    c->cfg = *cfg;
    c->layer_map.assign(cfg->layer_map, cfg->layer_map + cfg->small.n_layers);
    c->cfg.layer_map = c->layer_map.data();
    c->w.assign(weights->ptrs, weights->ptrs + weights->n_ptrs);
    c->lay = lay;
    c->arena = static_cast<unsigned char*>(arena);
    c->stream = static_cast<cudaStream_t>(cfg->stream);
    c->esz = cfg->dtype == TANDEM_DTYPE_BF16 ? 2 : 4;
    c->hidden = cfg->ff_tandem_hidden > 0 ? cfg->ff_tandem_hidden : cfg->small.d_model;
    c->large.kv_heads = kv_heads_of(cfg->large); c->large.d_kv = d_kv_of(cfg->large);
    c->small.kv_heads = kv_heads_of(cfg->small); c->small.d_kv = d_kv_of(cfg->small);
    c->large.d = cfg->large; c->large.wbase = 0; c->large.kv_off = lay.kv_large; c->large.kv_layer_elems = lay.kv_large_layer;
    c->small.d = cfg->small; c->small.wbase = 5 + 10 * cfg->large.n_layers; c->small.kv_off = lay.kv_small; c->small.kv_layer_elems = lay.kv_small_layer;
    c->tbase = c->small.wbase + 5 + 10 * cfg->small.n_layers;
    c->batch = 0; c->n_ub = 0; c->launches = 0; c->last_gamma = 0; c->hidden_at = lay.h_large;
    c->pinned_ints = std::max((size_t)lay.max_rows + 5 * cfg->max_batch + 64,
                              (size_t)cfg->max_batch * (2 * cfg->max_seq + 4) + 2 * 64 + 64);   // prompt rows going in; tokens, counters, histogram, lengths, scores coming out
    c->pinned = nullptr;
    LoopState& st = c->st;
    st.n = at<int>(*c, lay.st_n); st.pending = at<int>(*c, lay.st_pending); st.drafts = at<int>(*c, lay.st_drafts);
    st.targets = at<int>(*c, lay.st_targets); st.accept_len = at<int>(*c, lay.st_accept); st.emitted = at<int>(*c, lay.st_emitted);
    st.done = at<int>(*c, lay.st_done); st.out_ids = at<int>(*c, lay.st_out); st.counters = at<int>(*c, lay.st_counters);
    st.hist = at<unsigned long long>(*c, lay.st_hist);
    st.block_len = at<int>(*c, lay.st_block_len); st.drafting = at<int>(*c, lay.st_drafting);
    st.confidence = at<float>(*c, lay.st_confidence);
    st.out_cap = cfg->max_seq; st.gamma_limit = TANDEM_GAMMA_LIMIT;
    cudaError_t e = cudaMallocHost(reinterpret_cast<void**>(&c->pinned), c->pinned_ints * sizeof(int32_t));
    if (e == cudaSuccess) e = cudaHostAlloc(reinterpret_cast<void**>(&c->hflags), 16 * sizeof(int32_t), cudaHostAllocMapped);
    if (e == cudaSuccess) {
        memset(c->hflags, 0, 16 * sizeof(int32_t));
        int* dptr = nullptr;
        e = cudaHostGetDevicePointer(reinterpret_cast<void**>(&dptr), c->hflags, 0);
        st.host_flags = dptr;
    }
    if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&c->cap_stream, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&c->side, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&c->ev_join, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&c->ev_staged, cudaEventDisableTiming);
    for (int j = 0; j < cfg->small.n_layers && e == cudaSuccess; ++j) {
        cudaEvent_t ev = nullptr;
        e = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming);
        if (e == cudaSuccess) c->ev_fork.push_back(ev);
    }
    // Two diagnostic switches, read here once (see tandem.h): launch every kernel eagerly instead of replaying a
    // graph, and plain stream order instead of programmatic dependent launch.  Neither changes any result.
    c->use_graphs = getenv("TANDEM_NO_GRAPH") == nullptr;
    c->use_pdl = getenv("TANDEM_NO_PDL") == nullptr;
    c->n_sms = sm_count();
    c->amax_tiles = lay.vocab_tiles;
    if (e == cudaSuccess && cfg->dtype == TANDEM_DTYPE_BF16) {
        // two tensor maps per weight matrix: [out_features][in_features], 128 x 64 tiles and 32 x 64
        c->wmap.resize(c->w.size());
        c->wpart.resize(c->w.size());
        bool ok = tmap_encoder() != nullptr;
        auto add = [&](int idx, int rows, int cols) {
            ok = ok && make_tmap_bf16(&c->wmap[idx], c->w[idx], (uint64_t)rows, (uint64_t)cols, (uint64_t)cols) &&
                 make_tmap_bf16(&c->wpart[idx], c->w[idx], (uint64_t)rows, (uint64_t)cols, (uint64_t)cols, 32);
        };
        for (const Model* m : {&c->large, &c->small}) {
            const int d = m->d.d_model, dff = m->d.d_ff;
            for (int l = 0; l < m->d.n_layers; ++l) {
                add(wi_layer(*m, l, W_WQ), d, d); add(wi_layer(*m, l, W_WK), m->d_kv, d); add(wi_layer(*m, l, W_WV), m->d_kv, d);
                add(wi_layer(*m, l, W_WO), d, d); add(wi_layer(*m, l, W_W1), dff, d); add(wi_layer(*m, l, W_W2), d, dff);
            }
            add(wi_tail(*m, 2), m->d.vocab, d);
        }
        for (int j = 0; j < cfg->small.n_layers; ++j) {
            if (cfg->ff_tandem_kind == TANDEM_FF_LINEAR) add(wi_tandem(*c, j, 0), cfg->small.d_model, cfg->large.d_model);
            else { add(wi_tandem(*c, j, 0), c->hidden, cfg->large.d_model); add(wi_tandem(*c, j, 1), cfg->small.d_model, c->hidden); }
        }
        for (int mi = 0; mi < 2; ++mi) {   // decode activations and the LayerNorms' rows
            const Model& mm = mi == 0 ? c->large : c->small;
            for (int buf = 0; buf < 3; ++buf) {
                const uint64_t K = buf == 2 ? mm.d.d_ff : mm.d.d_model;
                const size_t at_off = buf == 0 ? lay.a32 : (buf == 1 ? lay.o32 : lay.f32);
                ok = ok && make_tmap_planes(&c->xmap[buf][mi], c->arena + at_off, (uint64_t)lay.dec_rows, K);
            }
            const uint64_t d = mm.d.d_model, n_ln = 2 * mm.d.n_layers + 1;
            ok = ok && make_tmap_bf16(&c->lnmap[mi], c->arena + (mi == 0 ? lay.ln_rows_large : lay.ln_rows_small), 4 * n_ln, d, d, 4);
        }
        std::vector<LnSource> lns;
        for (int mi = 0; mi < 2; ++mi) {
            const Model& mm = mi == 0 ? c->large : c->small;
            bf16* rows = at<bf16>(*c, mi == 0 ? lay.ln_rows_large : lay.ln_rows_small);
            for (int i = 0; i <= 2 * mm.d.n_layers; ++i) {
                const bool last = i == 2 * mm.d.n_layers;
                const void* b = last ? w_tail(*c, mm, 1) : w_layer(*c, mm, i / 2, i % 2 ? W_LN2B : W_LN1B);
                lns.push_back({static_cast<const float*>(ln_gain(*c, mm, i)), static_cast<const float*>(b), rows + (size_t)i * 4 * mm.d.d_model, mm.d.d_model});
            }
        }
        c->n_lns = (int)lns.size();
        e = cudaMemcpyAsync(c->arena + lay.ln_src, lns.data(), lns.size() * sizeof(LnSource), cudaMemcpyHostToDevice, c->stream);   // (pageable: staged before the call returns)
        if (!ok) {
            snprintf(g_cuda_err, sizeof(g_cuda_err), "cuTensorMapEncodeTiled unavailable or failed for a weight matrix");
            if (c->pinned) cudaFreeHost(c->pinned);
            if (c->hflags) cudaFreeHost(c->hflags);
            if (c->cap_stream) cudaStreamDestroy(c->cap_stream);
            release_side(*c);
            delete c;
            return TANDEM_ERR_CUDA;
        }
        const int dhL = cfg->large.d_model / cfg->large.n_heads;
        if (dhL == 64 || dhL == 128) {
            c->kmap.resize(cfg->large.n_layers);
            c->vmap.resize(cfg->large.n_layers);
            bool okm = true;
            const unsigned atc_kc = dhL == 128 ? AtcCfg<128>::KC : AtcCfg<64>::KC;
            const uint64_t kv_rows = (uint64_t)cfg->max_batch * c->large.kv_heads * cfg->max_seq;
            for (int l = 0; l < cfg->large.n_layers && okm; ++l)
                okm = make_tmap_bf16(&c->kmap[l], kv_ptr<bf16>(*c, c->large, l, 0), kv_rows, (uint64_t)dhL, (uint64_t)dhL, atc_kc) &&
                      make_tmap_bf16(&c->vmap[l], kv_ptr<bf16>(*c, c->large, l, 1), kv_rows, (uint64_t)dhL, (uint64_t)dhL, atc_kc);
            if (okm) { c->tc_prompt_attn = true; c->prompt_group = ATC_Q; }
        }
    }
    if (e == cudaSuccess) e = cudaMemsetAsync(c->arena + lay.st_n, 0, lay.h_large - lay.st_n, c->stream);
    // positions nobody has written yet are read (and masked, or weighted by zero) by chunked attention: keep them finite
    if (e == cudaSuccess) e = cudaMemsetAsync(c->arena + lay.kv_large, 0, lay.st_n - lay.kv_large, c->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
    if (e != cudaSuccess) {
        snprintf(g_cuda_err, sizeof(g_cuda_err), "%s in tandem_create", cudaGetErrorString(e));
        if (c->pinned) cudaFreeHost(c->pinned);
        if (c->hflags) cudaFreeHost(c->hflags);
        if (c->cap_stream) cudaStreamDestroy(c->cap_stream);
            release_side(*c);
        delete c;
        return TANDEM_ERR_CUDA;
    }
    *out = c;
    return TANDEM_OK;
}

extern "C" tandem_status tandem_destroy(tandem_ctx* c) {
    if (!c) return TANDEM_ERR_INVALID_ARG;
    cudaSetDevice(c->cfg.device);
    cudaError_t e = cudaStreamSynchronize(c->stream);
    if (c->pinned) cudaFreeHost(c->pinned);
    for (cudaEvent_t ev : c->prof.ev) cudaEventDestroy(ev);
    for (auto& g : c->graphs) if (g.exec) cudaGraphExecDestroy(g.exec);
    if (c->hflags) cudaFreeHost(c->hflags);
    if (c->cap_stream) cudaStreamDestroy(c->cap_stream);
    release_side(*c);
    delete c;
    if (e != cudaSuccess) {
        snprintf(g_cuda_err, sizeof(g_cuda_err), "%s in tandem_destroy", cudaGetErrorString(e));
        return TANDEM_ERR_CUDA;
    }
    return TANDEM_OK;
}

namespace {

// Prompt pass for n_queries prompts, each the start of `samples` sequences (query q owns sequences q * samples ..
// q * samples + samples - 1).  The large model reads each prompt once, into the first sequence of its query; the
// other sequences of the query get copies of the keys / values it produced (both caches) and the same pending token.
tandem_status prefill_impl(tandem_ctx* c, int n_queries, int samples, const int32_t* prompt_ids, const int32_t* prompt_lens) {
    if (!prompt_ids || !prompt_lens || n_queries < 1 || samples < 1) return TANDEM_ERR_INVALID_ARG;
    const long long batch_ll = (long long)n_queries * samples;
    if (batch_ll > c->cfg.max_batch) return TANDEM_ERR_CAPACITY;
    const int batch = (int)batch_ll;
    const int pos_cap = std::min(c->cfg.max_seq, std::min(c->cfg.large.max_pos, c->cfg.small.max_pos));
    long long rows = 0, total = 0, total_ids = 0;
    int n_max = 0;
    for (int q = 0; q < n_queries; ++q) {
        if (prompt_lens[q] < 1) return TANDEM_ERR_INVALID_ARG;
        if (prompt_lens[q] > pos_cap) return TANDEM_ERR_CAPACITY;
        rows += prompt_lens[q] - 1;
        total += (long long)prompt_lens[q] * samples;
        total_ids += prompt_lens[q];
        n_max = std::max(n_max, prompt_lens[q]);
    }
    if (rows > c->lay.max_rows) return TANDEM_ERR_CAPACITY;
    for (long long i = 0; i < total_ids; ++i)
        if (prompt_ids[i] < 0 || prompt_ids[i] >= c->cfg.large.vocab) return TANDEM_ERR_INVALID_ARG;

    // Queries per attention group: two tiles of 128 for a CTA of the tensor-core kernel, one where that leaves more than half of the
    // multiprocessors without a CTA (small pair's prompt passes of 512 / 900 tokens, 16 heads: 696 -> 685, 884 -> 848 us).
    int group = c->prompt_group;
    if (c->tc_prompt_attn && (rows / ATC_Q + n_queries) * c->cfg.large.n_heads * 2 <= c->n_sms) group = ATC_TILE;
    // The pass is enqueued behind whatever the stream still runs; only the staging buffer has to be free again, which it is
    // as soon as the previous pass's copy has gone.  (Everything else that uses the buffer waits before it returns.)
    CK(cudaEventSynchronize(c->ev_staged));
    const int M = (int)rows;
    int32_t* p_len = c->pinned;
    int32_t *p_id = p_len + n_queries, *p_row = p_id + n_queries, *p_grp = p_row + n_queries, *p_ids = p_grp + n_queries;
    int m = 0, groups = 0;
    long long off = 0;
    for (int q = 0; q < n_queries; ++q) {
        p_len[q] = prompt_lens[q]; p_id[q] = (int)off; p_row[q] = m; p_grp[q] = groups;
        off += prompt_lens[q];
        m += prompt_lens[q] - 1;
        groups += cdiv(prompt_lens[q] - 1, group);
    }
    memcpy(p_ids, prompt_ids, (size_t)total_ids * 4);
    cudaStream_t s = c->stream;
    CK(cudaMemsetAsync(c->arena + c->lay.st_n, 0, c->lay.row_tok - c->lay.st_n, s));
    CK(cudaMemcpyAsync(c->arena + c->lay.stage, c->pinned, ((size_t)4 * n_queries + total_ids) * 4, cudaMemcpyHostToDevice, s));
    CK(cudaEventRecord(c->ev_staged, s));
    c->batch = batch;
    c->n_ub = n_max;
    c->hidden_at = c->lay.h_large;
    c->n_sum = total;
    c->prompt_sq_sum = 0.0;
    for (int q = 0; q < n_queries; ++q) c->prompt_sq_sum += (double)(prompt_lens[q] - 1) * (prompt_lens[q] - 1);
    PromptStage ps;
    ps.len = at<int>(*c, c->lay.stage); ps.id_off = ps.len + n_queries; ps.row_off = ps.id_off + n_queries; ps.grp_off = ps.row_off + n_queries;
    ps.ids = ps.grp_off + n_queries;
    ps.n_queries = n_queries; ps.samples = samples; ps.rows = M; ps.group = group;
    const bool bf = c->cfg.dtype == TANDEM_DTYPE_BF16;
    {
        ProfScope prof(*c, PC_ROWS, (double)M * c->large.d.d_model * (4.0 + 2 * c->esz));
        auto begin = [&](auto* emb, auto* pos, auto kernel) {
            kernel<<<M + 1, 128, 0, s>>>(c->st, ps, at<int>(*c, c->lay.row_tok), at<int>(*c, c->lay.row_seq), at<int>(*c, c->lay.row_pos),
                                         at<int>(*c, c->lay.grp_row0), at<int>(*c, c->lay.grp_cnt), emb, pos, at<float>(*c, c->lay.h_large),
                                         c->large.d.d_model, (int)c->ticket, (int)c->router_ticket);
        };
        if (bf) begin((const bf16*)w_emb(*c, c->large), (const bf16*)w_pos(*c, c->large), prompt_begin_kernel<bf16>);
        else begin((const float*)w_emb(*c, c->large), (const float*)w_pos(*c, c->large), prompt_begin_kernel<float>);
        c->launches++;
    }
    if (M > 0) {
        Rows r; r.M = M; r.groups = groups; r.nq = 0; r.decode = false; r.n_chunks = 0; r.kv_positions = (double)rows;
        if (bf) large_layers<bf16>(*c, r, true);
        else large_layers<float>(*c, r, true);
    }
    if (samples > 1 && M > 0) {
        for (const Model* mdl : {&c->large, &c->small}) {
            const int row_bytes = mdl->d.d_model / mdl->d.n_heads * (int)c->esz;
            ProfScope prof(*c, PC_ROWS, 0.0);
            copy_samples_kernel<<<dim3(mdl->d.n_layers * 2, mdl->kv_heads, n_queries), 256, 0, s>>>(c->arena + mdl->kv_off, mdl->kv_layer_elems * c->esz,
                                                                                                 samples, c->cfg.max_seq, row_bytes, ps.len);
            c->launches++;
        }
    }
    return check_launch(*c);
}

}  // namespace

extern "C" tandem_status tandem_prefill(tandem_ctx* c, int32_t batch, const int32_t* prompt_ids, const int32_t* prompt_lens) {
    TRY(begin_call(c));
    return prefill_impl(c, batch, 1, prompt_ids, prompt_lens);
}

extern "C" tandem_status tandem_prefill_samples(tandem_ctx* c, int32_t n_queries, int32_t num_samples, const int32_t* prompt_ids,
                                                const int32_t* prompt_lens) {
    TRY(begin_call(c));
    return prefill_impl(c, n_queries, num_samples, prompt_ids, prompt_lens);
}

namespace {

tandem_status capacity_for(tandem_ctx* c, int extra_tokens, int gamma) {
    const int pos_cap = std::min(c->cfg.max_seq, std::min(c->cfg.large.max_pos, c->cfg.small.max_pos));
    // rows of the last iteration reach position (n_ub + extra - 1) + gamma
    if ((long long)c->n_ub + extra_tokens + gamma > pos_cap) return TANDEM_ERR_CAPACITY;
    return TANDEM_OK;
}

}  // namespace

extern "C" tandem_status tandem_block_step(tandem_ctx* c, int32_t gamma, int32_t accept_mode, uint64_t mode_seed,
                                           tandem_step_result* result) {
    TRY(begin_call(c));
    if (gamma < 0 || gamma > c->cfg.gamma_max || accept_mode < 0 || accept_mode > 4) return TANDEM_ERR_INVALID_ARG;
    if (accept_mode == TANDEM_ACCEPT_REPRESENTATION_ONLY && gamma < 1) return TANDEM_ERR_INVALID_ARG;
    if (c->batch == 0) return TANDEM_ERR_STATE;
    TRY(capacity_for(c, 0, gamma));
    launch_call_begin(*c, false);
    TRY(launch_iteration(*c, 0, gamma, accept_mode, mode_seed, INT_MAX));
    c->n_ub += gamma + 1;
    c->n_sum += (long long)c->batch * (gamma + 1);
    if (result) {
        int32_t* cnt = c->pinned;   // staging is idle outside prefill
        CK(cudaMemcpyAsync(cnt, c->st.counters, 5 * 4, cudaMemcpyDeviceToHost, c->stream));
        const int B = c->batch, GL = TANDEM_GAMMA_LIMIT;
        // everything lands in private buffers first: the caller's arrays are written only once the iteration is known to be good
        std::vector<int32_t> d((size_t)B * GL), t((size_t)B * (GL + 1)), acc((size_t)B), ncm((size_t)B);
        if (result->drafts) CK(cudaMemcpyAsync(d.data(), c->st.drafts, d.size() * 4, cudaMemcpyDeviceToHost, c->stream));
        if (result->targets) CK(cudaMemcpyAsync(t.data(), c->st.targets, t.size() * 4, cudaMemcpyDeviceToHost, c->stream));
        if (result->accept_len) CK(cudaMemcpyAsync(acc.data(), c->st.accept_len, (size_t)B * 4, cudaMemcpyDeviceToHost, c->stream));
        if (result->n_committed) CK(cudaMemcpyAsync(ncm.data(), c->st.n, (size_t)B * 4, cudaMemcpyDeviceToHost, c->stream));
        CK(cudaStreamSynchronize(c->stream));
        c->n_ub = cnt[3];
        c->n_sum = cnt[4];
        if (cnt[2] != 0) {
            snprintf(g_cuda_err, sizeof(g_cuda_err), "device-side wait expired (code %d)", cnt[2]);
            CK(cudaMemsetAsync(c->st.counters + 2, 0, 4, c->stream));
            return TANDEM_ERR_TIMEOUT;
        }
        for (int b = 0; b < B; ++b) {
            if (result->drafts) for (int i = 0; i < gamma; ++i) result->drafts[b * gamma + i] = d[(size_t)b * GL + i];
            if (result->targets) for (int i = 0; i <= gamma; ++i)   // no predictions of the large model in a representation-only round
                result->targets[b * (gamma + 1) + i] = accept_mode == TANDEM_ACCEPT_REPRESENTATION_ONLY ? -1 : t[(size_t)b * (GL + 1) + i];
            if (result->accept_len) result->accept_len[b] = acc[b];
            if (result->n_committed) result->n_committed[b] = ncm[b];
        }
    }
    return TANDEM_OK;
}

namespace {

// End of a generate call: counters, histogram, lengths and tokens come back in two copies behind one wait; the caller's
// buffers are written only once the call is known to be good.
tandem_status read_results(tandem_ctx* c, int max_new, int32_t* out_ids, int32_t* out_lens, unsigned long long* hist, int64_t* iters) {
    const int B = c->batch;
    int32_t* ids = c->pinned;   // staging is idle outside prefill
    unsigned char* tail = reinterpret_cast<unsigned char*>(c->pinned + align_up((size_t)B * max_new, 64));
    const size_t tail_bytes = c->lay.st_emitted + (size_t)B * 4 - c->lay.st_counters;
    CK(cudaMemcpyAsync(tail, c->arena + c->lay.st_counters, tail_bytes, cudaMemcpyDeviceToHost, c->stream));
    CK(cudaMemcpy2DAsync(ids, (size_t)max_new * 4, c->st.out_ids, (size_t)c->st.out_cap * 4, (size_t)max_new * 4, B,
                         cudaMemcpyDeviceToHost, c->stream));
    CK(cudaStreamSynchronize(c->stream));
    const int32_t* cnt = reinterpret_cast<const int32_t*>(tail);
    c->n_ub = cnt[3];
    c->n_sum = cnt[4];
    if (cnt[2] != 0) {   // a bounded device-side wait gave up somewhere in this call
        snprintf(g_cuda_err, sizeof(g_cuda_err), "device-side wait expired (code %d)", cnt[2]);
        CK(cudaMemsetAsync(c->st.counters + 2, 0, 4, c->stream));
        return TANDEM_ERR_TIMEOUT;
    }
    *iters = cnt[5];
    memcpy(hist, tail + (c->lay.st_hist - c->lay.st_counters), (TANDEM_GAMMA_LIMIT + 1) * 8);
    memcpy(out_ids, ids, (size_t)B * max_new * 4);
    if (out_lens) memcpy(out_lens, tail + (c->lay.st_emitted - c->lay.st_counters), (size_t)B * 4);
    return TANDEM_OK;
}

// lead_large_step: the call starts with one round of the large model alone over the pending token (a block of one
// row with projection and output head), which gives the first new token (Figure 2, left).
tandem_status run_generate(tandem_ctx* c, bool speculative, int gamma, int max_new, int mode, uint64_t seed,
                           int32_t* out_ids, int32_t* out_lens, tandem_stats* stats, bool lead_large_step = false) {
    if (!out_ids || max_new < 1) return TANDEM_ERR_INVALID_ARG;
    if (c->batch == 0) return TANDEM_ERR_STATE;
    if (max_new > c->cfg.max_seq) return TANDEM_ERR_CAPACITY;
    TRY(capacity_for(c, max_new, gamma));
    const int B = c->batch;
    const int64_t launches0 = c->launches;
    launch_call_begin(*c, true);
    // Iterations are enqueued ahead of the host's knowledge of their outcome, but only those that are certain to be
    // needed: every iteration gives a sequence at most per_iter tokens, so with `left` tokens still wanted by some
    // sequence after the last observed iteration, ceil(left / per_iter) more must run whatever is accepted.  Beyond
    // those the host waits for a result: a launch into an idle GPU costs about 10 us, a surplus iteration, which would find
    // every sequence frozen and change nothing, a whole pass (two of them at the end of a call were 8 % of a small
    // 64-token response and 15 % of the decode phase of a 32-token one).
    const int kind = speculative ? 0 : 1;
    const int64_t ticket0 = c->ticket;
    const int per_iter = (mode == TANDEM_ACCEPT_REPRESENTATION_ONLY || mode == 5) ? gamma : gamma + 1;   // most tokens one iteration can emit
    const int lead = lead_large_step ? 1 : 0;
    const int n_known0 = c->n_ub;
    int64_t enq = 0, seen = 0;   // iterations of this call enqueued / observed
    int n_known = n_known0;      // max_b n_b after the last observed iteration
    int64_t certain = lead + (max_new - lead + per_iter - 1) / per_iter;   // iterations that must follow the last observed one
    for (;;) {
        if (enq - seen >= certain) TRY(wait_ticket(*c, ticket0 + seen + 1));
        // take whatever has been published so far
        const int64_t pub = (int64_t)((volatile int32_t*)c->hflags)[0] - ticket0;
        if (pub > seen) {
            __sync_synchronize();
            seen = std::min<int64_t>(pub, enq);
            n_known = c->hflags[2];
            c->n_sum = c->hflags[3];
            if (c->hflags[1] <= 0) break;
            certain = std::max(1, (c->hflags[7] + per_iter - 1) / per_iter);
        }
        if (enq - seen >= certain) continue;
        if (enq > (int64_t)max_new + 1) return TANDEM_ERR_STATE;   // every live iteration emits a token
        c->n_ub = std::min<long long>((long long)n_known + (enq - seen) * (gamma + 1), (long long)n_known0 + max_new);
        if (lead && enq == 0) TRY(launch_iteration(*c, 0, 0, TANDEM_ACCEPT_NATURAL, 0ull, max_new));
        else TRY(launch_iteration(*c, kind, gamma, mode, seed, max_new));
        ++enq;
    }
    int64_t iters = 0;
    std::vector<unsigned long long> hist(TANDEM_GAMMA_LIMIT + 1);
    TRY(read_results(c, max_new, out_ids, out_lens, hist.data(), &iters));
    TRY(check_launch());
    if (stats) {
        memset(stats, 0, sizeof(*stats));
        stats->iterations = iters;
        stats->large_runs = iters;
        stats->small_runs = speculative ? std::max<int64_t>(0, iters - lead) * gamma : 0;
        stats->emitted = (int64_t)B * max_new;
        for (int i = 0; i <= TANDEM_GAMMA_LIMIT; ++i) stats->accept_hist[i] = (int64_t)hist[i];
        stats->kernel_launches = c->launches - launches0;
    }
    return TANDEM_OK;
}

}  // namespace

namespace {

// One adaptive iteration, synchronous: draft steps until the router has stopped every sequence (the host reads the
// count the router publishes after each step) or gamma_max drafts exist, then one verify pass over the longest block.
tandem_status adaptive_iteration(tandem_ctx* c, int gamma_max, int max_new, int* block_max) {
    int s = 0;
    for (; s < gamma_max; ++s) {
        TRY(launch_iteration(*c, 3, s, gamma_max, 0ull, max_new));
        if (c->cfg.dtype == TANDEM_DTYPE_BF16) TRY(launch_iteration(*c, 5, s, gamma_max, 0ull, 0));   // (no step depends on the tokens asked for: one graph for every length of response)
        TRY(wait_ticket(*c, c->router_ticket, 5));
        if (c->hflags[6] <= 0) { ++s; break; }
    }
    *block_max = s;
    TRY(launch_iteration(*c, 4, s, 0, 0ull, max_new));
    TRY(wait_ticket(*c, c->ticket, 0));
    c->n_ub = c->hflags[2];
    c->n_sum = c->hflags[3];
    return TANDEM_OK;
}

tandem_status check_error_word(tandem_ctx* c) {
    int32_t* cnt = c->pinned;   // staging is idle outside prefill
    CK(cudaMemcpyAsync(cnt, c->st.counters, 8 * 4, cudaMemcpyDeviceToHost, c->stream));
    CK(cudaStreamSynchronize(c->stream));
    if (cnt[2] != 0) {
        snprintf(g_cuda_err, sizeof(g_cuda_err), "device-side wait expired (code %d)", cnt[2]);
        CK(cudaMemsetAsync(c->st.counters + 2, 0, 4, c->stream));
        return TANDEM_ERR_TIMEOUT;
    }
    return TANDEM_OK;
}

}  // namespace

extern "C" tandem_status tandem_set_router(tandem_ctx* c, int32_t top_k, int32_t hidden, const void* w1, const void* b1, const void* w2,
                                           float b2, float tau) {
    TRY(begin_call(c));
    if (!w1 || !b1 || !w2 || top_k < 1 || top_k > RT_MAX_K || hidden < 1 || top_k > c->cfg.small.vocab) return TANDEM_ERR_INVALID_ARG;
    if (((uintptr_t)w1 | (uintptr_t)b1 | (uintptr_t)w2) & 3) return TANDEM_ERR_INVALID_ARG;
    if (sizeof(float) * (size_t)(1 + top_k + (size_t)top_k * c->cfg.small.d_model) > 48 * 1024) return TANDEM_ERR_SHAPE;   // the feature vector sits in shared memory
    CK(cudaStreamSynchronize(c->stream));   // the caller may release the former router's weights
    for (auto& g : c->graphs)               // (they are arguments of the captured draft steps)
        if (g.kind == 5 && g.exec) { cudaGraphExecDestroy(g.exec); g.exec = nullptr; }
    c->router.w1 = static_cast<const float*>(w1); c->router.b1 = static_cast<const float*>(b1); c->router.w2 = static_cast<const float*>(w2);
    c->router.b2 = b2; c->router.tau = tau; c->router.k = top_k; c->router.hidden = hidden;
    c->has_router = true;
    return TANDEM_OK;
}

extern "C" tandem_status tandem_adaptive_step(tandem_ctx* c, int32_t gamma_max, tandem_step_result* result, int32_t* block_len,
                                              float* confidence) {
    TRY(begin_call(c));
    if (gamma_max < 1 || gamma_max > c->cfg.gamma_max) return TANDEM_ERR_INVALID_ARG;
    if (c->batch == 0 || !c->has_router) return TANDEM_ERR_STATE;
    TRY(capacity_for(c, 0, gamma_max));
    launch_call_begin(*c, false);
    int block_max = 0;
    TRY(adaptive_iteration(c, gamma_max, INT_MAX, &block_max));
    TRY(check_error_word(c));
    const int B = c->batch, GL = TANDEM_GAMMA_LIMIT;
    std::vector<int32_t> d((size_t)B * GL), t((size_t)B * (GL + 1)), acc((size_t)B), ncm((size_t)B), bl((size_t)B);
    std::vector<float> cf((size_t)B * GL);
    CK(cudaMemcpyAsync(d.data(), c->st.drafts, d.size() * 4, cudaMemcpyDeviceToHost, c->stream));
    CK(cudaMemcpyAsync(t.data(), c->st.targets, t.size() * 4, cudaMemcpyDeviceToHost, c->stream));
    CK(cudaMemcpyAsync(acc.data(), c->st.accept_len, (size_t)B * 4, cudaMemcpyDeviceToHost, c->stream));
    CK(cudaMemcpyAsync(ncm.data(), c->st.n, (size_t)B * 4, cudaMemcpyDeviceToHost, c->stream));
    CK(cudaMemcpyAsync(bl.data(), c->st.block_len, (size_t)B * 4, cudaMemcpyDeviceToHost, c->stream));
    CK(cudaMemcpyAsync(cf.data(), c->st.confidence, cf.size() * 4, cudaMemcpyDeviceToHost, c->stream));
    CK(cudaStreamSynchronize(c->stream));
    for (int b = 0; b < B; ++b) {
        for (int i = 0; i < gamma_max; ++i) {   // entries beyond a sequence's own block length are -1 / 0
            const bool own = i < bl[b];
            if (result && result->drafts) result->drafts[b * gamma_max + i] = own ? d[(size_t)b * GL + i] : -1;
            if (confidence) confidence[b * gamma_max + i] = own ? cf[(size_t)b * GL + i] : 0.f;
        }
        if (result && result->targets) for (int i = 0; i <= gamma_max; ++i)
            result->targets[b * (gamma_max + 1) + i] = i <= bl[b] ? t[(size_t)b * (GL + 1) + i] : -1;
        if (result && result->accept_len) result->accept_len[b] = acc[b];
        if (result && result->n_committed) result->n_committed[b] = ncm[b];
        if (block_len) block_len[b] = bl[b];
    }
    return TANDEM_OK;
}

extern "C" tandem_status tandem_adaptive_generate(tandem_ctx* c, int32_t gamma_max, int32_t max_new, int32_t* out_ids, int32_t* out_lens,
                                                  tandem_stats* stats) {
    TRY(begin_call(c));
    if (gamma_max < 1 || gamma_max > c->cfg.gamma_max || !out_ids || max_new < 1) return TANDEM_ERR_INVALID_ARG;
    if (c->batch == 0 || !c->has_router) return TANDEM_ERR_STATE;
    if (max_new > c->cfg.max_seq) return TANDEM_ERR_CAPACITY;
    TRY(capacity_for(c, max_new, gamma_max));
    const int B = c->batch;
    const int64_t launches0 = c->launches;
    launch_call_begin(*c, true);
    int64_t iters = 0, small_runs = 0;
    for (;;) {
        if (iters > max_new) return TANDEM_ERR_STATE;   // every live iteration emits a token
        int block_max = 0;
        TRY(adaptive_iteration(c, gamma_max, max_new, &block_max));
        ++iters;
        small_runs += block_max;
        if (c->hflags[1] <= 0) break;
    }
    int64_t live_iters = 0;
    std::vector<unsigned long long> hist(TANDEM_GAMMA_LIMIT + 1);
    TRY(read_results(c, max_new, out_ids, out_lens, hist.data(), &live_iters));
    if (stats) {
        memset(stats, 0, sizeof(*stats));
        stats->iterations = iters;
        stats->large_runs = iters;
        stats->small_runs = small_runs;
        stats->emitted = (int64_t)B * max_new;
        for (int i = 0; i <= TANDEM_GAMMA_LIMIT; ++i) stats->accept_hist[i] = (int64_t)hist[i];
        stats->kernel_launches = c->launches - launches0;
    }
    return TANDEM_OK;
}

extern "C" tandem_status tandem_speculative_generate(tandem_ctx* c, int32_t gamma, int32_t max_new_tokens, int32_t accept_mode,
                                                     uint64_t mode_seed, int32_t* out_ids, int32_t* out_lens, tandem_stats* stats) {
    TRY(begin_call(c));
    if (gamma < 0 || gamma > c->cfg.gamma_max || accept_mode < 0 || accept_mode > 4) return TANDEM_ERR_INVALID_ARG;
    if (accept_mode == TANDEM_ACCEPT_REPRESENTATION_ONLY && gamma < 1) return TANDEM_ERR_INVALID_ARG;
    return run_generate(c, true, gamma, max_new_tokens, accept_mode, mode_seed, out_ids, out_lens, stats);
}

namespace {

// The bf16 form of the call below: one row per token that has a next one, in passes of as many as the work space holds.
tandem_status forced_forward(tandem_ctx* c, int gamma, int batch, const int32_t* ids, const int32_t* lens, long long total, float* nll, int32_t* top1) {
    CK(cudaEventSynchronize(c->ev_staged));   // (the staging buffer may still be read by a prompt pass's copy)
    int32_t *p_ids = c->pinned, *p_start = p_ids + total;
    memcpy(p_ids, ids, (size_t)total * 4);
    int rows = 0, max_len = 0;
    for (int b = 0; b < batch; ++b) {
        p_start[b] = rows;
        rows += lens[b] - 1;
        max_len = std::max(max_len, lens[b]);
    }
    p_start[batch] = rows;
    CK(cudaMemsetAsync(c->arena + c->lay.st_n, 0, c->lay.row_tok - c->lay.st_n, c->stream));
    CK(cudaMemcpyAsync(c->arena + c->lay.forced_ids, p_ids, (size_t)total * 4, cudaMemcpyHostToDevice, c->stream));
    CK(cudaMemcpyAsync(c->arena + c->lay.fr_start, p_start, (size_t)(batch + 1) * 4, cudaMemcpyHostToDevice, c->stream));
    CK(cudaEventRecord(c->ev_staged, c->stream));
    c->batch = batch; c->n_ub = max_len; c->n_sum = total; c->last_gamma = gamma;
    c->hidden_at = c->lay.proj_snap;
    launch_call_begin(*c, true);
    ForcedRows f;
    f.ids = at<int>(*c, c->lay.forced_ids); f.start = at<int>(*c, c->lay.fr_start); f.truth = at<int>(*c, c->lay.fr_truth);
    f.batch = batch; f.gamma = gamma; f.vocab = c->cfg.large.vocab;
    f.keep = at<int>(*c, c->lay.row_tok); f.row_seq = at<int>(*c, c->lay.row_seq); f.row_pos = at<int>(*c, c->lay.row_pos);
    f.nll = at<float>(*c, c->lay.forced_nll); f.top = at<int>(*c, c->lay.forced_top);
    f.hidden = at<float>(*c, c->lay.h_large); f.d_large = c->cfg.large.d_model;
    f.last_hidden = at<float>(*c, c->lay.proj_snap); f.last_logits = at<float>(*c, c->lay.logits_small);
    int b0 = 0;
    for (f.v0 = 0; f.v0 < rows; f.v0 += f.rows) {
        int end = std::min(rows, f.v0 + c->lay.fr_rows);
        while (p_start[b0 + 1] <= f.v0) ++b0;
        int groups_large = 0, groups_small = 0;
        double kv = 0.0;
        for (int b = b0; b < batch && p_start[b] < end; ++b) {
            const int first = std::max(p_start[b], f.v0);
            if (p_start[b + 1] > end) end -= (end - p_start[b]) % gamma;   // (a block is not cut)
            const int n = std::min(p_start[b + 1], end) - first;
            groups_large += cdiv(n, PASS_GROUP); groups_small += cdiv(n, gamma);
            kv += (double)n / PASS_GROUP * lens[b];
        }
        f.rows = end - f.v0;
        f.grp = f.top + f.v0; f.grp_pos = reinterpret_cast<int*>(f.nll) + f.v0;   // (read before the scores are written)
        forced_pass(*c, f, f.rows == rows, groups_large, groups_small, kv);
    }
    TRY(check_launch(*c));
    // scores and the error word come back behind one wait (the ids have long been copied out of the staging buffer)
    const size_t n = (size_t)(total - batch);
    int32_t* cnt = c->pinned + 2 * n;
    CK(cudaMemcpyAsync(c->pinned, c->arena + c->lay.forced_nll, n * 4, cudaMemcpyDeviceToHost, c->stream));
    CK(cudaMemcpyAsync(c->pinned + n, c->arena + c->lay.forced_top, n * 4, cudaMemcpyDeviceToHost, c->stream));
    CK(cudaMemcpyAsync(cnt, c->st.counters, 8 * 4, cudaMemcpyDeviceToHost, c->stream));
    CK(cudaStreamSynchronize(c->stream));
    if (cnt[2] != 0) {
        snprintf(g_cuda_err, sizeof(g_cuda_err), "device-side wait expired (code %d)", cnt[2]);
        CK(cudaMemsetAsync(c->st.counters + 2, 0, 4, c->stream));
        return TANDEM_ERR_TIMEOUT;
    }
    memcpy(nll, c->pinned, n * 4);
    if (top1) memcpy(top1, c->pinned + n, n * 4);
    return TANDEM_OK;
}

}  // namespace

extern "C" tandem_status tandem_teacher_forced_forward(tandem_ctx* c, int32_t gamma, int32_t batch, const int32_t* ids, const int32_t* lens,
                                                       float* nll, int32_t* top1) {
    TRY(begin_call(c));
    if (!ids || !lens || !nll || batch < 1 || gamma < 1 || gamma > c->cfg.gamma_max) return TANDEM_ERR_INVALID_ARG;
    if (batch > c->cfg.max_batch) return TANDEM_ERR_CAPACITY;
    int max_len = 0;
    long long total = 0;
    for (int b = 0; b < batch; ++b) {
        if (lens[b] < 2) return TANDEM_ERR_INVALID_ARG;
        max_len = std::max(max_len, lens[b]);
        total += lens[b];
    }
    const int pos_cap = std::min(c->cfg.max_seq, std::min(c->cfg.large.max_pos, c->cfg.small.max_pos));
    if ((long long)max_len + gamma > pos_cap) return TANDEM_ERR_CAPACITY;
    for (long long i = 0; i < total; ++i)
        if (ids[i] < 0 || ids[i] >= c->cfg.large.vocab) return TANDEM_ERR_INVALID_ARG;
    if (c->cfg.dtype == TANDEM_DTYPE_BF16) return forced_forward(c, gamma, batch, ids, lens, total, nll, top1);
    // an empty prompt pass: the first token of every sequence is its pending token
    std::vector<int32_t> first((size_t)batch), ones((size_t)batch, 1), padded((size_t)batch * c->cfg.max_seq, 0);
    long long off = 0;
    for (int b = 0; b < batch; ++b) {
        first[b] = ids[off];
        memcpy(padded.data() + (size_t)b * c->cfg.max_seq, ids + off, (size_t)lens[b] * 4);
        off += lens[b];
    }
    TRY(prefill_impl(c, batch, 1, first.data(), ones.data()));
    CK(cudaMemcpyAsync(c->arena + c->lay.forced_ids, padded.data(), padded.size() * 4, cudaMemcpyHostToDevice, c->stream));
    CK(cudaMemcpyAsync(c->arena + c->lay.forced_len, lens, (size_t)batch * 4, cudaMemcpyHostToDevice, c->stream));
    CK(cudaStreamSynchronize(c->stream));   // the host arrays above go out of scope
    std::vector<int32_t> scratch_ids((size_t)batch * (max_len - 1));
    TRY(run_generate(c, true, gamma, max_len - 1, 5, 0ull, scratch_ids.data(), nullptr, nullptr));
    std::vector<float> h_nll((size_t)batch * c->cfg.max_seq);
    std::vector<int32_t> h_top((size_t)batch * c->cfg.max_seq);
    CK(cudaMemcpyAsync(h_nll.data(), c->arena + c->lay.forced_nll, h_nll.size() * 4, cudaMemcpyDeviceToHost, c->stream));
    CK(cudaMemcpyAsync(h_top.data(), c->arena + c->lay.forced_top, h_top.size() * 4, cudaMemcpyDeviceToHost, c->stream));
    CK(cudaStreamSynchronize(c->stream));
    long long o = 0;
    for (int b = 0; b < batch; ++b)
        for (int p = 0; p + 1 < lens[b]; ++p, ++o) {
            nll[o] = h_nll[(size_t)b * c->cfg.max_seq + p];
            if (top1) top1[o] = h_top[(size_t)b * c->cfg.max_seq + p];
        }
    return TANDEM_OK;
}

extern "C" tandem_status tandem_set_sampling(tandem_ctx* c, float temp_large, float temp_small) {
    TRY(begin_call(c));
    if (!(temp_large > 0.f) || !(temp_small > 0.f)) return TANDEM_ERR_INVALID_ARG;
    if (temp_large == c->temp_large && temp_small == c->temp_small) return TANDEM_OK;
    // the temperatures are kernel arguments baked into the captured iterations: drop the sampled ones
    CK(cudaStreamSynchronize(c->stream));
    for (auto& g : c->graphs)
        if (g.mode == TANDEM_ACCEPT_SAMPLE && g.exec) { cudaGraphExecDestroy(g.exec); g.exec = nullptr; }
    c->temp_large = temp_large;
    c->temp_small = temp_small;
    return TANDEM_OK;
}

extern "C" tandem_status tandem_standalone_generate(tandem_ctx* c, int32_t gamma, int32_t variant, int32_t max_new_tokens,
                                                    int32_t* out_ids, int32_t* out_lens, tandem_stats* stats) {
    TRY(begin_call(c));
    if (gamma < 1 || gamma > c->cfg.gamma_max) return TANDEM_ERR_INVALID_ARG;
    switch (variant) {
        case TANDEM_STANDALONE_FREE_TOKEN:
            return run_generate(c, true, gamma, max_new_tokens, TANDEM_ACCEPT_ALL, 0ull, out_ids, out_lens, stats);
        case TANDEM_STANDALONE_REPRESENTATION_ONLY:
            return run_generate(c, true, gamma, max_new_tokens, TANDEM_ACCEPT_REPRESENTATION_ONLY, 0ull, out_ids, out_lens, stats);
        case TANDEM_STANDALONE_FREE_TOKEN_FULL_PROMPT:
            return run_generate(c, true, gamma, max_new_tokens, TANDEM_ACCEPT_ALL, 0ull, out_ids, out_lens, stats, true);
        default: return TANDEM_ERR_INVALID_ARG;
    }
}

extern "C" tandem_status tandem_large_greedy_generate(tandem_ctx* c, int32_t max_new_tokens, int32_t* out_ids, int32_t* out_lens,
                                                      tandem_stats* stats) {
    TRY(begin_call(c));
    return run_generate(c, false, 0, max_new_tokens, 0, 0ull, out_ids, out_lens, stats);
}

extern "C" int64_t tandem_launch_count(tandem_ctx* c) { return c ? c->launches : -1; }

extern "C" const char* tandem_profile_class_name(int32_t cls) {
    static const char* names[PC_COUNT] = {"gemm_smallm", "gemm_tiled", "attn_split", "attn_merge", "attn_prompt",
                                          "layernorm", "rows", "argmax", "verify", "gemm_tc_decode", "gemm_tc_tiled"};
    return (cls >= 0 && cls < PC_COUNT) ? names[cls] : nullptr;
}

extern "C" tandem_status tandem_profile_enable(tandem_ctx* c, int32_t max_launches) {
    TRY(begin_call(c));
    if (max_launches < 0) return TANDEM_ERR_INVALID_ARG;
    CK(cudaStreamSynchronize(c->stream));
    Prof& p = c->prof;
    p.on = max_launches > 0;
    p.used = 0;
    p.cls.clear();
    p.bytes.clear();
    while (p.ev.size() < (size_t)2 * max_launches) {
        cudaEvent_t e;
        CK(cudaEventCreate(&e));
        p.ev.push_back(e);
    }
    return TANDEM_OK;
}

extern "C" tandem_status tandem_profile_read(tandem_ctx* c, int32_t n_classes, double* ms, int64_t* launches, double* work) {
    TRY(begin_call(c));
    if (!ms || !launches || !work || n_classes < 1) return TANDEM_ERR_INVALID_ARG;
    CK(cudaStreamSynchronize(c->stream));
    for (int i = 0; i < n_classes; ++i) { ms[i] = 0; launches[i] = 0; work[i] = 0; }
    Prof& p = c->prof;
    for (size_t i = 0; i + 1 < p.used; i += 2) {
        const int cls = p.cls[i / 2];
        if (cls >= n_classes) continue;
        float t = 0.f;
        CK(cudaEventElapsedTime(&t, p.ev[i], p.ev[i + 1]));
        ms[cls] += t;
        launches[cls] += 1;
        work[cls] += p.bytes[i / 2];
    }
    p.used = 0;
    p.cls.clear();
    p.bytes.clear();
    return TANDEM_OK;
}

extern "C" tandem_status tandem_debug_expire_wait(tandem_ctx* c) {
    TRY(begin_call(c));
    if (c->cfg.dtype != TANDEM_DTYPE_BF16) return TANDEM_ERR_UNIMPLEMENTED;
    // One CTA of the decode GEMM over the first 128 x 64 corner of the large model's first query matrix, with the
    // weight loads withheld and a poll limit of 1024: the MMA thread's wait for operands runs out, the kernel
    // records the code in the context's error word and leaves through its normal tear-down.  The (meaningless)
    // product goes to the debug scratch area.
    TcScratch sc = tc_scratch(*c);
    sc.poll_limit = 1024;
    sc.withhold_weights = 1;
    const int d = c->large.d.d_model;
    TcW w = tcw(*c, wi_layer(c->large, 0, W_WQ), -1, -1, std::min(128, d), 64);
    c->next_launch_plain = true;
    launch_tc_decode<PRO_F32, EPI_STORE_F32>(*c, sc, at<float>(*c, c->lay.h_large), d, nullptr, nullptr, 1, w, false,
                                             epi_plain(at<float>(*c, c->lay.dbg), 128));
    return check_launch(*c);
}

extern "C" tandem_status tandem_debug_read(tandem_ctx* c, int32_t what, int32_t layer, int32_t seq, void* host_dst, size_t bytes) {
    TRY(begin_call(c));
    if (!host_dst) return TANDEM_ERR_INVALID_ARG;
    if (c->batch == 0) return TANDEM_ERR_STATE;
    const int B = c->batch, g = c->last_gamma, V = c->cfg.large.vocab;
    CK(cudaStreamSynchronize(c->stream));
    if (what == 0 || what == 1 || what == 2) {
        size_t n;
        const void* src;
        if (what == 0) { n = (size_t)B * (g + 1) * V; src = c->arena + c->lay.logits_large; }
        else if (what == 1) { n = (size_t)g * B * V; src = c->arena + c->lay.logits_small; }
        else { n = (size_t)B * (g + 1) * c->cfg.large.d_model; src = c->arena + c->hidden_at; }
        if (bytes != n * 4) return TANDEM_ERR_INVALID_ARG;
        if (n) CK(cudaMemcpy(host_dst, src, bytes, cudaMemcpyDeviceToHost));
        return TANDEM_OK;
    }
    if (what >= 3 && what <= 6) {
        const Model& m = (what <= 4) ? c->large : c->small;
        if (layer < 0 || layer >= m.d.n_layers || seq < 0 || seq >= B) return TANDEM_ERR_INVALID_ARG;
        int n_b = 0;
        CK(cudaMemcpy(&n_b, c->st.n + seq, 4, cudaMemcpyDeviceToHost));
        const int n = n_b - 1, H = m.kv_heads, dh = m.d.d_model / m.d.n_heads, d = m.d_kv;
        if (bytes != (size_t)n * d * 4) return TANDEM_ERR_INVALID_ARG;
        if (n == 0) return TANDEM_OK;
        const int which = (what == 3 || what == 5) ? 0 : 1;
        float* dbg = at<float>(*c, c->lay.dbg);
        const size_t total = (size_t)n * d;
        const size_t seq_off = (size_t)seq * H * c->cfg.max_seq * dh;
        if (c->cfg.dtype == TANDEM_DTYPE_BF16)
            gather_kv_kernel<bf16><<<(unsigned)((total + 255) / 256), 256, 0, c->stream>>>(kv_ptr<bf16>(*c, m, layer, which) + seq_off, dbg, n, H, dh, c->cfg.max_seq);
        else
            gather_kv_kernel<float><<<(unsigned)((total + 255) / 256), 256, 0, c->stream>>>(kv_ptr<float>(*c, m, layer, which) + seq_off, dbg, n, H, dh, c->cfg.max_seq);
        TRY(check_launch());
        CK(cudaMemcpyAsync(host_dst, dbg, bytes, cudaMemcpyDeviceToHost, c->stream));
        CK(cudaStreamSynchronize(c->stream));
        return TANDEM_OK;
    }
    if (what == 7) {
        if (bytes != (size_t)B * 4) return TANDEM_ERR_INVALID_ARG;
        CK(cudaMemcpy(host_dst, c->st.n, bytes, cudaMemcpyDeviceToHost));
        return TANDEM_OK;
    }
    return TANDEM_ERR_INVALID_ARG;
}

// ---------------------------------------------------------------------------------------------------
// stand-alone kernels
// ---------------------------------------------------------------------------------------------------

// Stand-alone calls: two launches of one call, or of consecutive calls on a stream, are chained by programmatic dependent
// launch, so that a kernel's set-up runs under its predecessor's end; the first kernel of a call reads nothing before its
// predecessor has finished (the caller's kernels may be writing the inputs).  Only the stream, the launch counter and
// the launch options of the context are used by the launch helpers.
namespace {
struct StandaloneCtx : tandem_ctx {
    explicit StandaloneCtx(void* s) {
        stream = static_cast<cudaStream_t>(s);
        n_sms = sm_count();
    }
};
// Work space that the attention entry points ask their callers for: two ints per sequence, kept in the contract (the
// kernel takes a sequence's number and position from its arguments now, which spared a kernel launch per call).
size_t attn_scratch_size(int batch) { return align_up((size_t)batch * 2 * 4); }
}  // namespace

extern "C" size_t tandem_decode_attention_scratch_bytes(int32_t batch, int32_t n_heads, int32_t d_head, int32_t derived_len, int32_t own_len) {
    if (batch < 1 || n_heads < 1 || d_head < 1 || derived_len < 0 || own_len < 0 || derived_len + own_len < 1) return 0;
    return attn_scratch_size(batch);
}

extern "C" tandem_status tandem_decode_attention(const void* q, const void* k_derived, const void* v_derived, const void* k_own,
                                                 const void* v_own, void* out, void* scratch, size_t scratch_bytes, int32_t batch,
                                                 int32_t n_heads, int32_t d_head, int32_t derived_len, int32_t own_len, void* stream) {
    if (!q || !out || !scratch) return TANDEM_ERR_INVALID_ARG;
    if (batch < 1 || n_heads < 1 || derived_len < 0 || own_len < 0 || derived_len + own_len < 1) return TANDEM_ERR_INVALID_ARG;
    if ((derived_len > 0 && (!k_derived || !v_derived)) || (own_len > 0 && (!k_own || !v_own))) return TANDEM_ERR_INVALID_ARG;
    if (d_head != 32 && d_head != 64 && d_head != 128) return TANDEM_ERR_SHAPE;
    if ((long long)batch * n_heads > 65535 * 16) return TANDEM_ERR_SHAPE;
    if (((uintptr_t)q | (uintptr_t)k_derived | (uintptr_t)v_derived | (uintptr_t)k_own | (uintptr_t)v_own | (uintptr_t)out | (uintptr_t)scratch) & 15)
        return TANDEM_ERR_INVALID_ARG;
    if (scratch_bytes < attn_scratch_size(batch)) return TANDEM_ERR_ARENA_TOO_SMALL;
    if (batch > 65535) return TANDEM_ERR_SHAPE;
    AttnArgs a; memset(&a, 0, sizeof(a));
    a.q = q; a.ldq = n_heads * d_head; a.kcache = k_derived; a.vcache = v_derived; a.k2 = k_own; a.v2 = v_own;
    a.split = derived_len; a.t_max = derived_len; a.t_max2 = own_len;
    a.out = out; a.ldo = n_heads * d_head; a.pos_all = derived_len + own_len - 1; a.wait_first = 1; a.nq = 1; a.n_heads = n_heads;
    a.scale = 1.0f / sqrtf((float)d_head);
    StandaloneCtx tmp(stream);
    launch_attn_decode(tmp, d_head, a, batch, 0.0);
    return check_launch();
}

// ---------------------------------------------------------------------------------------------------
// Decode attention for callers that cannot allocate device memory
// ---------------------------------------------------------------------------------------------------

extern "C" tandem_status tandem_decode_attention_static(const void* q, const void* k_derived, const void* v_derived,
                                                        const void* k_own, const void* v_own, void* out, int32_t batch,
                                                        int32_t n_heads, int32_t d_head, int32_t derived_len, int32_t own_len,
                                                        void* stream) {
    if (batch < 1 || n_heads < 1 || d_head < 1 || derived_len < 0 || own_len < 0 || derived_len + own_len < 1)
        return TANDEM_ERR_INVALID_ARG;
    const size_t need = attn_scratch_size(batch);
    if (need > (size_t)TANDEM_STATIC_SCRATCH_BYTES) {
        snprintf(g_cuda_err, sizeof(g_cuda_err),
                 "tandem_decode_attention_static: this batch needs %zu bytes of work space, the built-in buffer holds %d; "
                 "use tandem_decode_attention with your own scratch", need, TANDEM_STATIC_SCRATCH_BYTES);
        return TANDEM_ERR_CAPACITY;
    }
    // the kernel reads and writes no work space; the call below only wants a non-null, aligned argument
    return tandem_decode_attention(q, k_derived, v_derived, k_own, v_own, out, out, (size_t)TANDEM_STATIC_SCRATCH_BYTES, batch,
                                   n_heads, d_head, derived_len, own_len, stream);
}

// ---------------------------------------------------------------------------------------------------
// Stand-alone GEMM entry points: their bounded waits report into one word per device
// ---------------------------------------------------------------------------------------------------

static __device__ int g_standalone_err;

namespace {
int* g_standalone_err_addr[MAX_DEVICES] = {};
std::mutex g_standalone_err_mutex;

// Device address of the current device's error word (looked up once per device); null if the lookup fails, in
// which case the kernels run without reporting.
int* standalone_err_word() {
    const int dev = cur_dev();
    std::lock_guard<std::mutex> lock(g_standalone_err_mutex);
    if (!g_standalone_err_addr[dev]) {
        void* p = nullptr;
        if (cudaGetSymbolAddress(&p, g_standalone_err) == cudaSuccess) g_standalone_err_addr[dev] = static_cast<int*>(p);
    }
    return g_standalone_err_addr[dev];
}

struct ProjScratch { size_t yhat, a_s, total; };
ProjScratch proj_scratch_layout(int rows, int d_small) {
    ProjScratch p;
    size_t off = 0;
    p.yhat = off; off = align_up(off + (size_t)rows * d_small * 4);
    p.a_s = off; off = align_up(off + (size_t)rows * d_small * 4);
    p.total = off;
    return p;
}
}  // namespace

extern "C" tandem_status tandem_standalone_check(void* stream) {
    int* word = standalone_err_word();
    if (!word) return TANDEM_ERR_CUDA;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    int code = 0;
    CK(cudaMemcpyAsync(&code, word, sizeof(int), cudaMemcpyDeviceToHost, s));
    CK(cudaStreamSynchronize(s));
    if (code == 0) return TANDEM_OK;
    snprintf(g_cuda_err, sizeof(g_cuda_err), "device-side wait expired (code %d)", code);
    CK(cudaMemsetAsync(word, 0, sizeof(int), s));
    return TANDEM_ERR_TIMEOUT;
}

extern "C" size_t tandem_ff_tandem_project_scratch_bytes(int32_t rows, int32_t d_small) {
    if (rows < 1 || rows > 256 || d_small < 8) return 0;
    return proj_scratch_layout(rows, d_small).total;
}

extern "C" tandem_status tandem_ff_tandem_project(const void* x, const void* w_t, const void* ln_g, const void* ln_b, const void* wk,
                                                  const void* wv, void* k_out, void* v_out, void* scratch, size_t scratch_bytes,
                                                  int32_t rows, int32_t d_large, int32_t d_small, void* stream) {
    if (!x || !w_t || !ln_g || !ln_b || !wk || !wv || !k_out || !v_out || !scratch) return TANDEM_ERR_INVALID_ARG;
    if (rows < 1 || rows > 256 || d_large < 8 || d_small < 8) return TANDEM_ERR_INVALID_ARG;
    if (d_large % 8 || d_small % 8) return TANDEM_ERR_SHAPE;
    const ProjScratch pl = proj_scratch_layout(rows, d_small);
    if (scratch_bytes < pl.total) return TANDEM_ERR_ARENA_TOO_SMALL;
    if (((uintptr_t)x | (uintptr_t)w_t | (uintptr_t)wk | (uintptr_t)wv | (uintptr_t)k_out | (uintptr_t)v_out | (uintptr_t)scratch |
         (uintptr_t)ln_g | (uintptr_t)ln_b) & 15)
        return TANDEM_ERR_INVALID_ARG;
    StandaloneCtx tmp(stream);
    unsigned char* sc = static_cast<unsigned char*>(scratch);
    float* yhat = reinterpret_cast<float*>(sc + pl.yhat);
    float* a_s = reinterpret_cast<float*>(sc + pl.a_s);
    TcW wt, wkv;
    if (!cached_tmap_bf16(&wt.tm[0], w_t, (uint64_t)d_small, (uint64_t)d_large) || !cached_tmap_bf16(&wkv.tm[0], wk, (uint64_t)d_small, (uint64_t)d_small) ||
        !cached_tmap_bf16(&wkv.tm[1], wv, (uint64_t)d_small, (uint64_t)d_small)) {
        snprintf(g_cuda_err, sizeof(g_cuda_err), "cuTensorMapEncodeTiled unavailable or failed");
        return TANDEM_ERR_CUDA;
    }
    wt.tm[1] = wt.tm[2] = wt.tm[0]; wt.n_segs = 1; wt.seg_rows0 = wt.seg_rows = d_small; wt.K = d_large;
    wkv.tm[2] = wkv.tm[0]; wkv.n_segs = 2; wkv.seg_rows0 = wkv.seg_rows = d_small; wkv.K = d_small;
    EpiArgs e; memset(&e, 0, sizeof(e));
    e.kcache = k_out; e.vcache = v_out; e.n_heads = 1; e.d_head = d_small; e.t_max = 1; e.seg0 = e.seg = d_small;
    // weights streamed once per GEMM and group of 64 rows; for a few short rows the LayerNorm is fused into the
    // second GEMM's operand load
    TcScratch ts; ts.err = standalone_err_word();
    ts.wait_first = 1;
    launch_tc_decode<PRO_BF16, EPI_STORE_F32>(tmp, ts, x, d_large, nullptr, nullptr, rows, wt, true, epi_plain(yhat, d_small));
    ts.wait_first = 0;   // the kernels behind it start once everything older than the first GEMM has finished: the weights are final
    if (rows <= 8 && d_small <= 1024) {
        launch_tc_decode<PRO_LN, EPI_KV>(tmp, ts, yhat, d_small, ln_g, ln_b, rows, wkv, true, e);
    } else {
        launch_layernorm<float>(tmp, rows, yhat, ln_g, ln_b, a_s, d_small);
        launch_tc_decode<PRO_F32, EPI_KV>(tmp, ts, a_s, d_small, nullptr, nullptr, rows, wkv, true, e);
    }
    return check_launch();
}

extern "C" tandem_status tandem_block_linear(const void* x, const void* w, void* y, int32_t rows, int32_t in_features,
                                             int32_t out_features, void* stream) {
    if (!x || !w || !y) return TANDEM_ERR_INVALID_ARG;
    if (rows < 1 || rows > 64 || in_features < 8 || out_features < 1) return TANDEM_ERR_INVALID_ARG;
    if (in_features % 8) return TANDEM_ERR_SHAPE;
    if (((uintptr_t)x | (uintptr_t)w | (uintptr_t)y) & 15) return TANDEM_ERR_INVALID_ARG;
    StandaloneCtx tmp(stream);
    TcW tw;
    if (!cached_tmap_bf16(&tw.tm[0], w, (uint64_t)out_features, (uint64_t)in_features)) {
        snprintf(g_cuda_err, sizeof(g_cuda_err), "cuTensorMapEncodeTiled unavailable or failed");
        return TANDEM_ERR_CUDA;
    }
    tw.tm[1] = tw.tm[2] = tw.tm[0]; tw.n_segs = 1; tw.seg_rows0 = tw.seg_rows = out_features; tw.K = in_features;
    TcScratch ts; ts.err = standalone_err_word();
    ts.wait_first = 1;
    launch_tc_decode<PRO_BF16, EPI_STORE>(tmp, ts, x, in_features, nullptr, nullptr, rows, tw, true, epi_plain(y, out_features));
    return check_launch();
}
