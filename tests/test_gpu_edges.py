"""Edges of the kernels' dispatch rules and tiles, each against the fp64 checker."""
import os
import subprocess
import sys

import numpy as np
import pytest

from oracle import tandem_oracle as O
from paper_2402_08644_b200 import binding, build, synth
from test_gpu_parity import TOL_BF16, TOL_FP32, _adaptive_replay, _bf16_weights, _replay_compare, _sampled_replay, gpu_toy_shape, prompts_for, toy_weights

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    return binding.load_library()


@pytest.mark.parametrize("lens,gamma", [([65], 3),                    # 64 prompt rows on the few-row kernel; 4 block rows
                                        ([66, 126, 127, 2], 1),       # tiled prompt kernel; contexts that reach a chunk's end; 8 rows
                                        ([1, 128, 129], 2)])          # 9 rows: two groups of the 8-row kernel
def test_fp32_few_row_kernels_at_their_edges(lens, gamma):
    """Rows longer than the fused LayerNorm and one staging pass take (2080, 2400 > 2048), more columns than one per warp
    covers (2400 > 2368), one to nine rows, and attention over one chunk, exactly one, and two."""
    shape = gpu_toy_shape(large=(1, 2080, 65, 2400), small=(1, 64, 1, 136), max_pos=160, layer_map=(1,))
    w = toy_weights(shape, seed=3, std=0.02)
    assert _replay_compare(shape, w, prompts_for(shape, lens, seed=4), gamma, 3, TOL_FP32, 1e-6, check_kv=True) == 0


@pytest.mark.parametrize("width", [256, 288, 512, 544])   # LayerNorm in registers up to 256 elements with four columns per warp (the heads), 512 with one
@pytest.mark.parametrize("lens,gamma", [([6], 0), ([6], 3), ([5, 9, 3], 2)])   # one row, four, nine (eight and one)
def test_fp32_few_row_kernel_forms(width, lens, gamma):
    """Rows at and behind the lengths up to which a warp normalises them in its registers, in every row count's form."""
    shape = gpu_toy_shape(large=(1, width, width // 32, 264), small=(1, width, width // 32, 136), vocab=2400, max_pos=64, layer_map=(1,))
    w = toy_weights(shape, seed=5, std=0.03)
    assert _replay_compare(shape, w, prompts_for(shape, lens, seed=6), gamma, 3, TOL_FP32, 1e-6, check_kv=True) == 0


@pytest.mark.parametrize("lens", [[129],            # one row tile: K dealt to four CTAs (17 K-blocks: 4, 4, 4, 5)
                                  [130, 2, 1],      # two row tiles, the second of two rows; a prompt without processed rows
                                  [900, 385]])      # ten: two CTAs per tile, or one
def test_bf16_split_k_prompt_gemm_at_its_edges(lens):
    """Square tiles with one, two and four CTAs per tile: ragged last row tile and feature tile (1088 = 8.5 x 128, 1160),
    K-blocks that do not divide evenly, grouped-query key / value segments of half a tile, both head sizes' attention tiles
    (128 and 256 queries) with one row in the last one."""
    shape = gpu_toy_shape(dtype=synth.DTYPE_BF16, large=(2, 1088, 17, 1160), small=(1, 128, 2, 256), max_pos=960, layer_map=(1,), kv_heads=(1, 0))
    w = _bf16_weights(shape, seed=9, std=0.02)
    assert _replay_compare(shape, w, prompts_for(shape, lens, seed=5), 2, 2, TOL_BF16, 2 * TOL_BF16, check_kv=True) <= 4


@pytest.mark.parametrize("batch,gamma,offset", [(1, 0, 0.0), (3, 4, 0.5), (4, 3, 0.0), (1, 15, 0.5),      # 1, 15, 16 and 16 block rows
                                                (3, 5, 0.0), (11, 2, 0.5), (7, 6, 0.0), (4, 15, 0.0)])     # 18, 33, 49 and 64
def test_bf16_layernorm_behind_the_product(batch, gamma, offset):
    """LayerNorm applied in the epilogue of the map behind it, at every token-column width, one to sixteen rows per warp of
    statistics, row lengths that end inside a K-block (96, 160), and rows whose mean is several times their deviation."""
    shape = gpu_toy_shape(dtype=synth.DTYPE_BF16, large=(2, 160, 5, 288), small=(2, 96, 3, 136), max_pos=64, layer_map=(0, 2))
    w = _bf16_weights(shape, seed=gamma + 3, std=0.05)
    for tag in "LS":
        w[tag + ".pos"] = synth.round_to_bf16(w[tag + ".pos"] + offset)
    prompts = prompts_for(shape, [1 + 3 * (b % 5) for b in range(batch)], seed=batch)
    assert _replay_compare(shape, w, prompts, gamma, 2, TOL_BF16, 2 * TOL_BF16) <= 10


@pytest.mark.parametrize("vocab", [31, 2049, 32768, 32801])
def test_sampling_and_router_over_a_cluster(vocab):
    """Rows of logits dealt to eight CTAs: fewer logits than ranges, a ragged last range, the longest row that stays in registers
    and one that does not; draws, accept decisions, router features and block lengths against the checker."""
    shape = gpu_toy_shape(large=(1, 64, 2, 64), small=(1, 32, 1, 64), vocab=vocab, max_pos=48, layer_map=(1,))
    w = toy_weights(shape, seed=2, std=0.3)
    prompts = prompts_for(shape, [5, 9], seed=1)
    _sampled_replay(shape, w, prompts, 3, 3, 0.7, 0.9, seed=11, tol=TOL_FP32, eps=2e-5)
    _adaptive_replay(shape, w, prompts, 4, 3, TOL_FP32, 1e-4)


def test_bf16_pair_prompt_gemm_with_tiles_in_parts():
    """256 x 256 tiles on pairs of multiprocessors: 2104 rows are nine row tiles, the last with 56 rows (none for the second CTA);
    the tiles beyond the last full round of 74 pairs are cut into four parts (9 feature tiles: 81), two (27: 243) and left
    whole (12.5: 117, ragged features too)."""
    shape = gpu_toy_shape(dtype=synth.DTYPE_BF16, large=(1, 2304, 18, 3200), small=(1, 128, 2, 256), max_pos=2120, layer_map=(1,))
    w = _bf16_weights(shape, seed=6, std=0.02)
    assert _replay_compare(shape, w, prompts_for(shape, [2105], seed=7), 1, 1, TOL_BF16, 2 * TOL_BF16, check_kv=True) <= 1


@pytest.mark.parametrize("lens", [[300], [641, 60], [1100, 31], [1900]])
def test_bf16_prompt_gemm_between_the_two_kernels(lens):
    """Prompts of a few hundred rows, where the choice between slices of K and pairs of multiprocessors changes from map to map: pairs
    with fewer tiles than there are, tiles in four, two and one part, key / value segments of 128 features in tiles of 256, ragged
    row and feature tiles."""
    shape = gpu_toy_shape(dtype=synth.DTYPE_BF16, large=(2, 2176, 17, 2312), small=(1, 128, 2, 256), max_pos=1920, layer_map=(1,), kv_heads=(1, 0))
    w = _bf16_weights(shape, seed=19, std=0.015)
    assert _replay_compare(shape, w, prompts_for(shape, lens, seed=20), 1, 1, TOL_BF16, 2 * TOL_BF16, check_kv=True) <= 2


@pytest.mark.parametrize("width,heads,lens", [(992, 31, [258]), (1024, 16, [257]), (1056, 33, [250, 9]), (2048, 32, [262]), (2080, 65, [259])])
def test_bf16_prompt_layernorm_by_warps_and_blocks(width, heads, lens):
    """Around the rules that give a row of a prompt pass a warp (more than 256 rows, up to 1024 and 2048 elements) or a
    block: 256 to 261 rows, lanes without a last float4, and the copy of the rows that a projection reads."""
    shape = gpu_toy_shape(dtype=synth.DTYPE_BF16, large=(1, width, heads, 64), small=(1, 64, 1, 64), max_pos=288, layer_map=(0,))
    w = _bf16_weights(shape, seed=27, std=0.02)
    assert _replay_compare(shape, w, prompts_for(shape, lens, seed=28), 1, 1, TOL_BF16, 2 * TOL_BF16, check_kv=True) <= 2


@pytest.mark.parametrize("heads", [2, 1])   # head sizes 64 and 128: chunks of 64 and of 128 keys
def test_bf16_prompt_attention_at_chunk_edges(heads):
    """Prompts that end one query before, at and behind the end of a chunk and a tile, in one batch.  (So few heads: one tile of
    queries per CTA.)"""
    shape = gpu_toy_shape(dtype=synth.DTYPE_BF16, large=(1, 128, heads, 128), small=(1, 64, 1, 64), max_pos=640, layer_map=(1,))
    w = _bf16_weights(shape, seed=12, std=0.1)
    prompts = prompts_for(shape, [64, 65, 66, 128, 129, 130, 256, 257, 258, 386, 514], seed=13)
    assert _replay_compare(shape, w, prompts, 1, 1, TOL_BF16, 2 * TOL_BF16, check_kv=True) <= 4


@pytest.mark.parametrize("width", [384, 768])   # six heads of 64 and of 128
def test_bf16_prompt_attention_in_groups_of_two_tiles(width):
    """The same ends with heads enough that a CTA takes two tiles: a second tile of one query, one that ends at and behind a chunk, a
    group that ends at 256 and 257 queries."""
    lens, heads = [64, 65, 66, 128, 129, 130, 256, 257, 258, 386, 514], 6
    assert ((sum(lens) - len(lens)) // 256 + len(lens)) * heads * 2 > 148    # two tiles of queries per CTA on 148 multiprocessors
    shape = gpu_toy_shape(dtype=synth.DTYPE_BF16, large=(1, width, heads, 128), small=(1, 64, 1, 64), max_pos=640, layer_map=(1,))
    # what bf16 keys, values and activations cost grows with the logits' spread, std * sqrt(width): 2.2e-2 at 1.39, so 0.8 stays below 1.3e-2
    w = _bf16_weights(shape, seed=12, std=0.8 / width ** 0.5)
    assert _replay_compare(shape, w, prompts_for(shape, lens, seed=13), 1, 1, TOL_BF16, 2 * TOL_BF16, check_kv=True) <= 4


@pytest.mark.parametrize("width,ffn", [(512, 1160), (576, 1288), (1088, 2184)])   # 8, 9 and 17 K-blocks; 9 / 10, 11 and 18 feature tiles
def test_bf16_few_row_gemm_with_four_and_eight_slices(width, ffn):
    """Around the rule that gives wide matrices of short rows four K-slices instead of eight, ragged last tiles and slices."""
    shape = gpu_toy_shape(dtype=synth.DTYPE_BF16, large=(1, width, width // 64, ffn), small=(1, 64, 1, 64), max_pos=64, layer_map=(1,))
    w = _bf16_weights(shape, seed=14, std=0.03)
    assert _replay_compare(shape, w, prompts_for(shape, [5, 9, 2], seed=15), 3, 2, TOL_BF16, 2 * TOL_BF16) <= 4


@pytest.mark.parametrize("vocab", [31, 2049, 32801])
def test_teacher_forced_scores_over_a_cluster(vocab):
    """Rows of logits dealt to 64 warps: fewer logits than ranges, a ragged last range, and rows too long for registers."""
    shape = gpu_toy_shape(large=(1, 64, 2, 64), small=(1, 32, 1, 64), vocab=vocab, max_pos=48, layer_map=(1,))
    w = toy_weights(shape, seed=5, std=0.3)
    seqs = prompts_for(shape, [2, 11, 6], seed=6)
    t = binding.Tandem(shape, w, max_batch=3, max_seq=48, gamma_max=4)
    nll, top = t.tandem_teacher_forced_forward(seqs, 4)
    for b, ids in enumerate(seqs):
        want_nll, want_top = O.next_token_scores(O.teacher_forced_tandem_logits(shape, w, ids, 4), ids)
        assert abs(nll[b] - want_nll).max() < 2 * TOL_FP32
        assert top[b].tolist() == list(want_top)
    t.close()


@pytest.mark.parametrize("batch,heads,dh,derived,own", [(160, 2, 64, 130, 3), (301, 1, 128, 127, 1), (300, 2, 32, 0, 1)])
def test_decode_attention_by_lone_ctas(batch, heads, dh, derived, own):
    """More (sequence, head) pairs than clusters would fit: one CTA for each, whose result leaves with the fold of its warps' states
    (contexts of one and two chunks, and of one key)."""
    import torch
    g = torch.Generator().manual_seed(batch)
    mk = lambda *s: torch.randn(*s, generator=g).to(torch.bfloat16)
    q, kd, vd, ko, vo = mk(batch, heads, dh), mk(batch, heads, derived, dh), mk(batch, heads, derived, dh), mk(batch, heads, own, dh), mk(batch, heads, own, dh)
    out = binding.tandem_decode_attention(*(x.cuda() for x in (q, kd, vd, ko, vo))).double().cpu()
    K, V = torch.cat([kd, ko], 2).double(), torch.cat([vd, vo], 2).double()
    want = (torch.softmax((K @ q.double()[..., None])[..., 0] / dh ** 0.5, -1)[..., None, :] @ V)[..., 0, :]
    assert (out - want).abs().max() < TOL_BF16


@pytest.mark.parametrize("lens,gamma,prefill_rows,kw", [
    ([2, 140, 23], 4, 0, dict(layer_map=(1, 3), vocab=129)),                     # one pass of 162 rows, last blocks of one to three; a head tile of one feature
    ([131, 7, 66], 3, 20, dict(layer_map=(0, 2))),                               # passes of at most 20 rows, whole blocks: a sequence over many of them
    ([190, 180], 4, 0, dict(large=(2, 128, 2, 2048), layer_map=(0, 2), max_pos=200)),   # a work space that holds fewer rows than a prompt pass's
    ([130], 4, 130, dict(layer_map=(0, 2))),                                     # so few rows that the projections' results lie apart from the GELU outputs
    ([128], 5, 130, dict(kind=synth.FF_TANDEM_MLP, hidden=40, layer_map=(1, 1))),   # ... and two small layers read the same representations
    ([47], 15, 0, dict(large=(2, 256, 2, 264), small=(1, 256, 2, 136), kv_heads=(1, 1), layer_map=(2,))),   # blocks of 15, 128-wide heads, shared keys / values
    ([66, 2], 1, 0, dict(kind=synth.FF_TANDEM_MLP, hidden=40, layer_map=(0, 3), small=(2, 192, 6, 136))),  # 66 blocks of one row; a small model wider than the large one
    ([141], 1, 0, dict(layer_map=(0, 3), small=(2, 192, 6, 136))),               # 840 block heads: two warps share the keys of each (four up to 592)
    ([130, 70], 1, 0, dict(layer_map=(0, 3), small=(2, 192, 6, 136)))])          # 1188: one warp each (two up to 1184)
def test_bf16_teacher_forced_pass(lens, gamma, prefill_rows, kw):
    """All blocks of a teacher-forced forward in one pass or a few: ragged sequences, short last blocks, groups of eight rows of the large
    model, blocks that attend large-derived keys up to their start and their own from there."""
    shape = gpu_toy_shape(**{**dict(dtype=synth.DTYPE_BF16, max_pos=200), **kw})
    w = _bf16_weights(shape, seed=23, std=0.06)
    seqs = prompts_for(shape, lens, seed=24)
    t = binding.Tandem(shape, w, max_batch=len(lens), max_seq=200, gamma_max=gamma, max_prefill_rows=prefill_rows)
    for _ in range(2):   # (the second call finds the first one's keys and values in the caches)
        nll, top = t.tandem_teacher_forced_forward(seqs, gamma)
        differ = 0
        for b, ids in enumerate(seqs):
            logits = O.teacher_forced_tandem_logits(shape, w, ids, gamma)
            want_nll, want_top = O.next_token_scores(logits, ids)
            assert nll[b].shape == (len(ids) - 1,)
            assert np.abs(nll[b] - want_nll).max() < 2 * TOL_BF16
            for i in np.nonzero(top[b] != want_top)[0]:
                assert np.max(logits[i]) - logits[i][top[b][i]] < 2 * TOL_BF16
            differ += int((top[b] != want_top).sum())
        assert differ <= 4
    t.close()


@pytest.mark.parametrize("lens,gamma,prefill_rows,vocab", [([141, 23, 6], 4, 0, 129), ([33, 47], 5, 12, 50)])   # one pass; several
def test_bf16_logits_and_representations_of_the_last_blocks(lens, gamma, prefill_rows, vocab):
    """What a teacher-forced forward leaves to read: the small model's logits and the large model's representations of every
    sequence's last block, not those of the steps before the call."""
    shape = gpu_toy_shape(dtype=synth.DTYPE_BF16, max_pos=200, layer_map=(1, 3), vocab=vocab)
    w = _bf16_weights(shape, seed=31, std=0.06)
    seqs = prompts_for(shape, lens, seed=32)
    t = binding.Tandem(shape, w, max_batch=len(lens), max_seq=200, gamma_max=gamma, max_prefill_rows=prefill_rows)
    t.tandem_prefill([s[:3] for s in seqs])
    t.tandem_block_step(gamma)
    t.tandem_teacher_forced_forward(seqs, gamma)
    logits = t.tandem_debug_read(binding.READ_SMALL_LOGITS, gamma)
    hidden = t.tandem_debug_read(binding.READ_LARGE_HIDDEN, gamma).reshape(-1, shape.large.d_model)
    assert t.tandem_debug_read(binding.READ_COMMITTED).tolist() == lens
    for b, ids in enumerate(seqs):
        o = O.TandemOracle(shape, w)
        reps, _ = O.large_block_pass(o.large, o.large_cache, ids, 0)
        want = O.teacher_forced_tandem_logits(shape, w, ids, gamma)
        first = (len(ids) - 2) // gamma * gamma
        for p in range(first, len(ids) - 1):
            assert np.abs(logits[p - first, b] - want[p]).max() < TOL_BF16
            assert np.abs(hidden[b * gamma + p - first] - reps[-1][p]).max() < 2 * TOL_BF16
        keys = t.tandem_debug_read(binding.READ_LARGE_K, layer=1, seq=b)
        want = np.stack(o.large_cache.k[1][:len(ids) - 1]).reshape(len(ids) - 1, -1)
        assert (np.abs(keys - want) < 2 * TOL_BF16 * np.maximum(1, np.abs(want))).all()
        past = (len(ids) - 2) % gamma + 1
        assert not logits[past:, b].any() and not hidden[b * gamma + past:(b + 1) * gamma].any()
    t.tandem_prefill([s[:3] for s in seqs])       # and a decode iteration's own again
    res = t.tandem_block_step(gamma)
    hidden = t.tandem_debug_read(binding.READ_LARGE_HIDDEN, gamma)
    for b, ids in enumerate(seqs):
        o = O.TandemOracle(shape, w)
        o.prefill(ids[:3])
        _, _, reps = o.verify(res["drafts"][b].tolist())
        assert np.abs(hidden[b] - np.stack(reps[-1])).max() < 2 * TOL_BF16
    t.close()


@pytest.mark.parametrize("kw", [dict(layer_map=(1, 3)), dict(kind=synth.FF_TANDEM_MLP, hidden=40, layer_map=(0, 3))])
def test_bf16_teacher_forced_pass_beyond_the_forked_rows(kw):
    """2100 rows in one pass: the projections stay in the large model's stream, before the queries and GELU outputs that share
    their place, and the output head runs in three parts.  First, middle and last sequence against the checker."""
    shape = gpu_toy_shape(dtype=synth.DTYPE_BF16, max_pos=200, **kw)
    w = _bf16_weights(shape, seed=26, std=0.06)
    seqs = prompts_for(shape, [141] * 15, seed=25)
    t = binding.Tandem(shape, w, max_batch=15, max_seq=200, gamma_max=14)
    nll, top = t.tandem_teacher_forced_forward(seqs, 14)
    differ = 0
    for b in (0, 7, 14):
        logits = O.teacher_forced_tandem_logits(shape, w, seqs[b], 14)
        want_nll, want_top = O.next_token_scores(logits, seqs[b])
        assert np.abs(nll[b] - want_nll).max() < 2 * TOL_BF16
        for i in np.nonzero(top[b] != want_top)[0]:
            assert np.max(logits[i]) - logits[i][top[b][i]] < 2 * TOL_BF16
        differ += int((top[b] != want_top).sum())
    assert differ <= 4
    parts = t.tandem_teacher_forced_forward(seqs[:8], 14)[0] + t.tandem_teacher_forced_forward(seqs[8:], 14)[0]
    for got, want in zip(nll, parts):
        assert np.abs(got - want).max() < 2 * TOL_BF16
    t.close()


_CAPTURES = """
import sys
sys.path[:0] = [{root!r}, {root!r} + "/tests"]
import torch
from paper_2402_08644_b200 import binding, synth
from test_gpu_parity import _bf16_weights, gpu_toy_shape, prompts_for
shape = gpu_toy_shape(dtype=synth.DTYPE_BF16)
t = binding.Tandem(shape, _bf16_weights(shape, seed=1, std=0.05), max_batch=1, max_seq=128, gamma_max=4)
t.tandem_set_router(synth.make_router(shape, 2, 8, 1), 0.0)    # tau 0: every block has four drafts
def respond(new):
    t.tandem_prefill(prompts_for(shape, [7], seed=3))
    return t.tandem_adaptive_generate(4, new)[0].tolist()
respond(24)
with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CPU, torch.profiler.ProfilerActivity.CUDA]) as p:
    got = respond(31)
    torch.cuda.synchronize()
names = [e.name for e in p.events()]
print(names.count("cudaStreamBeginCapture"), sum("GraphLaunch" in n for n in names), got == respond(31))
"""


def test_bf16_adaptive_response_of_another_length_finds_its_graphs():
    """The draft steps do not depend on the number of tokens asked for: a longer response captures the verify half (whose kernel
    does) and none of the four steps again."""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    out = subprocess.run([sys.executable, "-c", _CAPTURES.format(root=root)], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stderr[-2000:]
    captures, launches, same = out.stdout.split()[-3:]
    assert same == "True" and int(launches) >= 8
    assert int(captures) <= 1


def test_bf16_layernorm_parameters_changed_between_calls():
    """Gains and biases that the caller changes after the prompt pass, and again between two steps, hold from the next call on, in
    every map behind a LayerNorm and in the projection."""
    shape = gpu_toy_shape(dtype=synth.DTYPE_BF16, large=(2, 128, 2, 256), small=(2, 64, 1, 136), max_pos=64, layer_map=(0, 2))
    w = _bf16_weights(shape, seed=17, std=0.08)
    prompt, gamma = prompts_for(shape, [9], seed=18)[0], 3
    t = binding.Tandem(shape, w, max_batch=1, max_seq=64, gamma_max=gamma)
    t.tandem_prefill([prompt])
    o = O.TandemOracle(shape, w)
    o.prefill(prompt)
    for factor, shift in ((1.5, 0.25), (0.5, -0.5)):
        w = {k: (v * factor + shift).astype("float32") if synth.is_norm_param(k) else v for k, v in w.items()}
        for name, v in binding.upload_weights(shape, w, t.device).items():
            if synth.is_norm_param(name):
                t.weights[name].copy_(v)
        o.large = O.Decoder(w, "L", shape.large.n_layers, shape.large.n_heads)
        o.small = O.Decoder(w, "S", shape.small.n_layers, shape.small.n_heads)
        res = t.tandem_block_step(gamma)
        drafts, targets = res["drafts"][0].tolist(), res["targets"][0].tolist()
        _, sl = o.draft(gamma, forced=drafts)
        _, ll, reps = o.verify(drafts)
        assert abs(t.tandem_debug_read(binding.READ_SMALL_LOGITS, gamma)[:, 0] - sl).max() < TOL_BF16
        assert abs(t.tandem_debug_read(binding.READ_LARGE_LOGITS, gamma)[0] - ll).max() < TOL_BF16
        o.commit(int(res["accept_len"][0]), drafts, targets, reps)
    t.close()


@pytest.mark.parametrize("batch,gamma", [(1, 3), (7, 15)])     # 4 block rows, and 112: two groups of 64
@pytest.mark.parametrize("offset", [0.0, 40.0])
def test_bf16_layernorm_of_rows_far_from_zero(batch, gamma, offset):
    """Rows whose mean is 200 times their deviation lose nothing to the 16 bits of the planes.  The layers add zero (output and second
    FFN maps of zeros), so the heads see LayerNorm(Emb + Pos) itself: embedded rows beyond and within one block's registers,
    and rows that every residual add has written anew.  Entries are multiples of 2^-8: all sums of x are exact.
    Bound: each term of a logit carries its operand's 16 bits (at most 2^-16 of the term; independent roundings, four deviations are
    less than 4 / sqrt(3) of the terms' norm), the bias its own, and the row's fp32 mean half a unit in its last place."""
    shape = gpu_toy_shape(dtype=synth.DTYPE_BF16, large=(2, 1088, 17, 128), small=(2, 96, 3, 136), max_pos=64, layer_map=(0, 2))
    w = _bf16_weights(shape, seed=19, std=0.05)
    for tag, m in (("L", shape.large), ("S", shape.small)):
        w[tag + ".emb"] = np.round(w[tag + ".emb"] * 4 * 256).astype(np.float32) / 256
        w[tag + ".pos"] = np.full_like(w[tag + ".pos"], offset)
        for l in range(m.n_layers):
            w[f"{tag}.{l}.wo"] = np.zeros_like(w[f"{tag}.{l}.wo"])
            w[f"{tag}.{l}.w2"] = np.zeros_like(w[f"{tag}.{l}.w2"])
    prompts = prompts_for(shape, [1 + b for b in range(batch)], seed=20)
    t = binding.Tandem(shape, w, max_batch=batch, max_seq=64, gamma_max=gamma)
    t.tandem_prefill(prompts)
    drafts = t.tandem_block_step(gamma)["drafts"]
    small, large = t.tandem_debug_read(binding.READ_SMALL_LOGITS, gamma), t.tandem_debug_read(binding.READ_LARGE_LOGITS, gamma)
    t.close()
    for b in range(batch):
        tokens = [prompts[b][-1]] + drafts[b].tolist()
        for tag, got in (("S", small[:, b]), ("L", large[b])):
            g, bias, head = (w[tag + n].astype(np.float64) for n in (".lnf_g", ".lnf_b", ".w_out"))
            for r, row in enumerate(got):
                x = w[tag + ".emb"][tokens[r]].astype(np.float64) + offset
                z = (x - x.mean()) / np.sqrt(x.var() + 1e-5)
                want = (z * g + bias) @ head.T
                bound = 4 / np.sqrt(3) * 2.0 ** -16 * (np.linalg.norm(z * g * head, axis=1) + np.linalg.norm(bias * head, axis=1))
                bound += 2.0 ** -24 * (abs(x.mean()) / x.std() * abs(head @ g) + 8 * abs(z * g * head).sum(1))
                assert (abs(row - want) <= bound).all()


def test_standalone_calls_refuse_arguments_on_another_device():
    """Any one argument left on the host is refused (an empty segment, which no kernel touches, is not)."""
    import torch
    on = lambda *n, dtype=torch.bfloat16: torch.zeros(n, dtype=dtype, device="cuda")  # noqa: E731
    f32 = torch.float32
    kv, scratch = [on(1, 2, 4, 64) for _ in range(4)], on(1 << 16, dtype=torch.uint8)
    calls = [(binding.tandem_decode_attention, [on(1, 2, 64), *kv, on(1, 2, 64), scratch]),
             (binding.tandem_decode_attention_static, [on(1, 2, 64), *kv, on(1, 2, 64)]),
             (binding.tandem_ff_tandem_project, [on(1, 64), on(64, 64), on(64, dtype=f32), on(64, dtype=f32), on(64, 64), on(64, 64), scratch]),
             (binding.tandem_block_linear, [on(1, 64), on(64, 64), on(1, 64)])]
    for call, args in calls:
        call(*args)
        for i in range(len(args)):
            with pytest.raises(ValueError):
                call(*[a.cpu() if j == i else a for j, a in enumerate(args)])
    none = torch.zeros(1, 2, 0, 64, dtype=torch.bfloat16)
    assert binding.tandem_decode_attention(on(1, 2, 64), none, none, kv[0], kv[1]).shape == (1, 2, 64)
