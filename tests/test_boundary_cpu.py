"""Host-only checks of the C boundary: the library builds for sm_100a, loads without a GPU, exports every
symbol the header declares, and validates arguments before touching a device."""
import ctypes as C
import os
import re

import pytest

from paper_2402_08644_b200 import binding, build, synth

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib():
    build.build()
    return binding.load_library()


def _declared_symbols():
    text = open(os.path.join(ROOT, "include", "tandem.h")).read()
    return sorted(set(re.findall(r"TANDEM_API\s+[\w\s\*]+?\b(tandem_\w+)\s*\(", text)))


def test_every_declared_symbol_is_exported(lib):
    names = _declared_symbols()
    assert len(names) >= 13 and "tandem_block_step" in names and "tandem_speculative_generate" in names
    assert sorted(binding.EXPORTS) == [n for n in names if n in binding.EXPORTS]
    for n in names:
        assert hasattr(lib, n), n


def test_status_strings(lib):
    assert lib.tandem_status_string(0) == b"ok"
    assert lib.tandem_status_string(4) == b"capacity exceeded"
    assert len({lib.tandem_status_string(i) for i in range(9)}) == 9


def test_query_arena_validates_and_sizes(lib):
    shape = synth.named_config("small")
    cfg, keep = binding.make_config(shape, max_batch=1, max_seq=1024, gamma_max=3)
    n = binding.tandem_query_arena(cfg)
    kv = (12 * 2 * 1024 * 1024 + 4 * 2 * 1024 * 512) * 2          # both KV caches, bf16
    assert kv < n < kv + (1 << 30)
    bad, keep2 = binding.make_config(shape, max_batch=1, max_seq=1024, gamma_max=16)
    with pytest.raises(binding.TandemError) as e:
        binding.tandem_query_arena(bad)
    assert e.value.status == 1
    odd = synth.make_shape(synth.ModelDims(2, 96, 4, 128, 50, 32), synth.ModelDims(1, 64, 2, 64, 50, 32))
    cfg3, keep3 = binding.make_config(odd, 1, 32, 2)              # head size 24 is not supported
    with pytest.raises(binding.TandemError) as e:
        binding.tandem_query_arena(cfg3)
    assert e.value.status == 2
    out = C.c_size_t(0)
    assert lib.tandem_query_arena(None, C.byref(out)) == 1
    assert lib.tandem_query_arena(C.byref(cfg), None) == 1


def _pair(large, small, vocab, max_pos, kind=synth.FF_TANDEM_LINEAR, hidden=0, dtype=synth.DTYPE_BF16):
    return synth.make_shape(synth.ModelDims(*large, vocab, max_pos), synth.ModelDims(*small, vocab, max_pos), kind, hidden, None, dtype)


@pytest.mark.parametrize("shape,limits,most", [
    (synth.named_config("tiny"), (1, 101, 4, 32), 1595904),
    (synth.named_config("small"), (4, 262, 4, 771), 86630400),
    (synth.named_config("small"), (1, 33, 4, 28), 4482048),
    (synth.named_config("medium", 8192), (16, 8192, 3, 0), 35298047744),
    (synth.named_config("large"), (1, 8448, 5, 0), 5666430976),
    (_pair((2, 128, 2, 136), (2, 192, 6, 136), 50, 200, synth.FF_TANDEM_MLP, 40), (2, 200, 3, 0), 2650880),      # a small model wider than the large one
    (_pair((2, 128, 2, 136), (2, 192, 6, 136), 50, 200, synth.FF_TANDEM_MLP, 40), (1, 200, 15, 1), 882688),      # prompts of one token, long blocks
    (synth.with_dtype(synth.named_config("small"), synth.DTYPE_FP32), (2, 512, 4, 512), 144989952)])
def test_contexts_fit_the_memory_that_prompt_and_decode_passes_need(lib, shape, limits, most):
    """Teacher-forced passes and the heads' arg-max results live in space that other passes have anyway.  `most`: caches, loop state,
    work space of the prompt pass and buffers of the decode passes of these limits, added up without either of the two."""
    cfg, keep = binding.make_config(shape, *limits[:3], max_prefill_rows=limits[3])
    assert binding.tandem_query_arena(cfg) <= most


def test_null_context_calls_fail_cleanly(lib):
    assert lib.tandem_destroy(None) == 1
    assert lib.tandem_block_step(None, 1, 0, 0, None) == 1
    assert lib.tandem_decode_attention_scratch_bytes(0, 1, 64, 1, 1) == 0
    assert lib.tandem_decode_attention_scratch_bytes(2, 16, 64, 1000, 4) >= 2 * 2 * 4


@pytest.mark.parametrize("lead", [0, 1])   # an extra leading dimension: refused too
def test_standalone_calls_refuse_tensors_that_no_kernel_may_touch(lib, lead):
    """Host tensors, and a first argument of another rank, are refused before anything is launched or allocated."""
    import torch
    z = lambda *n, dtype=torch.bfloat16: torch.zeros(n, dtype=dtype)  # noqa: E731
    first = lambda *n: z(*[1] * lead, *n)  # noqa: E731
    kv, scratch = z(1, 2, 4, 64), z(64, dtype=torch.uint8)
    with pytest.raises(ValueError):
        binding.tandem_decode_attention(first(1, 2, 64), kv, kv, kv, kv, z(1, 2, 64), scratch)
    with pytest.raises(ValueError):
        binding.tandem_decode_attention_static(first(1, 2, 64), kv, kv, kv, kv, z(1, 2, 64))
    with pytest.raises(ValueError):
        binding.tandem_ff_tandem_project(first(1, 64), z(64, 64), z(64), z(64), z(64, 64), z(64, 64), scratch)
    with pytest.raises(ValueError):
        binding.tandem_block_linear(first(1, 64), z(64, 64), z(1, 64))
