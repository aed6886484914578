"""Edges of the kernels' dispatch rules and tiles, each against the fp64 checker."""
import pytest

from paper_2402_08644_b200 import binding, build, synth
from test_gpu_parity import TOL_FP32, _replay_compare, gpu_toy_shape, prompts_for, toy_weights

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
