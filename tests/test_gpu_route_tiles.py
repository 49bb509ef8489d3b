"""Router logits with one and two tiles of eight experts to a warp, the last tile part empty, at token counts on both sides of the lines for the
split of d_model (148 and 296 blocks of 32 tokens): indices bit-exact against the CPU oracle."""
import pytest

from paper_2506_18145_b200 import synth
from rom_testlib import check_route_exact, gpu_route
from test_gpu_parity import check_layer, small_shape

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("E,K", [(8, 1), (9, 2), (16, 2), (17, 1), (33, 3), (64, 2)])
@pytest.mark.parametrize("tokens", [33, 4737, 9473])
def test_route_tiles(dtype, E, K, tokens):
    s = small_shape(B=1, L=tokens, E=E, K=K, dtype=dtype, d_model=320)
    p = synth.make_inputs(s, recipe="unit")
    check_route_exact(gpu_route(s, p), s, p)


@pytest.mark.parametrize("tokens", [9, 4729, 4737, 9473])
def test_layer_rows_gathered_by_several_blocks_a_chunk(tokens):
    """Four, two and one block to a chunk of 32 tokens, the last chunk short of some of its blocks' tokens."""
    check_layer(small_shape(B=1, L=tokens, d_model=64, d_inner=64, E=8, K=2), "unit")
