"""Router logits with one and two tiles of eight experts to a warp, the last tile part empty, at token counts on both sides of the lines for the
split of d_model (144, 147, 148 and 296 blocks of 32 tokens), into at most four ranges and into as many as there are (16, 8, 4), uneven ones:
indices bit-exact against the CPU oracle.  And which instance and split the rule takes."""
import pytest
import torch

from paper_2506_18145_b200 import binding as rb
from paper_2506_18145_b200 import synth
from rom_testlib import check_route_exact, gpu_route, launched_kernels
from test_gpu_parity import check_layer, small_shape

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("E,K", [(8, 1), (9, 2), (16, 2), (17, 1), (33, 3), (64, 2)])
@pytest.mark.parametrize("tokens", [33, 4737, 9473])
@pytest.mark.parametrize("d_model", [320, 1088])
def test_route_tiles(dtype, E, K, tokens, d_model):
    s = small_shape(B=1, L=tokens, E=E, K=K, dtype=dtype, d_model=d_model, d_inner=64)
    p = synth.make_inputs(s, recipe="unit")
    check_route_exact(gpu_route(s, p), s, p)


@pytest.mark.parametrize("dtype,tokens,E,tiles,warps", [
    ("bf16", 1000, 8, 1, 16), ("bf16", 1000, 16, 1, 16), ("bf16", 1000, 17, 1, 12), ("bf16", 1000, 40, 1, 10), ("bf16", 4608, 32, 1, 16),
    ("bf16", 4640, 32, 1, 8), ("bf16", 4640, 24, 1, 12), ("bf16", 4736, 32, 1, 16),
    ("bf16", 6000, 8, 1, 8), ("bf16", 6000, 16, 1, 8), ("bf16", 6000, 24, 1, 6), ("bf16", 6000, 40, 1, 10),
    ("bf16", 9473, 8, 1, 4), ("bf16", 9473, 16, 2, 4), ("bf16", 9473, 24, 1, 6), ("bf16", 9473, 40, 1, 5), ("bf16", 9473, 64, 2, 4),
    ("f32", 1000, 16, 1, 16), ("f32", 6000, 16, 1, 8), ("f32", 9473, 16, 1, 8), ("f32", 9473, 64, 1, 8),
])
def test_route_split(dtype, tokens, E, tiles, warps):
    cfg = rb.make_config(1, tokens, 1024, 64, 16, 4, 16, E, 1, dtype)
    tdt = torch.bfloat16 if dtype == "bf16" else torch.float32
    x, W = torch.ones(tokens, 1024, dtype=tdt, device="cuda"), torch.ones(E, 1024, dtype=tdt, device="cuda")
    idx, gates = torch.empty(tokens, 1, dtype=torch.int32, device="cuda"), torch.empty(tokens, 1, device="cuda")
    ws = rb.alloc_workspace(cfg)

    def call():
        rb.rom_route(cfg, x, W, None, idx, gates, None, None, None, None, ws)
    call()
    (name, threads), = [k for k in launched_kernels(call) if "route_logits_topk" in k[0]]
    assert f"Li{tiles}EE" in name and threads == 32 * warps
    assert not idx.any()


@pytest.mark.parametrize("tokens", [9, 4729, 4737, 9473])
def test_layer_rows_gathered_by_several_blocks_a_chunk(tokens):
    """Four, two and one block to a chunk of 32 tokens, the last chunk short of some of its blocks' tokens."""
    check_layer(small_shape(B=1, L=tokens, d_model=64, d_inner=64, E=8, K=2), "unit")
