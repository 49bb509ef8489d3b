"""The device-side timeout path of every kernel with bounded waits that the first grouped projection can run on (one CTA per tile, CTA
pairs, the streamed projections of the single-token step) and of the x Proj and dt Proj kernels.  The host asks for the fault injection; the call must return, report the
wait that ran out, and leave the workspace usable."""
import numpy as np
import pytest
import torch

from paper_2506_18145_b200 import binding as rb
from paper_2506_18145_b200 import synth

from rom_testlib import TOL, GpuLayer, assert_close, np64, oracle_layer
from test_gpu_parity import _status_detail, small_shape
from test_gpu_step_small import one_step

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kw", [
    dict(E=8, K=1, B=1, L=130, d_model=256),             # experts average less than a row tile: one CTA per tile
    dict(E=1, K=1, B=1, L=200, d_model=256),             # one pair
    dict(E=4, K=2, B=2, L=333, d_model=1024),            # more K blocks than stages, half-empty pairs, several tiles a pair
    dict(E=2, K=1, B=2, L=300, d_model=128),             # fewer
])
def test_stalled_projection_is_reported(kw):
    s = small_shape(**kw)
    p = synth.make_inputs(s, recipe="unit")
    g = GpuLayer(s, p, flags=rb.ROM_FLAG_TEST_STALL)
    rb.rom_layer_forward(g.cfg, g.weights, g.dev["x"], g.out, g.idx, g.gates, g.counts, g.ws)
    torch.cuda.synchronize()
    assert _status_detail(g.ws)[1] in (1, 2, 3)
    assert rb.rom_get_status(g.ws) == -6
    good = GpuLayer(s, p)
    good.ws = g.ws
    out = good.forward()
    ref, im = oracle_layer(s, p)
    np.testing.assert_array_equal(good.idx.cpu().numpy(), im["idx"])
    assert_close(np64(out), ref, TOL["bf16"], "out after a timed-out call")


@pytest.mark.parametrize("L,d_inner,dt_rank", [
    (200, 2048, 128),                                    # clusters of eight, four K blocks a CTA; two K blocks and one row tile of the dt Proj
    (300, 1088, 48),                                     # four, uneven shares
    (4300, 2048, 16),                                    # two, more K blocks than stages; more row tiles than stages of the dt Proj
])
def test_stalled_small_projections_are_reported(L, d_inner, dt_rank):
    s = synth.RomShape("stall", 1, L, 128, d_inner, 16, 4, dt_rank, 2, 1, "bf16", 3100 + L)
    p = synth.make_inputs(s, recipe="unit")
    good = GpuLayer(s, p)
    ref = good.forward().clone()
    g = GpuLayer(s, p, flags=rb.ROM_FLAG_TEST_STALL)
    rb.rom_layer_forward(g.cfg, g.weights, g.dev["x"], g.out, g.idx, g.gates, g.counts, g.ws)
    torch.cuda.synchronize()
    waits = int(g.ws[:16].view(torch.int32).cpu()[3])    # bit i: wait 31 + i gave up
    assert waits & 0b111, "dt Proj"
    assert waits & (0b111 << 10), "x Proj"
    assert rb.rom_get_status(g.ws) == -6
    good.ws = g.ws
    assert torch.equal(good.forward(), ref)


@pytest.mark.parametrize("B,E,K,d_model,where", [
    (3, 8, 1, 1024, (1, 2, 3)),                          # no bounded wait in the step's own kernels: the general sequence
    (9, 8, 1, 128, (1, 2, 3)),                           # one operand stage: the same
    (4, 8, 1, 1024, (4, 5, 6, 7)),
    (70, 1, 1, 192, (4, 5, 6, 7)),                       # two passes of columns
    (33, 8, 2, 1024, (4, 5, 6, 7)),
])
def test_stalled_step_is_reported(B, E, K, d_model, where):
    s = small_shape(B=B, L=1, E=E, K=K, d_model=d_model, d_inner=1024, dtype="bf16")
    p = synth.make_inputs(s, recipe="unit")
    ref = one_step(s, p, B)
    ws = one_step(s, p, B, flags=rb.ROM_FLAG_TEST_STALL)[-1]
    assert _status_detail(ws)[1] in where
    assert rb.rom_get_status(ws) == -6
    again = one_step(s, p, B)
    for a, b in zip(again[:5], ref[:5]):
        assert torch.equal(a, b)
