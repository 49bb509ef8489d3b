"""Routing of few tokens, where every block of the scatter forms its own offsets (up to 148 chunks of 32 tokens), and of one token more:
indices and counts against the oracle, the tables by the device's own checks, on workspaces that held garbage."""
import numpy as np
import pytest
import torch

from paper_2506_18145_b200 import binding as rb
from paper_2506_18145_b200 import synth
from oracle import rom_oracle as O
from rom_testlib import np64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,E,K", [(1, 4, 1), (31, 8, 2), (33, 5, 1), (1025, 64, 2), (2 * 148 * 16, 8, 1), (148 * 32, 33, 2), (148 * 32 + 1, 33, 2)])
def test_route_few_chunks(T, E, K):
    s = synth.RomShape("own", 1, T, 64, 128, 16, 4, 16, E, K, "bf16", 5100 + T)
    p = {k: None if v is None else v.cuda() for k, v in synth.make_inputs(s, recipe="unit").items()}
    cfg = rb.config_from_shape(s)
    ws = rb.alloc_workspace(cfg)
    ws.random_()                                   # nothing may be expected of a workspace
    out, ref = torch.empty_like(p["x"]), torch.empty_like(p["x"])
    idx, counts = torch.empty((T, K), dtype=torch.int32, device="cuda"), torch.empty((E,), dtype=torch.int32, device="cuda")
    gates = torch.empty((T, K), dtype=torch.float32, device="cuda")
    for _ in range(2):
        rb.rom_layer_forward(cfg, rb.make_weights(p), p["x"], out, idx, gates, counts, ws)
    torch.cuda.synchronize()
    assert rb.rom_get_status(ws) == 0
    want = O.route(np64(p["x"].cpu()).reshape(T, 64), np64(p["W_r"].cpu()), None if p["b_r"] is None else np64(p["b_r"].cpu()), K, 0)[0]
    np.testing.assert_array_equal(idx.cpu().numpy(), want)
    np.testing.assert_array_equal(counts.cpu().numpy(), np.bincount(want.ravel(), minlength=E))
    # the tables are validated on the device (ranges, inverse maps, tiles, padded offsets)
    dbg = rb.config_from_shape(s)
    dbg.flags |= rb.ROM_FLAG_DEBUG_CHECKS
    ws2 = rb.alloc_workspace(dbg)
    ws2.random_()
    rb.rom_layer_forward(dbg, rb.make_weights(p), p["x"], ref, None, None, None, ws2)
    torch.cuda.synchronize()
    assert rb.rom_get_status(ws2) == 0
    assert torch.equal(out, ref)
