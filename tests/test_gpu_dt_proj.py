"""dt Proj + softplus of the tensor path against fp64 on the rows it was given: one and two K blocks (and a rank beyond, which the
general GEMM takes), token and channel counts that no tile divides, more row tiles than accumulators and operand stages."""
import numpy as np
import pytest
import torch

from paper_2506_18145_b200 import synth
from rom_testlib import GpuLayer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,L,De,R,with_bias", [
    (1, 1, 64, 16, True), (1, 127, 320, 64, True), (2, 65, 192, 80, False), (1, 129, 576, 128, True), (3, 1371, 256, 48, True),
    (1, 9000, 4096, 128, True), (1, 200, 128, 144, True),
])
def test_dt_proj(B, L, De, R, with_bias):
    s = synth.RomShape("dt", B, L, 64, De, 16, 4, R, 2, 1, "bf16", 4711 + De + R)
    p = synth.make_inputs(s, recipe="unit")
    if with_bias:      # both ends of softplus: results that are nearly zero and nearly the argument
        p["b_dt"] = torch.linspace(-30.0, 30.0, De)[torch.randperm(De, generator=torch.Generator().manual_seed(1))].contiguous()
    else:
        p["b_dt"] = None
    g = GpuLayer(s, p)
    g.tap("Delta", torch.bfloat16, De).fill_(-1.0)
    g.forward()
    v = g.tap("delta_r", torch.bfloat16, R).double() @ g.dev["W_dt"].double().T
    if with_bias:
        v = v + g.dev["b_dt"].double()
    ref = torch.nn.functional.softplus(v, threshold=100.0).cpu().numpy()
    got = g.tap("Delta", torch.bfloat16, De).double().cpu().numpy()
    # bf16 rounding (8 significant bits: 2^-8 relative), the fit of log1p (6.3e-5 relative), fp32 sums of R products and the bias (2^-24 of their
    # magnitudes each, passed on to exp by the slope of softplus, at most 1)
    mag = (g.tap("delta_r", torch.bfloat16, R).double().abs() @ g.dev["W_dt"].double().abs().T).cpu().numpy() + 30.0 * with_bias
    bound = ref * (2.0 ** -8 + 1e-4) + np.minimum(ref, 1.0) * mag * (R + 2) * 2.0 ** -24 + 1e-30
    assert (np.abs(got - ref) <= bound).all(), float((np.abs(got - ref) / bound).max())
