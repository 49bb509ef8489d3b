"""Row passes of the layer's backward in their bf16 top-1 / top-2 forms (reverse of the combine, dx): token counts off the four tokens
of a block and the eight of a thread, widths off the 128 vectors of a pass, 4, 8 and 16 experts and a count without its own form.
(Sums over too few tokens do not average the bf16 roundings down to the 2e-2 of the comparison: one token leaves 3.8e-2 in dW_x, 70 of
six experts 2.25e-2 in dA, the general forms the same.)"""
import pytest

from test_gpu_backward import bshape, run_layer_backward

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kw", [
    dict(B=1, L=131, E=8, K=1, d_model=192, d_inner=320), dict(B=2, L=77, E=8, K=2, d_model=64, d_inner=1088),
    dict(B=1, L=93, E=16, K=1), dict(B=3, L=43, E=16, K=2, d_model=320), dict(B=1, L=70, E=4, K=2), dict(B=1, L=133, E=6, K=2),
])
def test_backward_row_passes(kw):
    run_layer_backward(bshape(dtype="bf16", **kw))
