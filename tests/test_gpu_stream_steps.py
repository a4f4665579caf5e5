"""3x3 layers with streamed filters whose steps have one to four tiles of 128 positions, and with resident ones: every operator's output against the validation
convolutions, at batches where a CTA has one step or several, the last one partial, filters that stay and filters that come with every
step, a projection taken in (its filter blocks on top), wide images."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2010_16165_b200 import workloads as wl
from test_gpu_op_output import close, outputs
from test_gpu_parity import Gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2010_16165_b200 import binding
    binding.lib()
    return binding


@pytest.mark.parametrize("layers, widths, hw, batch, p", [
    ((2,), (96,), 112, 64, 0.0),            # 421 tiles: one step of three a CTA
    ((2,), (96,), 112, 23, 0.0),            # a tile or two a step
    ((2,), (160,), 100, 57, 0.1),           # two filter tiles or three tiles of 144 filters
    ((1, 1), (64, 112), 120, 70, 0.0),      # a projection's blocks behind the layer's own
    ((2,), (48,), 232, 9, 0.0),             # 58 pixels wide: steps share the halo, the filters stay
    ((2,), (80,), 248, 33, 0.3),            # 62 pixels wide, several steps a CTA, the last one partial
    ((1,), (256,), 72, 47, 0.0),            # filters that take longer than the MMAs of a tile
    ((2,), (64,), 120, 25, 0.0),            # filters that stay as a whole, one or two tiles a CTA: teams that take every other tile
    ((2,), (64,), 120, 61, 0.3),            # the same with narrow tiles, three and four a CTA
])
def test_steps_of_tiles(B, layers, widths, hw, batch, p):
    net = wl.resnet_imagenet_basic(layers, widths, in_hw=hw, n_classes=5, name="steps")
    w = wl.Workload("steps", net, batch, 29, True, wl.uniform_ratios(p), "uniform")
    g, slow = Gpu(B, w, B.FP_COMPUTE_BF16_TC), Gpu(B, w, B.FP_COMPUTE_BF16_SIMT, keep_outputs=1)
    try:
        for x in (g, slow):
            B.fp_prune(x.h, w.ratios)
        logits = g.forward(w.x)
        slow.forward(w.x)
        got, want = outputs(B, g, w), outputs(B, slow, w)
        seen = 0
        for i, o in enumerate(B.op_infos(g.h)):
            if o.kind == 0 and got[i] is not None and want.get(i) is not None and got[i].shape == want[i].shape:
                assert close(got[i], want[i]), i
                seen += 1
        assert seen >= 2 * sum(layers)
        for _ in range(5):                                    # nothing depends on who was first
            np.testing.assert_array_equal(g.forward(w.x), logits)
        np.testing.assert_array_equal(g.forward(w.x[:1]), logits[:1])
    finally:
        g.close()
        slow.close()
