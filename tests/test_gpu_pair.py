"""Bottleneck networks whose stream-writing 1x1 layers run with the 1x1 layer behind them in one kernel (pair_tc.cu): every operator's
output against a handle that runs each layer on its own, at the edges of a group (64 channels), of a tile (128 positions) and of what
shared memory holds - filters that stay, filters that come with every tile, one and two stages of either tensor."""
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


def bottleneck(layers, widths, hw, batch, ratios):
    net = wl.resnet_imagenet_bottleneck(layers, widths, in_hw=hw, n_classes=9, stem_width=16)
    return wl.Workload("pair", net, batch, 43, True, ratios, "pair")


@pytest.mark.parametrize("layers, widths, hw, batch, ratios, pairs", [
    ((2, 1), (16, 24), 64, 66, wl.inner_bottleneck_ratios(0.3), 2),      # one group a tile; the second stream parity-split, a quarter written
    ((1, 2), (20, 40), 56, 87, wl.uniform_ratios(0.3), 1),               # a last group of 16 and of 32 channels
    ((3,), (64,), 36, 191, wl.uniform_ratios(0.0), 2),                   # 9 x 9 pixels, filters stay
    ((2, 2), (128, 128), 52, 99, wl.inner_bottleneck_ratios(0.2), 1),    # odd images (no parity split), filters with every tile
    ((3,), (160,), 20, 531, wl.uniform_ratios(0.0), 1),                  # one stage of x and of the second sums
    ((2,), (48,), 112, 23, wl.inner_bottleneck_ratios(0.5), 1),          # a few tiles a CTA, the last one partial
])
def test_layers_that_run_as_pairs(B, layers, widths, hw, batch, ratios, pairs):
    w = bottleneck(layers, widths, hw, batch, ratios)
    g, kept = Gpu(B, w, B.FP_COMPUTE_BF16_TC), Gpu(B, w, B.FP_COMPUTE_BF16_TC, keep_outputs=1)
    try:
        for x in (g, kept):
            B.fp_prune(x.h, w.ratios)
        logits = g.forward(w.x)
        assert close(logits, kept.forward(w.x))                          # (of what a forward stores; the outputs below are stored whole)
        infos = B.op_infos(g.h)
        assert sum(o.kind == 0 and B.CONV_KERNELS[o.kernel] == "conv_pair_kernel" for o in infos) >= 2 * pairs
        got, want = outputs(B, g, w), outputs(B, kept, w)
        for i, o in enumerate(infos):
            if o.kind == 0:
                assert got[i] is not None and close(got[i], want[i]), i
        for _ in range(10):                                              # nothing depends on who was first
            np.testing.assert_array_equal(g.forward(w.x), logits)
    finally:
        g.close()
        kept.close()


def test_a_smaller_batch_than_the_handle_is_made_for(B):
    w = bottleneck((2, 1), (32, 32), 64, 70, wl.inner_bottleneck_ratios(0.3))
    g = Gpu(B, w, B.FP_COMPUTE_BF16_TC)
    try:
        B.fp_prune(g.h, w.ratios)
        logits = g.forward(w.x)
        for n in (1, 2, 69):
            np.testing.assert_array_equal(g.forward(w.x[:n]), logits[:n])
    finally:
        g.close()


@pytest.mark.parametrize("width, blocks, hw, batch", [
    (16, 2, 24, 40),       # one group of 64 channels
    (20, 2, 23, 41),       # groups of 64 and 16
    (48, 3, 17, 70),       # three groups, filters that stay
    (96, 2, 14, 131),      # six groups, filters with every tile
])
def test_a_pair_computes_what_its_two_layers_do(B, width, blocks, hw, batch):
    """Blocks without projections, so that both handles give the pair the same inputs: every operator's output is the same bits as
    that of a launch of its own."""
    net = wl.Net(3, hw, hw, "pairs_alone")
    x = net.relu(net.bn(net.conv(-1, 4 * width, 3, 1, 1, 0), 4 * width))
    for b in range(blocks):
        x = wl._bottleneck(net, x, 4 * width, width, 1, False, b)
    net.fc(net.gavgpool(x, 4 * width), 5, 4 * width)
    net.n_blocks = blocks
    w = wl.Workload("pairs_alone", net, batch, 59, True, wl.uniform_ratios(0.0), "none")
    g, kept = Gpu(B, w, B.FP_COMPUTE_BF16_TC), Gpu(B, w, B.FP_COMPUTE_BF16_TC, keep_outputs=1)
    try:
        infos = B.op_infos(g.h)
        assert sum(o.kind == 0 and B.CONV_KERNELS[o.kernel] == "conv_pair_kernel" for o in infos) == 2 * (blocks - 1)
        np.testing.assert_array_equal(g.forward(w.x), kept.forward(w.x))
        got, want = outputs(B, g, w), outputs(B, kept, w)
        for i, o in enumerate(infos):
            if o.kind == 0:
                np.testing.assert_array_equal(got[i], want[i], err_msg=str(i))
    finally:
        g.close()
        kept.close()
