"""GPU parity of the average pooling and FC layer: batches at the edges of the image groups (1, 4, 8), classes per warp (1, 2,
4), tiles of 8 to 32 images times 8 to 32 classes, channels around the 2048 and the 128 held at a time, image sizes below and above a warp of positions."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2010_16165_b200 import workloads as wl
from test_gpu_parity import Gpu, TOL_BF16, TOL_FP32, err, oracle_pruned

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2010_16165_b200 import binding
    binding.lib()
    return binding


def one_layer(batch, hw, channels, classes):
    net = wl.Net(3, hw, hw, "one_layer")
    x = net.relu(net.bn(net.conv(-1, channels, 3, 1, 1, 0), channels))
    net.fc(net.gavgpool(x, channels), classes, channels)
    net.n_blocks = 0
    return wl.Workload("one_layer", net, batch, 29, False, wl.uniform_ratios(0.0), "none")


@pytest.mark.parametrize("batch, hw, channels, classes", [
    (1, 7, 2048, 1000), (1, 4, 2064, 11), (2, 9, 72, 1003), (4, 3, 4112, 9), (5, 7, 512, 1000), (8, 2, 24, 1),
    (9, 7, 2032, 130), (24, 5, 136, 1000), (83, 3, 520, 1000), (97, 3, 2080, 801),
    (16, 2, 1024, 32), (33, 2, 272, 70), (64, 2, 16, 1000), (129, 2, 784, 1001),      # tiles of 8 images x 8 classes, of 16 x 32
    (31, 2, 144, 1000), (48, 2, 272, 1003), (257, 2, 144, 1000),                      # of 8 x 16, 16 x 16 and 32 x 32
])
@pytest.mark.parametrize("compute", ["fp32", "tc"])
def test_head_matches_oracle(B, fpo, batch, hw, channels, classes, compute):
    w = one_layer(batch, hw, channels, classes)
    g = Gpu(B, w, B.FP_COMPUTE_FP32 if compute == "fp32" else B.FP_COMPUTE_BF16_TC)
    try:
        gp, _, _, _ = oracle_pruned(fpo, w)
        assert err(g.forward(w.x), fpo.fused_forward(gp, w.x)) < (TOL_FP32 if compute == "fp32" else TOL_BF16)
    finally:
        g.close()


@pytest.mark.parametrize("made, hw, channels, classes", [(40, 3, 272, 1000), (300, 2, 144, 70), (16, 4, 2048, 33), (15, 4, 2048, 1000), (64, 2, 528, 31), (20, 2, 2080, 100), (33, 2, 1040, 45), (16, 3, 16, 540_001), (270, 2, 272, 1000)])
@pytest.mark.parametrize("compute", ["fp32", "tc"])
def test_logits_do_not_depend_on_the_batch_of_the_call(B, made, hw, channels, classes, compute):
    """One handle, calls on both sides of 16 images and of the tiles' widths: an image's logits are the same bits in each."""
    w = one_layer(made, hw, channels, classes)
    g = Gpu(B, w, B.FP_COMPUTE_FP32 if compute == "fp32" else B.FP_COMPUTE_BF16_TC)
    try:
        full = g.forward(w.x)
        for n in sorted({n for n in (1, 2, 4, 5, 8, 9, 15, 16, 17, 24, 33, 48, 129, made - 1) if n < made}):
            np.testing.assert_array_equal(g.forward(w.x[:n]), full[:n], err_msg=str(n))
    finally:
        g.close()


@pytest.mark.parametrize("batch, channels, classes", [(1, 32, 11), (3, 32, 11), (9, 528, 9), (24, 528, 1000), (83, 528, 1000)])
@pytest.mark.parametrize("compute", ["fp32", "tc"])
def test_an_infinite_average_stays_infinite(B, batch, channels, classes, compute):
    """Every logit is plus or minus infinity by the sign of its weight for the last channel, whose average is infinite; none is NaN."""
    w = one_layer(batch, 5, channels, classes)
    w.x[:] = 1e20
    bank = w.weights[:channels * 3].reshape(channels, 3)
    bank[:-1] = 1e-3
    bank[-1] = 1e20
    fc = w.weights[channels * 3:channels * 3 + classes * channels].reshape(classes, channels)
    g = Gpu(B, w, B.FP_COMPUTE_FP32 if compute == "fp32" else B.FP_COMPUTE_BF16_TC)
    try:
        np.testing.assert_array_equal(g.forward(w.x), np.broadcast_to(np.sign(fc[:, -1]) * np.inf, (batch, classes)))
    finally:
        g.close()


def test_more_classes_than_one_grid_dimension_holds(B, fpo):
    w = one_layer(2, 3, 16, 540_001)
    g = Gpu(B, w, B.FP_COMPUTE_BF16_TC)
    try:
        gp, _, _, _ = oracle_pruned(fpo, w)
        assert err(g.forward(w.x), fpo.fused_forward(gp, w.x)) < TOL_BF16
    finally:
        g.close()
