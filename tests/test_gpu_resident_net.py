"""A whole CIFAR-shaped network as one kernel: every way of giving images to CTAs (four or two CTAs per image, one image per
CTA, two images taking turns, several rounds), the layer shapes at which its pieces change, and what is left to the other
kernels.  Against the oracle, and bit for bit between batch sizes: a result must not depend on how the batch was divided."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2010_16165_b200 import workloads as wl
from test_gpu_parity import Gpu, err, oracle_pruned, TOL_BF16

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2010_16165_b200 import binding
    binding.lib()
    return binding


def test_batches_divided_every_way(B, fpo):
    w = wl.tiny_cifar(widths=(16, 32, 64), in_hw=32, batch=7, n_per_stage=1, p=0.3)
    gp, _, _, _ = oracle_pruned(fpo, w)
    ref = fpo.fused_forward(gp, w.x)
    g = Gpu(B, w, B.FP_COMPUTE_BF16_TC, max_batch=600)
    try:
        B.fp_prune(g.h, w.ratios)
        assert B.fp_query_int(g.h, B.FP_Q_N_LAUNCHES) <= 2           # what full rounds of pairs leave over is a launch of its own
        one = g.forward(w.x)
        assert err(one, ref) < TOL_BF16
        for n in (1, 2, 36, 37, 38, 74, 75, 147, 148, 149, 296, 297, 445, 600):
            x = np.concatenate([w.x] * (n // 7 + 1))[:n]
            np.testing.assert_array_equal(g.forward(x), np.concatenate([one] * (n // 7 + 1))[:n])
        assert B.fp_query_int(g.h, B.FP_Q_DEVICE_STATUS) == 0
    finally:
        g.close()


@pytest.mark.parametrize("widths,hw", [((16, 32, 64), 32), ((8, 8, 8), 32), ((9, 17, 33), 32), ((7, 24, 40), 32), ((16, 48, 56), 32),
                                       ((24, 64), 16), ((33, 50), 16), ((64,), 8), ((12,), 8)])
@pytest.mark.parametrize("batch", [2, 90, 160])          # four CTAs per image, one image per CTA, two images per CTA
def test_layer_shapes(B, fpo, widths, hw, batch):
    net = wl.resnet_cifar(2, widths, in_hw=hw, n_classes=11, pad_lo_centered=True, name="resident_shapes")
    w = wl.Workload("resident_shapes", net, 2, 31 + hw + sum(widths), True, wl.uniform_ratios(0.25), "uniform 0.25")
    g = Gpu(B, w, B.FP_COMPUTE_BF16_TC, max_batch=batch)
    try:
        B.fp_prune(g.h, w.ratios)
        x = np.concatenate([w.x] * (batch // 2))
        got = g.forward(x)
        gp, _, _, _ = oracle_pruned(fpo, w)
        ref = fpo.fused_forward(gp, w.x)
        assert err(got[:2], ref) < TOL_BF16
        np.testing.assert_array_equal(got, np.concatenate([got[:2]] * (batch // 2)))
    finally:
        g.close()


@pytest.mark.parametrize("p", [0.2, 0.55])
def test_second_image_of_a_pair_keeps_its_filters(B, p):
    """ResNet-32 at ratios where filters lie in the place of the next layer's result: the first image of a pair must not clear it
    before the second one has read them."""
    net = wl.resnet_cifar(5)
    w = wl.Workload("resident_pairs", net, 8, 53, True, wl.uniform_ratios(p), "uniform")
    g = Gpu(B, w, B.FP_COMPUTE_BF16_TC, max_batch=296)
    try:
        B.fp_prune(g.h, w.ratios)
        one = np.concatenate([g.forward(w.x[i:i + 1]) for i in range(8)])
        x = np.concatenate([w.x] * 37)
        for _ in range(5):
            np.testing.assert_array_equal(g.forward(x), np.concatenate([one] * 37))
    finally:
        g.close()


@pytest.mark.parametrize("hw, widths", [(32, (16, 32, 64)), (8, (24,))])
def test_rows_that_never_come_are_reported(B, hw, widths):
    """CTAs that share an image wait for each other's border rows: with one of them announcing its rows on the wrong barrier, the wait runs
    out after a millisecond, the status says so - once - and the next forward is as before."""
    net = wl.resnet_cifar(2, widths, in_hw=hw)
    w = wl.Workload("resident_expiry", net, 3, 59, True, wl.uniform_ratios(0.3), "uniform")
    g = Gpu(B, w, B.FP_COMPUTE_BF16_TC)
    try:
        B.fp_prune(g.h, w.ratios)
        assert B.fp_query_int(g.h, B.FP_Q_N_LAUNCHES) == 1
        before = g.forward(w.x)
        B.fp_debug_expire_wait(g.h)
        torch.cuda.synchronize()
        assert B.fp_query_int(g.h, B.FP_Q_DEVICE_STATUS) == B.FP_ERR_TIMEOUT
        assert B.fp_query_int(g.h, B.FP_Q_DEVICE_STATUS) == 0
        np.testing.assert_array_equal(g.forward(w.x), before)
    finally:
        g.close()


@pytest.mark.parametrize("per_stage, batch, one_kernel", [(3, 444, True), (9, 256, True), (9, 444, False), (18, 444, False), (18, 1024, False)])
def test_one_kernel_or_layer_by_layer(B, per_stage, batch, one_kernel):
    """The form is chosen by the batch that the handle is made for.  Deep networks on many images go in runs of layers - several images per
    group, several groups per CTA - and agree with the one-kernel form of a handle for few images; a result is the same for every batch."""
    net = wl.resnet_cifar(per_stage)
    w = wl.Workload("forms", net, 8, 61, True, wl.uniform_ratios(0.3), "uniform")
    few, many = Gpu(B, w, B.FP_COMPUTE_BF16_TC), Gpu(B, w, B.FP_COMPUTE_BF16_TC, max_batch=batch)
    try:
        for g in (few, many):
            B.fp_prune(g.h, w.ratios)
        want = few.forward(w.x)
        assert B.fp_query_int(few.h, B.FP_Q_N_LAUNCHES) == 1
        x = np.concatenate([w.x] * (batch // 8 + 1))[:batch]
        got = many.forward(x)
        assert (B.fp_query_int(many.h, B.FP_Q_N_LAUNCHES) <= 2) == one_kernel
        # two orders of fp32 sums with every layer rounded to bf16: 1.5e-2 between two such paths at 109 layers (test_gpu_parity.py)
        assert err(got[:8], want) < TOL_BF16
        np.testing.assert_array_equal(got, np.concatenate([got[:8]] * (batch // 8 + 1))[:batch])
        np.testing.assert_array_equal(many.forward(w.x[:3]), got[:3])
    finally:
        few.close()
        many.close()
