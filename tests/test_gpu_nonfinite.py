"""An image with an infinity or a NaN in a corner pixel: the logits of the images before and behind it are the same bits as without it -
in networks that run as one kernel, as runs of layers (both kernels, images 8, 16 and 32 pixels wide) and layer
by layer.  Corner pixels, because in shared and global memory the next image lies right behind the last pixel's row of zeros."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2010_16165_b200 import workloads as wl
from test_gpu_parity import Gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2010_16165_b200 import binding
    binding.lib()
    return binding


def cifar(widths, hw, per_stage=2):
    return wl.resnet_cifar(per_stage, widths, in_hw=hw, n_classes=9, name="nonfinite")


NETS = {
    # network, images, of a handle made for, kernels among those that run
    "one_kernel": (lambda: cifar((16, 32, 64), 32), 11, 11, {"resident_net_kernel"}),
    "runs32": (lambda: cifar((16, 48, 72), 32), 301, 701, {"chain_quad_kernel", "chain_tc_kernel"}),
    "runs32_wide": (lambda: cifar((32, 72), 32), 301, 301, {"chain_tc_kernel"}),
    "runs32_16_8": (lambda: cifar((16, 32, 64), 32, 9), 301, 701, {"chain_quad_kernel", "chain_tc_kernel"}),
    "runs16": (lambda: cifar((16, 72, 80), 16), 40, 600, {"chain_tc_kernel"}),
    "layers": (lambda: wl.resnet_imagenet_basic((2, 1), (16, 40), in_hw=72, n_classes=9), 37, 37, {"conv_split_kernel"}),
    "pairs": (lambda: wl.resnet_imagenet_bottleneck((2, 1), (16, 24), in_hw=64, n_classes=33, stem_width=16), 66, 66, {"conv_pair_kernel"}),
}


@pytest.mark.parametrize("name", list(NETS))
def test_an_image_that_is_not_finite_touches_no_other(B, name):
    make, batch, made, kernels = NETS[name]
    net = make()
    w = wl.Workload("nonfinite", net, batch, 57, True, wl.uniform_ratios(0.1), "uniform 0.1")
    g = Gpu(B, w, B.FP_COMPUTE_BF16_TC, max_batch=made)
    try:
        B.fp_prune(g.h, w.ratios)
        assert kernels <= {B.CONV_KERNELS[o.kernel] for o in B.op_infos(g.h) if o.kind == 0}
        clean = g.forward(w.x)
        assert np.isfinite(clean).all()
        for value in (np.inf, -np.inf, np.nan):
            for corner in ((0, 0), (0, -1), (-1, 0), (-1, -1)):
                bad = [1, 4, 5, batch - 1]
                x = w.x.copy()
                x[(bad, slice(None)) + corner] = value
                got = g.forward(x)
                rest = np.setdiff1d(np.arange(batch), bad)
                np.testing.assert_array_equal(got[rest], clean[rest], err_msg=f"{value} at {corner}")
        np.testing.assert_array_equal(g.forward(w.x), clean)      # nor what runs behind it
    finally:
        g.close()
