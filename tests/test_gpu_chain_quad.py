"""Runs of 16-filter layers on images 32 pixels wide (chain_quad.cu) against the CPU oracle: heights whose blocks end inside a tile, one and
two images a group, a last group of one, several groups a CTA, both input types, a run that does not begin at the network's input."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2010_16165_b200 import workloads as wl
from test_gpu_parity import Gpu, TOL_BF16, err, oracle_pruned

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2010_16165_b200 import binding
    binding.lib()
    return binding


def rect(H, widths, batch, bf16, p, per_stage=2):
    net = wl.resnet_cifar(per_stage, widths, in_hw=32, n_classes=5, name="quad")
    net.in_H = H
    return wl.Workload("quad", net, batch, 71, bf16, wl.uniform_ratios(p), "uniform")


def quad_layers(B, g):
    return sum(o.kind == 0 and B.CONV_KERNELS[o.kernel] == "chain_quad_kernel" for o in B.op_infos(g.h))


@pytest.mark.parametrize("H, widths, batch, bf16, p", [
    (2, (16, 16, 16), 3, True, 0.0), (12, (16, 32, 64), 7, False, 0.3), (24, (7, 12, 23), 5, True, 0.3), (30, (16, 20, 40), 2, True, 0.0),
    (34, (16, 32, 32), 3, False, 0.5), (24, (12, 16, 16), 149, True, 0.25), (16, (16, 16, 16), 301, False, 0.0),
])
def test_heights_and_groups(B, fpo, H, widths, batch, bf16, p):
    w = rect(H, widths, batch, bf16, p)
    g = Gpu(B, w, B.FP_COMPUTE_BF16_TC)
    try:
        B.fp_prune(g.h, w.ratios)
        assert quad_layers(B, g) >= 5
        got = g.forward(w.x)
        gp, _, _, _ = oracle_pruned(fpo, w)
        assert err(got, fpo.fused_forward(gp, w.x)) < TOL_BF16
        for _ in range(5):                                    # nothing depends on who was first
            np.testing.assert_array_equal(g.forward(w.x), got)
        np.testing.assert_array_equal(g.forward(w.x[:1]), got[:1])
    finally:
        g.close()


def test_a_run_behind_another_layer(B, fpo):
    """A stem and pooling in front: the run reads a planar tensor that another kernel wrote, and its first layer is one of a block."""
    w = wl.tiny_imagenet_basic(layers=(3, 1, 1), widths=(16, 24, 40), in_hw=128, batch=5, p=0.3)
    g = Gpu(B, w, B.FP_COMPUTE_BF16_TC)
    try:
        B.fp_prune(g.h, w.ratios)
        assert quad_layers(B, g) >= 4                       # (layers that write tensors others read run by themselves)
        got = g.forward(w.x)
        gp, _, _, _ = oracle_pruned(fpo, w)
        assert err(got, fpo.fused_forward(gp, w.x)) < TOL_BF16
    finally:
        g.close()
