"""FP_Q_OP_OUTPUT on operators that run inside another launch: the first convolution that is pooled in its own kernel, projections inside
the layer that adds them, strided layers of a network that is one kernel - against a handle that keeps every output, and without a
trace in the forwards that follow."""
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


def outputs(B, g, w):
    """operator -> its output, or None where it is refused"""
    got = {}
    for i, o in enumerate(B.op_infos(g.h)):
        if o.kind == 2:
            continue
        channels = [w.net.in_C] if o.kind == 3 else [o.K]
        if o.kind == 0:                                              # kept filters only, or the full width with zeros
            channels.append(B.fp_query_int(g.h, B.FP_Q_CONV_K_FUSED, o.conv_index))
        for C in channels:
            try:
                got[i] = B.fp_query_array(g.h, B.FP_Q_OP_OUTPUT, i, np.float32, w.batch * C * o.P * o.Q)
                break
            except B.FpError as e:
                assert e.status == B.FP_ERR_UNSUPPORTED or (e.status == B.FP_ERR_ARG and C != channels[-1])
                got[i] = None
    return got


def close(a, b):
    return a.shape == b.shape and np.abs(a - b).max() <= 2e-2 * np.abs(b).max()


CASES = {
    "basic_f32": (lambda: wl.tiny_imagenet_basic(batch=3, p=0.3), False),
    "basic_bf16": (lambda: wl.tiny_imagenet_basic(widths=(32, 64, 96), in_hw=48, batch=3, p=0.3), True),
    "bottleneck_odd": (lambda: wl.Workload("odd", wl.resnet_imagenet_bottleneck((1, 1), (16, 32), in_hw=51, n_classes=7, stem_width=16), 2, 71, True,
                                           wl.uniform_ratios(0.3), "uniform"), True),
}


@pytest.mark.parametrize("name", list(CASES))
def test_convolutions_computed_inside_another_launch(B, name):
    make, bf16 = CASES[name]
    w = make()
    g, kept = Gpu(B, w, B.FP_COMPUTE_BF16_TC, in_bf16=bf16), Gpu(B, w, B.FP_COMPUTE_BF16_TC, in_bf16=bf16, keep_outputs=1)
    try:
        for x in (g, kept):
            B.fp_prune(x.h, w.ratios)
        logits = g.forward(w.x)
        kept.forward(w.x)
        launches = B.fp_query_int(g.h, B.FP_Q_N_LAUNCHES)
        assert launches < B.fp_query_int(kept.h, B.FP_Q_N_LAUNCHES)
        got, want = outputs(B, g, w), outputs(B, kept, w)
        infos = B.op_infos(g.h)
        for i, o in enumerate(infos):
            if o.kind == 0 and o.chain < 0:
                assert got[i] is not None and close(got[i], want[i]), i
        assert B.fp_query_int(g.h, B.FP_Q_N_LAUNCHES) == launches
        np.testing.assert_array_equal(g.forward(w.x), logits)
    finally:
        g.close()
        kept.close()


def test_strided_layers_of_a_network_in_one_kernel(B):
    w = wl.tiny_cifar(widths=(16, 32, 64), in_hw=32, batch=3, n_per_stage=2, p=0.3)
    g, kept = Gpu(B, w, B.FP_COMPUTE_BF16_TC), Gpu(B, w, B.FP_COMPUTE_BF16_TC, keep_outputs=1)
    try:
        for x in (g, kept):
            B.fp_prune(x.h, w.ratios)
        logits = g.forward(w.x)
        assert B.fp_query_int(g.h, B.FP_Q_N_LAUNCHES) == 1
        kept.forward(w.x)
        got, want = outputs(B, g, w), outputs(B, kept, w)
        infos = [o for o in B.op_infos(g.h) if o.kind != 2]
        for i, o in enumerate(infos):
            if o.kind == 0:
                last = i + 1 == len(infos) or infos[i + 1].stride == 2
                assert (got[i] is not None) == (o.stride == 2 or last), i
                assert got[i] is None or close(got[i], want[i]), i
        np.testing.assert_array_equal(g.forward(w.x), logits)
    finally:
        g.close()
        kept.close()
