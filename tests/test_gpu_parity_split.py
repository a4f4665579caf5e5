"""Tensors stored as four parity images, written by conv_tc_kernel for images of odd height and width: the odd-parity images then have a row and a
column that do not exist and are read.  Filters that stay (four epilogue warps, teams that take every other tile) and streamed ones (sixteen
warps), whole and scattered outputs: every operator's output against the validation convolutions, and the same logits again behind a forward
that leaves large values and NaN wherever nobody writes."""
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


@pytest.mark.parametrize("widths, hw, batch, p, scatter, form", [
    ((48, 64), 100, 70, 0.0, 0, dict(tps=1, stays=1, epi_warps=4, alternate=0)),
    ((64, 96), 100, 70, 0.0, 0, dict(tps=1, stays=1, epi_warps=8, alternate=1)),
    ((160, 96), 100, 70, 0.0, 0, dict(tps=2, stays=0, epi_warps=16)),
    ((160, 96), 100, 70, 0.3, 1, dict(tps=3, stays=0, epi_warps=8)),
    ((64, 96), 108, 70, 0.3, 1, dict(tps=1, stays=1, epi_warps=4, alternate=0)),
    ((80, 96), 108, 70, 0.3, 1, dict(tps=1, stays=1, epi_warps=8, alternate=1)),
    ((96, 96), 108, 70, 0.3, 1, dict(tps=3, stays=0, epi_warps=8)),
])
def test_odd_images(B, widths, hw, batch, p, scatter, form):
    net = wl.resnet_imagenet_basic((2, 1), widths, in_hw=hw, n_classes=5, name="odd")
    w = wl.Workload("odd", net, batch, 41, True, wl.uniform_ratios(p), "uniform")
    g, slow = Gpu(B, w, B.FP_COMPUTE_BF16_TC, scatter=scatter), Gpu(B, w, B.FP_COMPUTE_BF16_SIMT, keep_outputs=1)
    try:
        for x in (g, slow):
            B.fp_prune(x.h, w.ratios)
        writer, reader = 6, 7                                    # the first stage's last layer, the second one's first
        logits = g.forward(w.x)
        infos, plan = B.op_infos(g.h), B.fp_query_plan(g.h, writer)
        assert {k: plan[k] for k in form} == form
        assert infos[writer].P % 2 == 1 and infos[reader].stride == 2 and infos[reader].H == infos[writer].P
        assert B.CONV_KERNELS[infos[reader].kernel] == "conv_split_kernel"      # which reads a strided layer's input as parity images only
        slow.forward(w.x)
        got, want = outputs(B, g, w), outputs(B, slow, w)
        for i in (writer, reader, reader + 1):
            assert got[i] is not None and got[i].shape == want[i].shape and close(got[i], want[i]), i
        for x in (w.x * 1e4, np.full_like(w.x, np.nan)):
            g.forward(x)
            np.testing.assert_array_equal(g.forward(w.x), logits)
        np.testing.assert_array_equal(g.forward(w.x[:3]), logits[:3])
    finally:
        g.close()
        slow.close()
