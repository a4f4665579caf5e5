"""GPU parity of the first convolution with its max pooling (stem_pool.cu) beyond the sizes of test_gpu_parity: odd heights
and widths, the widest row one tile holds, runs of pooled rows that end inside an image, fp32 input, unaligned input pointers -
the pooled tensor and its zero border against the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2010_16165_b200 import workloads as wl
from test_gpu_parity import Gpu, TOL_BF16, _stem_net, err, oracle_pruned

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2010_16165_b200 import binding
    binding.lib()
    return binding


@pytest.mark.parametrize("H, W, K, C, batch", [
    (8, 8, 16, 3, 1), (9, 11, 24, 3, 3), (61, 37, 64, 3, 7), (35, 255, 48, 2, 2), (24, 256, 50, 3, 5), (128, 128, 64, 3, 9),
    (50, 129, 64, 1, 4), (23, 200, 33, 3, 40), (38, 24, 16, 3, 150), (64, 40, 64, 3, 70),
])
@pytest.mark.parametrize("bf16", [True, False])
def test_stem_sizes(B, fpo, H, W, K, C, batch, bf16):
    w = wl.Workload("stem_pool", _stem_net(H, W, K, C), batch, 37, bf16, wl.uniform_ratios(0.0), "none")
    g = Gpu(B, w, B.FP_COMPUTE_BF16_TC)
    try:
        assert B.fp_query_int(g.h, B.FP_Q_N_LAUNCHES) == 4          # stem + pooling, convolution, two head kernels
        gp, _, _, _ = oracle_pruned(fpo, w)
        ref_all = fpo.fused_forward(gp, w.x, return_all=True)
        pooled_ref = ref_all[gp.ops[1]["out"]]
        got = g.forward(w.x)
        info = B.op_infos(g.h)[2]
        pooled = B.fp_query_array(g.h, B.FP_Q_OP_OUTPUT, 2, np.float32, batch * pooled_ref.shape[1] * info.P * info.Q)
        assert err(pooled.reshape(pooled_ref.shape).astype(np.float64), pooled_ref) < TOL_BF16
        assert err(got, fpo.fused_forward(gp, w.x)) < TOL_BF16      # the 3x3 convolution behind it reads the border
        # an input that starts in the middle of a pair of columns
        flat = torch.empty(w.x.size + 1, device="cuda", dtype=torch.bfloat16 if bf16 else torch.float32)
        flat[1:] = torch.from_numpy(w.x).cuda().reshape(-1).to(flat.dtype)
        out = torch.empty(batch, g.n_classes, device="cuda")
        B.fp_forward(g.h, flat[1:].view(w.x.shape), batch, out)
        torch.cuda.synchronize()
        np.testing.assert_array_equal(out.cpu().numpy().astype(np.float64), got)
    finally:
        g.close()


@pytest.mark.parametrize("H, W, K, C, batch", [
    (13, 257, 48, 3, 2), (21, 258, 16, 3, 3), (32, 288, 64, 3, 2), (17, 399, 24, 2, 2), (12, 504, 40, 1, 3), (9, 511, 64, 3, 1), (24, 512, 64, 3, 2),
    (30, 40, 65, 3, 9), (23, 100, 80, 3, 40), (16, 184, 96, 3, 5), (11, 256, 112, 1, 2), (40, 33, 128, 3, 7), (18, 290, 128, 3, 2), (26, 381, 100, 2, 1),
])
@pytest.mark.parametrize("bf16", [True, False])
def test_rows_in_strips_and_filters_in_parts(B, fpo, H, W, K, C, batch, bf16):
    """More than 128 convolution columns, more than 64 filters: at the edges of the strips and parts, with one and several CTAs each."""
    test_stem_sizes(B, fpo, H, W, K, C, batch, bf16)
