"""GPU parity of the convolutions with few output positions (conv_split.cu): reductions split over clusters of 1 to 8 CTAs,
narrow and ragged filter tiles, rings shorter than a CTA's share of the reduction, projections taken in, and parity-split
tensors of odd height and width."""
import pytest

torch = pytest.importorskip("torch")

from paper_2010_16165_b200 import workloads as wl
from test_gpu_parity import Gpu, TOL_BF16, _compare_ops, err, oracle_pruned

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2010_16165_b200 import binding
    binding.lib()
    return binding


def basic(batch, hw, widths, p):
    return wl.tiny_imagenet_basic(layers=(1, 2, 1), widths=widths, in_hw=hw, batch=batch, p=p)


def bottleneck(batch, hw, widths, p):
    return wl.tiny_bottleneck(layers=(1, 2, 1), widths=widths, in_hw=hw, batch=batch, p=p)


CASES = [
    # 10, 5 and 3 pixels wide inside (5 -> 3: an odd tensor in parity form); one tile and several
    (basic, 1, 40, (32, 64, 96), 0.0),
    (basic, 7, 40, (16, 48, 160), 0.3),
    # 22, 11, 6: ragged last tiles; K steps from 1 to 45 per CTA
    (basic, 5, 88, (24, 72, 320), 0.3),
    # the widest reductions: 9 x 512 and 2048 long, 7 -> 4 pixels
    (basic, 2, 56, (64, 256, 512), 0.3),
    (bottleneck, 1, 56, (16, 128, 512), 0.4),
    (bottleneck, 9, 72, (8, 40, 96), 0.4),
]


@pytest.mark.parametrize("make, batch, hw, widths, p", CASES)
def test_few_positions_match_oracle(B, fpo, make, batch, hw, widths, p):
    w = make(batch, hw, widths, p)
    gp, _, _, _ = oracle_pruned(fpo, w)
    ref = fpo.fused_forward(gp, w.x)
    for keep in (1, 0):                  # every operator on its own and compared; then with projections taken in
        g = Gpu(B, w, B.FP_COMPUTE_BF16_TC, keep_outputs=keep)
        try:
            B.fp_prune(g.h, w.ratios)
            got = g.forward(w.x)
            if keep:
                _compare_ops(B, g, w, gp, fpo, TOL_BF16)
            assert err(got, ref) < TOL_BF16
            assert (g.forward(w.x) == got).all(), "the sum over the cluster depends on the order of arrival"
        finally:
            g.close()
