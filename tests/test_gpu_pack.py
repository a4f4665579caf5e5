"""GPU parity of the filter packing: banks of one to seventeen units (chunks of 8 channels, eight of them with 1x1 filters),
i.e. runs of one, two and four units with and without a remainder, filters of more than nine taps in several pieces,
filter counts around the 32 rows of a block; channels removed in between."""
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


def two_layers(first, channels, second, filters):
    """A convolution that loses channels, and one that reads what is left of them."""
    net = wl.Net(3, 6, 6, "two_layers")
    x = net.relu(net.bn(net.conv(-1, channels, 3, first, 1, first // 2), channels))
    x = net.relu(net.bn(net.conv(x, filters, channels, second, 1, second // 2), filters))
    net.fc(net.gavgpool(x, filters), 5, filters)
    net.n_blocks = 0
    return wl.Workload("two_layers", net, 3, 31, False, wl.uniform_ratios(0.3), "p0.3")


@pytest.mark.parametrize("first, channels, second, filters", [
    (3, 24, 3, 44), (3, 92, 3, 46), (3, 190, 3, 90), (1, 96, 1, 33), (1, 740, 1, 47), (1, 1500, 1, 31), (5, 40, 5, 48),
    (7, 20, 7, 17),
])
@pytest.mark.parametrize("compute", ["fp32", "tc"])
def test_packed_filters_match_oracle(B, fpo, first, channels, second, filters, compute):
    w = two_layers(first, channels, second, filters)
    g = Gpu(B, w, B.FP_COMPUTE_FP32 if compute == "fp32" else B.FP_COMPUTE_BF16_TC)
    try:
        B.fp_prune(g.h, w.ratios)
        gp, _, _, _ = oracle_pruned(fpo, w)
        assert err(g.forward(w.x), fpo.fused_forward(gp, w.x)) < (TOL_FP32 if compute == "fp32" else TOL_BF16)
    finally:
        g.close()
