"""Device memory of a handle from plan to plan: what a plan that could not be made leaves behind, how much is taken at a time, and what a
smaller plan gives back."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2010_16165_b200 import workloads as wl
from test_gpu_parity import Gpu, to_dev

pytestmark = pytest.mark.gpu

@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2010_16165_b200 import binding
    binding.lib()
    return binding

def forward(B, h, w):
    dx = to_dev(w.x)
    out = torch.empty(w.batch, w.net.n_classes(), device="cuda")
    B.fp_forward(h, dx.to(torch.bfloat16) if w.in_bf16 else dx, w.batch, out)
    torch.cuda.synchronize()
    return out.cpu().numpy().astype(np.float64)

class Pool:
    """A caller's allocator that counts, and refuses what goes over `limit` bytes or the next allocations but `refuse_after`."""

    def __init__(self, B):
        self.live, self.bytes, self.peak, self.limit, self.refuse_after = {}, 0, 0, 1 << 60, -1

        def alloc(n, _user):
            if self.refuse_after == 0 or self.bytes + n > self.limit:
                return None
            self.refuse_after -= 1
            p = torch.cuda.caching_allocator_alloc(int(n))
            self.live[p] = int(n)
            self.bytes += int(n)
            self.peak = max(self.peak, self.bytes)
            return p

        def free(p, _user):
            self.bytes -= self.live.pop(p)
            torch.cuda.caching_allocator_delete(p)

        self.alloc, self.dealloc = B.ALLOC_FN(alloc), B.DEALLOC_FN(free)

@pytest.mark.parametrize("refuse_after", [0, 1, 2])
def test_another_plan_right_behind_one_that_failed(B, refuse_after):
    w = wl.tiny_imagenet_basic(widths=(32, 64, 96), in_hw=48, batch=3, p=0.3)
    g = Gpu(B, w, B.FP_COMPUTE_BF16_TC)
    try:
        B.fp_prune(g.h, w.ratios)
        want = g.forward(w.x)
    finally:
        g.close()
    pool = Pool(B)
    dw, dbn = to_dev(w.weights), to_dev(w.bn)
    h = B.fp_fuse(w.net, dw, dbn, w.batch, B.FP_COMPUTE_BF16_TC, B.FP_DTYPE_BF16 if w.in_bf16 else B.FP_DTYPE_F32, 0, 0, 0, pool)
    try:
        B.fp_prune(h, w.ratios)                                      # (the selection's own buffers are there from now on)
        for _ in range(3):
            pool.refuse_after = refuse_after
            with pytest.raises(B.FpError) as e:
                B.fp_prune(h, np.full(w.net.n_convs(), 0.5))
            assert e.value.status == B.FP_ERR_NOMEM
            with pytest.raises(B.FpError) as e:
                forward(B, h, w)
            assert e.value.status == B.FP_ERR_ARG
            pool.refuse_after = -1
            B.fp_prune(h, w.ratios)
            np.testing.assert_array_equal(forward(B, h, w), want)
    finally:
        B.fp_destroy(h)
    assert not pool.live


def straight_net(hw):
    """Convolutions in a row, most of the activations in the first two, most of the weights in the last."""
    net = wl.Net(3, hw, hw, "straight")
    x, C = -1, 3
    for K, stride in ((64, 1), (64, 1), (16, 2), (16, 2), (16, 2), (512, 1), (512, 1)):
        x = net.relu(net.bn(net.conv(x, K, C, 3, stride, 1), K))
        C = K
    net.fc(net.gavgpool(x, C), 10, C)
    net.n_blocks = 0
    return net


def test_a_plan_takes_no_more_than_the_larger_of_two(B):
    """From few filters where the weights are to few filters where the activations are: with a caller's allocator the old plan's memory is
    back before the new plan's is taken, so room for either is room for the change."""
    w = wl.Workload("straight", straight_net(24), 64, 67, True, wl.uniform_ratios(0.0), "none")
    wide, narrow = np.array([0.0, 0, 0, 0, 0, 0.9, 0.9]), np.array([0.75, 0.75, 0, 0, 0, 0, 0])
    pool = Pool(B)
    dw, dbn = to_dev(w.weights), to_dev(w.bn)
    h = B.fp_fuse(w.net, dw, dbn, w.batch, B.FP_COMPUTE_BF16_TC, B.FP_DTYPE_BF16, 0, 0, 0, pool)
    try:
        B.fp_prune(h, narrow)
        few_activations, want = pool.bytes, forward(B, h, w)
        B.fp_prune(h, wide)
        pool.limit = max(pool.bytes, few_activations)
        B.fp_prune(h, narrow)
        np.testing.assert_array_equal(forward(B, h, w), want)
        B.fp_prune(h, wide)
    finally:
        B.fp_destroy(h)
    assert not pool.live


def test_pruning_gives_memory_back(B):
    w = wl.Workload("straight", straight_net(24), 2, 67, True, wl.uniform_ratios(0.0), "none")
    dw, dbn = to_dev(w.weights), to_dev(w.bn)
    h = B.fp_fuse(w.net, dw, dbn, 8192, B.FP_COMPUTE_BF16_TC, B.FP_DTYPE_BF16, 0, 1)
    try:
        free = lambda: torch.cuda.mem_get_info()[0]                  # noqa: E731
        before = free()
        B.fp_prune(h, np.array([0.75, 0.75, 0, 0, 0, 0, 0]))
        # the first two layers' outputs, 64 -> 16 channels of 26 x 26 positions, less a quarter of what is left of all layers'
        freed, kept = 2 * 8192 * 26 * 26 * 48 * 2, free() - before
        assert kept > freed // 2
        small = forward(B, h, w)
        B.fp_prune(h, np.zeros(7))
        forward(B, h, w)
        B.fp_prune(h, np.array([0.75, 0.75, 0, 0, 0, 0, 0]))
        np.testing.assert_array_equal(forward(B, h, w), small)
    finally:
        B.fp_destroy(h)
