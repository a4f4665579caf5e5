"""Scoring, ranking and masking one bank at the sizes where the kernels change shape: one filter, fewer filters than a
cluster has CTAs or warps, the last bank a single launch takes and the first it does not (by filters and by weights), and
batches of loads that end inside a filter.  Scores are exact doubles in a fixed order, so ranks and masks are one answer.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2010_16165_b200 import binding
    return binding


@pytest.mark.parametrize("norm", [0, 1])
@pytest.mark.parametrize("K,per", [(1, 1), (3, 27), (8, 31), (64, 576), (65, 32), (255, 513), (256, 512), (257, 512), (512, 256),
                                   (512, 255), (513, 9), (1000, 4609), (4096, 3)])
def test_static_rank_sizes(B, K, per, norm):
    from oracle import fpo
    rng = np.random.default_rng(K * 7919 + per)
    w = rng.standard_normal((K, per)).astype(np.float32)
    if K > 8:
        w[K // 2] = w[1]                     # a tie: the lower index comes first
    q = K // 3
    bank = torch.from_numpy(w).cuda()
    rank = torch.full((K,), -1, dtype=torch.int32, device="cuda")
    mask = torch.full((K,), 7, dtype=torch.uint8, device="cuda")
    B.fp_rank_filters_static(bank, K, per, norm, q, rank, mask)
    torch.cuda.synchronize()
    scores = fpo.score_filters(w.reshape(K, per, 1, 1), norm)
    want_mask, want_rank = fpo.rank_mask(scores, q)
    np.testing.assert_array_equal(rank.cpu().numpy(), want_rank)
    np.testing.assert_array_equal(mask.cpu().numpy(), want_mask)


def test_all_masks_at_once(B):
    """FP_Q_ALL_MASKS gives what FP_Q_MASK and FP_Q_RANK give convolution by convolution, absorbed ones included."""
    from paper_2010_16165_b200 import workloads as wl
    w = wl.tiny_imagenet_basic(aggressive=True, p=0.3)
    h = B.fp_fuse(w.net, torch.from_numpy(w.weights).cuda(), torch.from_numpy(w.bn).cuda(), 2)
    try:
        B.fp_prune(h, w.ratios)
        for ci, (mask, rank) in B.masks_and_ranks(h).items():
            K = B.fp_query_int(h, B.FP_Q_CONV_K_FUSED, ci)
            if K == 0:
                assert mask is None and rank is None
                continue
            np.testing.assert_array_equal(mask, B.fp_query_array(h, B.FP_Q_MASK, ci, np.uint8, K))
            np.testing.assert_array_equal(rank, B.fp_query_array(h, B.FP_Q_RANK, ci, np.int32, K))
    finally:
        B.fp_destroy(h)
