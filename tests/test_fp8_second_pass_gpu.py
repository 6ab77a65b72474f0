"""The FP8 path's second pass (BF16 contraction where more than an eighth of the pixels stay
ambiguous): exact labels with and without it, and the statistics describe the FP8 contraction."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def vq():
    from paper_2306_15010_gb300 import build
    build.build()
    import paper_2306_15010_gb300 as m
    torch.cuda.set_device(0)
    return m


@pytest.mark.parametrize("n,D,k,near,runs", [
    (1, 16, 2, 0.0, None),
    (127, 64, 33, 0.0, False),      # well-separated centroids: few ambiguous pixels
    (5000, 128, 24, 0.0, False),
    (129, 64, 33, 0.02, True),      # pairs of close centroids: nearly every pixel ambiguous
    (5000, 128, 24, 0.02, True),
    (4097, 1024, 128, 0.02, True),
])
def test_labels_and_statistics(vq, n, D, k, near, runs):
    g = torch.Generator().manual_seed(n + D + k)
    C = torch.rand((k, D), generator=g)
    if near:
        C[k // 2:] = C[:k - k // 2] + near * torch.randn((k - k // 2, D), generator=g)
    X = C[torch.randint(0, k, (n,), generator=g)] + 0.01 * torch.randn((n, D), generator=g)
    stats = torch.zeros(4, dtype=torch.int64, device="cuda")
    got = vq.vqnnf_assign(X.cuda(), C.cuda(), "fp8", stats=stats).cpu().long().reshape(-1)
    d = torch.cdist(X.double(), C.double(), compute_mode="donot_use_mm_for_euclid_dist") ** 2
    at, best = d.gather(1, got[:, None])[:, 0], d.min(1).values
    assert torch.all(at <= best * (1 + 1e-10) + 1e-30)
    flagged, cand, deep, _ = stats.cpu().tolist()
    assert 0 <= flagged <= n and 2 * flagged <= cand <= k * flagged and deep <= flagged
    if runs is not None:
        assert (flagged > n // 8) == runs
