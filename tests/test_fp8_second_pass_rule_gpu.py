"""The FP8 path's second pass on both sides of its rule: exact labels, and whether it ran, told by the
candidates that were re-scored (all that the FP8 contraction left, or the few that the second pass left)."""
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


def _counters(ws, D, k, n_flagged):
    """(second list's pixels, candidates re-scored) from the workspace: the counters come after the mean,
    the codebook's three copies and its four bounds, each on 256 bytes."""
    off = 0
    for nbytes in (4 * D, 4 * k * D, 2 * k * D, 2 * k * D, 4 * k, 4 * k, 4 * k, 4 * k):
        off = (off + 255) // 256 * 256 + nbytes
    off = (off + 255) // 256 * 256
    words = ws.tensor[off:off + 256].cpu()
    count = words.view(torch.int32)
    assert int(count[0]) == n_flagged                       # the place is right
    return int(count[1]), int(words[64:].view(torch.int64)[1])


@pytest.mark.parametrize("n,D,k,near,noise,runs", [
    (8192, 128, 33, 1, 0.01, False),      # 2^20 values, separated centroids: the first list, nearly empty
    (8192, 128, 33, 8, 0.01, True),       # eight centroids close to each other
    (8191, 128, 33, 8, 0.01, False),      # below 2^20 values
    (65536, 16, 16, 4, 0.01, True),
    (16385, 64, 40, 2, 0.01, True),
    (4099, 512, 64, 2, 0.01, False),      # every pixel ambiguous, two candidates each: re-scoring is faster
    (4099, 512, 64, 16, 0.01, True),
    (1031, 1024, 24, 2, 0.01, False),     # features beyond the registers
    (3001, 1024, 24, 6, 0.01, True),
    (65537, 64, 128, 1, 0.3, False),      # some ambiguous pixels, few candidates
])
def test_labels_and_route(vq, n, D, k, near, noise, runs):
    g = torch.Generator().manual_seed(n + D + k)
    base = torch.rand(((k + near - 1) // near, D), generator=g)
    C = (base.repeat(near, 1)[:k] + 0.03 * torch.randn((k, D), generator=g)).cuda()
    X = C[torch.randint(0, k, (n,), generator=g)] + noise * torch.randn((n, D), generator=g).cuda()
    ws = vq.Workspace(vq.vqnnf_workspace_bytes(1, 1, n, D, k, prec="fp8"))
    stats = torch.zeros(4, dtype=torch.int64, device="cuda")
    got = vq.vqnnf_assign(X, C, "fp8", stats=stats, ws=ws).long().reshape(-1)
    d = torch.cdist(X.double(), C.double(), compute_mode="donot_use_mm_for_euclid_dist") ** 2
    at, best = d.gather(1, got[:, None])[:, 0], d.min(1).values
    assert torch.all(at <= best * (1 + 1e-10) + 1e-30)
    flagged, left, _, _ = stats.cpu().tolist()
    second, rescored = _counters(ws, D, k, flagged)
    if runs:
        assert rescored < left and second < flagged
    else:
        assert rescored == left and second == 0
