"""The FP32 contraction's tile sizes (chosen by the number of pixels and centroids) at their edges:
labels against 64-bit distances."""
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


@pytest.mark.parametrize("n", [1, 31, 33, 4096, 4097, 4225])
@pytest.mark.parametrize("k", [1, 31, 32, 33, 64, 65, 127, 128, 129, 256])
@pytest.mark.parametrize("D", [4, 20, 68])
def test_labels_equal_64_bit_argmin(vq, n, k, D):
    g = torch.Generator().manual_seed(n * 1000 + k * 3 + D)
    C = torch.rand((k, D), generator=g)
    X = C[torch.randint(0, k, (n,), generator=g)] + 0.02 * torch.randn((n, D), generator=g)
    d = ((X.double()[:, None, :] - C.double()[None]) ** 2).sum(-1) if n * k * D < 1 << 24 else \
        torch.cdist(X.double(), C.double(), compute_mode="donot_use_mm_for_euclid_dist") ** 2
    got = vq.vqnnf_assign(X.cuda(), C.cuda(), "fp32").cpu().long().reshape(-1)
    best = d.min(1).values
    at = d.gather(1, got[:, None])[:, 0]
    # exact but for near-ties of relative gap 1e-11 or less
    assert torch.all(at <= best * (1 + 1e-10) + 1e-30)
