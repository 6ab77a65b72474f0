"""A score workspace made for one query serves every smaller one: the size never grows as the
query's rows, columns or clusters shrink (the bands of the integral image get shorter on small
images, so their number does not follow the image)."""
import random

import pytest

from paper_2306_15010_gb300 import _lib, api


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2306_15010_gb300 import build
    build.build()


def _smaller(r, H, W, k, th, tw):
    """Another query of the same template, smaller in one direction or in several."""
    by = lambda: r.choice([0, 1, r.randint(1, 64), r.randint(0, 2048)])  # noqa: E731
    return max(th, H - by()), max(tw, W - by()), max(1, k - r.choice([0, 0, 1, r.randint(0, 255)]))


def test_smaller_query_never_needs_more():
    r = random.Random(5)
    score = lambda H, W, k, th, tw: api.vqnnf_workspace_bytes(_lib.OP_SCORE, H, W, 0, k, th, tw, 1)  # noqa: E731
    host = lambda H, W, k, th, tw: api.vqnnf_match_host_workspace_bytes(H, W, 16, k, th, tw, 1, "fp32")  # noqa: E731
    assert score(1936, 290, 60, 64, 64) <= score(1939, 290, 60, 64, 64)
    for _ in range(30000):
        th, tw = r.randint(8, 300), r.randint(8, 300)
        H, W = max(th, int(2 ** r.uniform(4, 12))), max(tw, int(2 ** r.uniform(4, 12)))
        k = r.randint(1, 256)
        h, w, kk = _smaller(r, H, W, k, th, tw)
        assert score(h, w, kk, th, tw) <= score(H, W, k, th, tw), (H, W, k, h, w, kk, th, tw)
        assert host(h, w, min(kk, th * tw), th, tw) <= host(H, W, min(k, th * tw), th, tw), (H, W, k, h, w, kk, th, tw)


def test_soft_workspace_holds_no_row_sums_where_one_kernel_takes_the_boxes():
    B, H, W, D, k, side, G = 8, 512, 512, 256, 64, 64, 3
    from paper_2306_15010_gb300 import soft
    plane = 4 * B * k * H * W
    classes = 4                                          # cells of 21 and 22 pixels either way
    used = plane * (1 + 2 * classes + 2)                 # p, box sums and adjoint rows by class, two gradients
    l1 = 4 * B * G * G * (H - side + 1) ** 2
    got = soft.soft_workspace_bytes(B, H, W, D, k, side, side, G)
    assert used + l1 <= got < used + l1 + plane // 2
    # cells too large for it keep them
    assert soft.soft_workspace_bytes(1, 300, 300, 4, 8, 200, 200, 1) >= 4 * 8 * 300 * 300 * (1 + 1 + 2 + 2)
