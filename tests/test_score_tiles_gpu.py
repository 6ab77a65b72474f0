"""The score's tile kernel against the dense kernel and the oracle.

A grid bank over an image of at least 512 tiles (64 x 4 windows) with more than 16 clusters is
scored by the tile kernel where the labels are coherent, by the dense kernel where they are not.
Row bands of fewer tiles always take the dense kernel; the two add the same integers in the same
float order, so the whole image's heatmap equals its bands' bit for bit.
"""
import numpy as np
import pytest
import torch

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def vq():
    from paper_2306_15010_gb300 import build
    build.build()
    import paper_2306_15010_gb300 as m
    torch.cuda.set_device(0)
    return m


def _labels(H, W, k, salt, seed):
    q = synth.query_map(H, W, 4, M=6, n_sp=max(8, H * W // 150), seed=seed)
    lab = (q.sp_id.numpy() * 7 % k).astype(np.uint8)
    r = np.random.default_rng(seed)
    noise = r.random((H, W)) < salt
    lab[noise] = r.integers(0, k, size=int(noise.sum()))
    return lab


def _score(vq, lab, k, th, tw, bank, tc):
    heat, am = vq.vqnnf_score(torch.as_tensor(lab).cuda(), k, th, tw, bank, torch.as_tensor(tc.astype(np.int32)).cuda())
    return heat.cpu().numpy(), tuple(am.cpu().tolist())


@pytest.mark.parametrize("salt", [0.0, 0.02, 1.0])
@pytest.mark.parametrize("H,W,th,tw,k,G,full", [
    (160, 1100, 32, 29, 17, 3, True),        # the smallest k; ragged last tile in x and y
    (160, 1100, 32, 29, 129, 3, False),      # two words of clusters, the second nearly empty
    (203, 837, 41, 60, 256, 4, True),        # every label byte; 17 slots
    (460, 741, 200, 240, 45, 2, True),       # regions that reach the 16-bit table's modulus: untested slots
    (400, 1300, 257, 256, 40, 3, True),      # 32-bit table
    (2070, 130, 20, 67, 100, 1, True),       # one tile wide
])
def test_tiles_equal_dense_bands(vq, H, W, th, tw, k, G, full, salt):
    lab = _labels(H, W, k, salt, H + k)
    t = lab[5:5 + th, 3:3 + tw].astype(np.int32)
    bank = synth.grid_bank(th, tw, G, full=full)
    tc = oracle.filter_counts(t, k, bank)
    heat, am = _score(vq, lab, k, th, tw, bank, tc)
    HO, WO = heat.shape
    assert ((WO + 63) // 64) * ((HO + 3) // 4) >= 512
    rows = max(1, 4 * (511 // ((WO + 63) // 64)) - 4)
    for y0 in range(0, HO, rows):
        y1 = min(HO, y0 + rows)
        band, _ = _score(vq, lab[y0:y1 + th - 1], k, th, tw, bank, tc)
        assert np.array_equal(band, heat[y0:y1]), np.argwhere(band != heat[y0:y1])[:5] + [y0, 0]
    assert am == divmod(int(heat.argmax()), WO)


@pytest.mark.parametrize("k", [17, 130])
def test_tiles_equal_oracle(vq, k):
    H, W, th, tw = 152, 1111, 21, 34
    lab = _labels(H, W, k, 0.02, k)
    bank = synth.grid_bank(th, tw, 3)
    tc = oracle.filter_counts(lab[40:40 + th, 900:900 + tw].astype(np.int32), k, bank)
    ref, _ = oracle.score(lab.astype(np.int32), k, th, tw, bank, tc)
    heat, am = _score(vq, lab, k, th, tw, bank, tc)
    # one count of any filter changes H by at least 1 / A_f
    assert np.abs(heat - ref).max() < 0.5 / (th * tw)
    assert am == divmod(int(heat.argmax()), heat.shape[1])


@pytest.mark.parametrize("gauss", ["equal", "exp"])
@pytest.mark.parametrize("H,W,th,tw,k", [(64, 200, 62, 33, 20), (70, 333, 40, 47, 256), (330, 300, 260, 255, 9)])
def test_weighted_grid_tiles_equal_oracle(vq, H, W, th, tw, k, gauss):
    """Fewer window rows than a tile, ragged tiles, every label byte, a 32-bit table; filters by
    whole rows and columns of cells ("equal") and by single cells ("exp")."""
    lab = _labels(H, W, k, 0.02, H + k)
    bank = synth.paper_bank(th, tw, "2,3-rect", 3, gauss)
    tc = oracle.filter_counts(lab[1:1 + th, 2:2 + tw].astype(np.int32), k, bank)
    ref, _ = oracle.score(lab.astype(np.int32), k, th, tw, bank, tc)
    heat, _ = _score(vq, lab, k, th, tw, bank, tc)
    bound = 0.5 * min(f["w_f"] / f["area"] * min(abs(r[4]) for r in f["rects"]) for f in bank)
    # float32 sums of 15 terms of magnitude up to |H|: 16 roundings of 2^-24 |H| each at most
    assert np.abs(heat - ref).max() < bound + 16 * 2.0 ** -24 * np.abs(ref).max()


def test_tiles_counts_beyond_the_table(vq):
    """Template counts of a caller's own beyond 65,535, over a 16-bit table."""
    H, W, th, tw, k = 160, 1100, 32, 29, 17
    lab = _labels(H, W, k, 0.02, 3)
    bank = synth.grid_bank(th, tw, 3, full=True)
    tc = oracle.filter_counts(lab[5:5 + th, 3:3 + tw].astype(np.int32), k, bank)
    tc[:, ::2] += 65537
    heat, _ = _score(vq, lab, k, th, tw, bank, tc)
    band, _ = _score(vq, lab[:40 + th - 1], k, th, tw, bank, tc)          # few tiles: the dense kernel
    assert np.array_equal(band, heat[:40])
