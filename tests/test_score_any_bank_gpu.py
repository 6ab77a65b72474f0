"""Banks that are neither grids nor weighted grids, against the oracle: at the number of warps where the
kernel goes over to tiles of four rows, with one cluster and every label byte, 16- and 32-bit tables,
template counts of either sign, many distinct row offsets, and grid banks wider than the grid kernels take."""
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


def _bank(th, tw, F, rects, r):
    out = []
    for _ in range(F):
        rs = []
        for _ in range(rects):
            x0, y0 = int(r.integers(tw)), int(r.integers(th))
            rs.append((x0, y0, int(r.integers(x0 + 1, tw + 1)), int(r.integers(y0 + 1, th + 1)), int(r.choice([-2, -1, 1, 3]))))
        out.append(dict(rects=rs, w_f=0.75, area=float(th * tw)))
    return out


@pytest.mark.parametrize("H,W,th,tw,k,F,rects", [
    (308, 838, 5, 7, 17, 5, 5),          # 26 x 76 tiles of four rows: the fewest that are taken
    (308, 806, 5, 7, 17, 5, 5),          # 25 x 76: one row a warp
    (306, 839, 4, 8, 1, 5, 3),           # the last tile moved up, one cluster
    (60, 75, 33, 31, 256, 6, 20),
    (270, 300, 260, 253, 9, 5, 7),       # 32-bit table; 68 row offsets
    (41, 300, 40, 20, 130, 6, 4),        # two window rows
    (90, 400, 70, 300, 33, 10, 0),       # a 3 x 3 grid and its full window, too wide for the grid kernels
    (262, 330, 256, 270, 5, 5, 0),       # a 2 x 2 grid, 32-bit table
])
def test_equal_oracle(vq, H, W, th, tw, k, F, rects):
    r = np.random.default_rng(H + W + k)
    lab = r.integers(0, k, size=((H + 8) // 9, (W + 8) // 9)).repeat(9, 0).repeat(9, 1)[:H, :W].astype(np.uint8)
    noise = r.random((H, W)) < 0.03
    lab[noise] = r.integers(0, k, size=int(noise.sum()))
    bank = _bank(th, tw, F, rects, r) if rects else synth.grid_bank(th, tw, 3 if F == 10 else 2)
    tc = oracle.filter_counts(lab[:th, :tw].astype(np.int32), k, bank)
    ref, _ = oracle.score(lab.astype(np.int32), k, th, tw, bank, tc)
    heat, am = vq.vqnnf_score(torch.as_tensor(lab).cuda(), k, th, tw, bank, torch.as_tensor(tc.astype(np.int32)).cuda())
    heat = heat.cpu().numpy()
    # F non-negative terms in float32: each from a weight rounded twice and a rounded sum, and added with a
    # rounding: at most F + 3 roundings of 2^-24 |H|
    assert np.abs(heat - ref).max() <= (F + 3) * 2.0 ** -24 * np.abs(ref).max()
    assert tuple(am.cpu().tolist()) == divmod(int(heat.argmax()), heat.shape[1])
