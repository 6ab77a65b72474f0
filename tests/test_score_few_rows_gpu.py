"""Weighted-grid banks on queries with fewer window rows than a tile: the rows of a taller query, bit
for bit (a window's score depends on its own labels alone), and the oracle's."""
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


@pytest.mark.parametrize("gauss", ["equal", "exp"])
@pytest.mark.parametrize("W,th,tw,k", [(200, 62, 33, 20), (333, 40, 47, 256), (300, 260, 255, 9)])
def test_rows_of_a_taller_query(vq, W, th, tw, k, gauss):
    r = np.random.default_rng(W + k)
    H = th + 8
    lab = r.integers(0, k, size=((H + 6) // 7, (W + 6) // 7)).repeat(7, 0).repeat(7, 1)[:H, :W].astype(np.uint8)
    noise = r.random((H, W)) < 0.05
    lab[noise] = r.integers(0, k, size=int(noise.sum()))
    bank = synth.paper_bank(th, tw, "2,3-rect", 3, gauss)
    bank = [bank[i] for i in r.permutation(len(bank))]           # the grids' filters interleaved
    tc = oracle.filter_counts(lab[3:3 + th, 2:2 + tw].astype(np.int32), k, bank)

    def score(y0, y1):
        heat, am = vq.vqnnf_score(torch.as_tensor(np.ascontiguousarray(lab[y0:y1])).cuda(), k, th, tw, bank,
                                  torch.as_tensor(tc.astype(np.int32)).cuda())
        return heat.cpu().numpy(), tuple(am.cpu().tolist())

    whole, _ = score(0, H)
    for y0 in (0, 4):
        for rows in (1, 2, 3):
            heat, am = score(y0, y0 + th + rows - 1)
            assert heat.shape[0] == rows
            assert np.array_equal(heat.view(np.uint32), whole[y0:y0 + rows].view(np.uint32))
            assert am == divmod(int(heat.argmax()), heat.shape[1])
            ref, _ = oracle.score(lab[y0:y0 + th + rows - 1].astype(np.int32), k, th, tw, bank, tc)
            # float32 sums of 15 terms of magnitude up to |H|: 16 roundings of 2^-24 |H| each at most
            assert np.abs(heat - ref).max() <= 16 * 2.0 ** -24 * np.abs(ref).max()
