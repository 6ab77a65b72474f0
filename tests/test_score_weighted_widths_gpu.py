"""Weighted-grid banks over the range of template widths (staged corner by corner), against the oracle:
one window column, the widest template, 16- and 32-bit tables, one cluster and every label byte."""
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
@pytest.mark.parametrize("H,W,th,tw,k", [
    (25, 256, 16, 256, 5),
    (70, 307, 60, 250, 130),
    (300, 290, 270, 256, 3),
    (45, 97, 9, 9, 256),
    (321, 351, 310, 219, 1),
    (40, 190, 33, 127, 64),
])
def test_equal_oracle(vq, H, W, th, tw, k, gauss):
    r = np.random.default_rng(H + W + k)
    lab = r.integers(0, k, size=((H + 10) // 11, (W + 10) // 11)).repeat(11, 0).repeat(11, 1)[:H, :W].astype(np.uint8)
    noise = r.random((H, W)) < 0.03
    lab[noise] = r.integers(0, k, size=int(noise.sum()))
    bank = synth.paper_bank(th, tw, "2,3-rect", 3, gauss)
    tc = oracle.filter_counts(lab[:th, :tw].astype(np.int32), k, bank)
    ref, _ = oracle.score(lab.astype(np.int32), k, th, tw, bank, tc)
    heat, am = vq.vqnnf_score(torch.as_tensor(lab).cuda(), k, th, tw, bank, torch.as_tensor(tc.astype(np.int32)).cuda())
    heat = heat.cpu().numpy()
    # 15 non-negative terms in float32: each from a weight rounded twice and a rounded count, and added
    # with a rounding: at most 18 roundings of 2^-24 |H|
    assert np.abs(heat - ref).max() <= 18 * 2.0 ** -24 * np.abs(ref).max()
    assert tuple(am.cpu().tolist()) == divmod(int(heat.argmax()), heat.shape[1])
