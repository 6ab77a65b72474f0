"""Weighted grids over a 32-bit table: the tile kernel where the labels are coherent, the dense one where
most clusters are in every window; which one ran is told by the probe's sign in the workspace."""
import numpy as np
import pytest
import torch

import oracle
import synth

pytestmark = pytest.mark.gpu

AUX = 17664        # the workspace ends with the probe's words: 17,504 bytes from a 256-byte boundary


@pytest.fixture(scope="module")
def vq():
    from paper_2306_15010_gb300 import build
    build.build()
    import paper_2306_15010_gb300 as m
    torch.cuda.set_device(0)
    return m


@pytest.mark.parametrize("H,W,th,tw,k,filters,gauss,coherent", [
    (300, 700, 262, 251, 40, "gauss", "exp", True),      # one filter a grid, fewer than 304 dense blocks
    (300, 700, 262, 251, 40, "gauss", "exp", False),
    (300, 700, 262, 251, 39, "gauss", "equal", False),   # whole columns and rows, one filter a grid
    (570, 340, 262, 256, 33, "2,3-rect", "exp", True),   # five filters a grid
    (570, 340, 262, 256, 33, "2,3-rect", "exp", False),
    (263, 258, 262, 256, 6, "gauss", "exp", False),      # two window rows
    (440, 1300, 330, 200, 130, "2-rect", "exp", False),  # the narrower of the dense strips; a third block in x
    (300, 700, 262, 251, 40, "2,3-rect", "equal", None),  # no probe
])
def test_routes_equal_oracle(vq, H, W, th, tw, k, filters, gauss, coherent):
    r = np.random.default_rng(H + W + k)
    if coherent:                                          # each cluster in a band of columns of its own
        lab = (np.arange(W) * k // W).astype(np.uint8)[None].repeat(H, 0).copy()
    else:
        lab = r.integers(0, k, size=(H, W)).astype(np.uint8)
    bank = synth.paper_bank(th, tw, filters, 3, gauss)
    tc = oracle.filter_counts(lab[:th, :tw].astype(np.int32), k, bank)
    ref, _ = oracle.score(lab.astype(np.int32), k, th, tw, bank, tc)
    nb = vq.vqnnf_workspace_bytes(3, H, W, 0, k, th, tw, len(bank))
    ws = vq.Workspace(nb)
    heat, am = vq.vqnnf_score(torch.as_tensor(lab).cuda(), k, th, tw, bank, torch.as_tensor(tc.astype(np.int32)).cuda(), ws=ws)
    heat = heat.cpu().numpy()
    # non-negative terms in float32: each from a weight rounded twice and a rounded sum, and added with a
    # rounding
    assert np.abs(heat - ref).max() <= (len(bank) + 3) * 2.0 ** -24 * np.abs(ref).max()
    assert tuple(am.cpu().tolist()) == divmod(int(heat.argmax()), heat.shape[1])
    probe = int(ws.tensor[nb - AUX + 8:nb - AUX + 16].cpu().view(torch.int64)[0])
    assert probe == 0 if coherent is None else (probe < 0) == coherent and probe != 0
