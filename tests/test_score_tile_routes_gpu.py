"""Grid banks by the tile kernel and by the dense kernel, told apart by the probe in the workspace: coherent
labels (a cluster per column band) take the tiles, with the 32-bit table, with regions too large to be
tested, with template counts beyond 16 bits, at the fewest and the most clusters.  Row bands of fewer
than 512 tiles are always dense; the whole image's heatmap equals theirs bit for bit."""
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


def _score(vq, lab, k, th, tw, bank, tc):
    nb = vq.vqnnf_workspace_bytes(3, lab.shape[0], lab.shape[1], 0, k, th, tw, len(bank))
    ws = vq.Workspace(nb)
    heat, am = vq.vqnnf_score(torch.as_tensor(np.ascontiguousarray(lab)).cuda(), k, th, tw, bank,
                              torch.as_tensor(tc.astype(np.int32)).cuda(), ws=ws)
    probe = int(ws.tensor[nb - AUX + 8:nb - AUX + 16].cpu().view(torch.int64)[0])
    return heat.cpu().numpy(), tuple(am.cpu().tolist()), probe


@pytest.mark.parametrize("H,W,th,tw,k,G,full,extra,kind", [
    (160, 1100, 32, 29, 17, 3, True, 0, "bands"),        # the fewest clusters
    (160, 1100, 32, 29, 129, 3, False, 0, "bands"),      # two words of clusters, the second nearly empty
    (203, 837, 41, 60, 256, 4, True, 0, "bands"),        # every label byte; 17 slots
    (460, 741, 200, 240, 90, 2, True, 0, "bands"),       # the full window's region reaches the 16-bit modulus
    (400, 1300, 257, 256, 120, 3, True, 0, "bands"),     # 32-bit table
    (2080, 300, 300, 220, 60, 2, False, 0, "rows"),      # the same, two tiles wide
    (160, 1100, 32, 29, 100, 3, True, 65537, "bands"),   # counts beyond the 16-bit table
    (160, 1100, 32, 29, 17, 3, True, 0, "noise"),
    (400, 1300, 257, 256, 40, 3, True, 0, "noise"),
])
def test_route_and_bits(vq, H, W, th, tw, k, G, full, extra, kind):
    r = np.random.default_rng(H + k)
    if kind == "noise":
        lab = r.integers(0, k, size=(H, W)).astype(np.uint8)
    else:
        n = W if kind == "bands" else H
        line = (np.arange(n) * k // n).astype(np.uint8)
        lab = line[None].repeat(H, 0) if kind == "bands" else line[:, None].repeat(W, 1)
        lab = np.ascontiguousarray(lab)
        at = r.random((H, W)) < 5e-5                      # single pixels of other clusters
        lab[at] = r.integers(0, k, size=int(at.sum()))
    bank = synth.grid_bank(th, tw, G, full=full)
    tc = oracle.filter_counts(lab[5:5 + th, 3:3 + tw].astype(np.int32), k, bank)
    tc[:, ::2] += extra
    heat, am, probe = _score(vq, lab, k, th, tw, bank, tc)
    HO, WO = heat.shape
    ntx, tiles = (WO + 63) // 64, (WO + 63) // 64 * ((HO + 3) // 4)
    assert tiles >= 512
    step = tiles // 509 | 1 if tiles // 509 > 1 else 1
    dense_from = 25 * k * ((tiles + step - 1) // step)
    assert (probe <= dense_from) == (kind != "noise")
    rows = max(1, 4 * (511 // ntx) - 4)
    for y0 in range(0, HO, rows):
        y1 = min(HO, y0 + rows)
        band, _, none = _score(vq, lab[y0:y1 + th - 1], k, th, tw, bank, tc)
        assert none == 0                                  # not probed: the dense kernel
        assert np.array_equal(band.view(np.uint32), heat[y0:y1].view(np.uint32))
    assert am == divmod(int(heat.argmax()), WO)
