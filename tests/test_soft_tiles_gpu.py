"""Soft-VQ at the edges of its tiles, against the FP64 oracle: 128- or 64-pixel tiles and chunks of
32 feature dimensions of the soft assignment (16-byte and scalar loads), 64 x 32 tiles of the box
sums and of the adjoint column pass (one or two cell widths and heights, cells too large for the
tiles), 1 to 16 cells per size class of the gradient gather.  Tolerances as in test_soft_gpu.py."""
import numpy as np
import pytest

from .test_soft_gpu import _case, _check, vq  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,H,W,D,k,th,tw,G", [
    (1, 38, 70, 33, 17, 15, 15, 2),      # 32 x 64 outputs of the smaller cell, 31 x 63 of the larger; scalar loads
    (2, 39, 71, 36, 33, 15, 14, 2),      # one more of each; one width, two heights; a chunk of four dimensions
    (1, 33, 65, 32, 8, 4, 5, 2),         # cells of two rows; two widths, one height
    (1, 40, 66, 64, 32, 12, 12, 2),      # one size class of four cells, the most centroids of the smallest tile
    (1, 41, 30, 4, 65, 13, 14, 3),       # 65 centroids; classes of four, two, two and one cells
    (1, 36, 34, 8, 5, 17, 16, 4),        # classes of twelve and four cells
    (1, 34, 33, 8, 5, 16, 16, 4),        # sixteen cells in one class
    (1, 130, 120, 4, 3, 100, 90, 1),     # box-sum tile too large for shared memory
    (1, 400, 12, 4, 2, 390, 5, 1),       # adjoint tile too large as well
])
def test_soft_tile_edges(vq, B, H, W, D, k, th, tw, G):  # noqa: F811
    # logit gaps of about 3 to 5, so that gradients stay well above FP32's range limits
    Q, T, C = _case(B, H, W, D, k, th, tw, seed=H * 100 + W, scale=float(np.sqrt(2.5 * 0.3 / D)))
    _check(vq, Q, T, C, 0.3, G, mask=True, delta=1e-5)
