"""The in-order FP64 column sums of the Lloyd update, 64 members at a time: bit-identical to the
oracle where groups are exact, where single values round, and where the running sum crosses a
power of two with its lowest bits in use."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def vq():
    from paper_2306_15010_gb300 import build
    build.build()
    import paper_2306_15010_gb300 as m
    torch.cuda.set_device(0)
    return m


@pytest.mark.parametrize("kind", ["tiny", "fine_bits", "signs", "wide", "zeros", "special_range"])
@pytest.mark.parametrize("l", [63, 64, 65, 129, 1500, 9001])
def test_in_order_sums_bit_exact(vq, l, kind):
    r = np.random.default_rng(l + len(kind))
    D, k = 36, 1                                             # the second 32 columns ragged
    T = r.uniform(0.0, 1.0, (l, D)).astype(np.float32)
    if kind == "tiny":                                       # a few values below the last place of the sum
        T[r.random((l, D)) < 0.01] = np.float32(3e-13)
        T[r.random((l, D)) < 0.01] *= np.float32(2.0 ** -22)
    elif kind == "fine_bits":                                # every value uses bits far below 2^-40
        T = (T * 2.0 ** -12).astype(np.float32)
        T[::50] += np.float32(1.7)
    elif kind == "signs":
        T[r.random((l, D)) < 0.5] *= -1
        T[r.random((l, D)) < 0.02] *= np.float32(2.0 ** -25)
    elif kind == "wide":                                     # outside the 64-bit group sums' range
        T[r.random((l, D)) < 0.02] = np.float32(123.75)
        T[r.random((l, D)) < 0.02] = np.float32(2.0 ** -40)
    elif kind == "zeros":
        T[:] = 0
        T[l // 2] = np.float32(2.0 ** -30)
        T[-1, ::2] = -0.0
    else:                                                    # at the ends of that range, 2^-27 and 2^6
        T[r.random((l, D)) < 0.1] = np.float32(2.0 ** -27)
        T[r.random((l, D)) < 0.1] = np.nextafter(np.float32(64), np.float32(0))
        T[r.random((l, D)) < 0.01] = np.nextafter(np.float32(2.0 ** -27), np.float32(0))
    T = T.reshape(1, l, D)
    ref = oracle.fit_codebook(T, k, 1, 3)
    got = vq.vqnnf_fit_codebook(torch.as_tensor(T).cuda(), k, 1, 3, "fp32").cpu().numpy()
    assert np.array_equal(got.view(np.uint32), np.asarray(ref, np.float32).view(np.uint32))
