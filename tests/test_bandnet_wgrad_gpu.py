"""The weight gradient where its tiles end: infinities and NaN beside the ends of
a row; rows of up to 16 pixels, four to a stage; and calls in which every stage
of a CTA's three-stage ring is refilled several times (the other tests give a
CTA at most three tiles)."""
import numpy as np
import pytest

from oracle import band_net as N
from paper_2504_05148_gb300 import sgmf as S
from test_bandnet_gpu import _Err, _bits, _dev, _rand_bf16

pytestmark = pytest.mark.gpu


def _wgrad(n, h, w, xd, dyd):
    import torch
    dw = torch.zeros(32 * 288, dtype=torch.float32, device="cuda")
    db = torch.zeros(32, dtype=torch.float32, device="cuda")
    err = _Err()
    S.sgmf_bn_wgrad(n, h, w, xd.data_ptr(), dyd.data_ptr(), dw.data_ptr(), db.data_ptr(), err.ptr)
    err.check()
    return dw.cpu().numpy().reshape(32, 3, 3, 32), db.cpu().numpy()


@pytest.mark.parametrize("w", [1, 5, 15, 16, 17, 100, 127, 128, 129, 143, 144, 145, 311])
def test_non_finite_activations_reach_their_own_taps_only(gpu, w):
    """An activation that is no finite number makes the taps that multiply it
    with an output gradient non-finite, and no others: column 0 has no part in
    kx = 2, the last column none in kx = 0.  The finite entries differ from the
    reference by f32 accumulation only (test_bandnet_tiles_gpu.py)."""
    n, h = 2, 4
    rng = np.random.default_rng(77 + w)
    x = _rand_bf16(rng, (n, h, w, 32))
    dy = _rand_bf16(rng, (n, h, w, 32), 0.1)
    dy[dy == 0] = 0.125
    clean = x.copy()
    # one odd value a channel: the row's ends, its first row's and last row's, and a tile's ends
    for c, (img, y, px, v) in enumerate([(0, 1, w - 1, np.inf), (1, 2, w - 1, np.nan), (0, 2, 0, -np.inf),
                                         (1, 0, 0, np.nan), (0, 0, w - 1, -np.inf), (1, h - 1, w - 1, np.inf),
                                         (1, 1, min(127, w - 1), np.inf), (0, 1, min(128, w - 1), np.nan)]):
        x[img, y, px, c] = v
        clean[img, y, px, c] = 0.0
    dw, db = _wgrad(n, h, w, _dev(_bits(x)), _dev(_bits(dy)))
    with np.errstate(invalid="ignore"):
        rw, rb = N.conv3x3_wgrad(x, dy)
    np.testing.assert_array_equal(np.isfinite(dw), np.isfinite(rw))
    np.testing.assert_array_equal(np.isnan(dw), np.isnan(rw))
    inf = np.isinf(rw)
    np.testing.assert_array_equal(dw[inf], rw[inf])
    fin = np.isfinite(rw)
    sw, _ = N.conv3x3_wgrad(np.abs(clean), np.abs(dy))
    assert (np.abs(dw[fin] - rw[fin]) <= 3e-5 * (sw[fin] + 1e-30)).all()
    assert np.isfinite(db).all()


@pytest.mark.parametrize("n,h,w", [(16, 120, 130), (16, 76, 17), (11, 113, 140), (16, 270, 9), (15, 241, 16), (3, 1, 1),
                                   (5, 2, 3), (16, 400, 1)])
def test_ring_refilled(gpu, n, h, w):
    """13, 4 and 9 tiles a CTA (the third with a shorter last CTA); rows of up to 16
    pixels: 4, 3, 1, 1 and 6 stages of four rows, the last one of the call full or
    not.  An entry is at most 13 x 8 accumulations and 10 + 31 partial sums, each
    off by at most 2^-22 of the terms' magnitudes: 4e-5.  The order of the sums is
    fixed, so that a second call gives the same bits."""
    rng = np.random.default_rng(n + h + w)
    x = N.bf16_round(np.maximum(rng.normal(size=(n, h, w, 32)), 0.0))
    dy = _rand_bf16(rng, (n, h, w, 32), 0.1)
    xd, dyd = _dev(_bits(x)), _dev(_bits(dy))
    dw, db = _wgrad(n, h, w, xd, dyd)
    rw, rb = N.conv3x3_wgrad(x, dy)
    sw, sb = N.conv3x3_wgrad(np.abs(x), np.abs(dy))
    assert (np.abs(dw - rw) <= 4e-5 * sw).all()
    assert (np.abs(db - rb) <= 4e-5 * sb).all()
    again, dagain = _wgrad(n, h, w, xd, dyd)
    np.testing.assert_array_equal(again, dw)
    np.testing.assert_array_equal(dagain, db)
