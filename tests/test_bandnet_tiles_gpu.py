"""The band network's tensor-core kernels at the edges of their tiles (128 pixels
of a row, three staged rows, several tiles a CTA through the three-stage ring):
forward, data gradient and weight gradient against the float64 reference.

Tolerance: products of two bf16 values are exact in f32; an output of the
weight gradient is at most (tiles a CTA) x 8 accumulations followed by 32 + 32
partial sums, an output of a convolution 18, each off by at most 2^-22 of the
sum of the terms' magnitudes: below 3e-5 of it in every case here.  Values
stored as bf16 add half a unit of 2^-8."""
import numpy as np
import pytest

from oracle import band_net as N
from paper_2504_05148_gb300 import sgmf as S
from test_bandnet_gpu import _Err, _bits, _dev, _from_bits, _pack, _rand_bf16

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,h,w", [(1, 1, 127), (2, 1, 128), (1, 3, 129), (1, 2, 257), (4, 100, 130), (7, 61, 1)])
def test_layer_at_tile_edges(gpu, n, h, w):
    import torch
    rng = np.random.default_rng(n + 10 * h + 1000 * w)
    x = N.bf16_round(np.maximum(rng.normal(size=(n, h, w, 32)), 0.0))
    dy = _rand_bf16(rng, (n, h, w, 32), 0.1)
    wt = _rand_bf16(rng, (32, 3, 3, 32), 0.1)
    b = rng.normal(size=32).astype(np.float32)
    pf, pd = _pack(wt)
    xd, dyd, bd = _dev(_bits(x)), _dev(_bits(dy)), _dev(b)
    y = torch.empty((n, h, w, 32), dtype=torch.float32, device="cuda")
    dx = torch.empty((n, h, w, 32), dtype=torch.int16, device="cuda")
    dw = torch.ones(32 * 288, dtype=torch.float32, device="cuda")     # accumulated into
    db = torch.ones(32, dtype=torch.float32, device="cuda")
    err = _Err()
    S.sgmf_bn_conv(n, h, w, xd.data_ptr(), pf.data_ptr(), bd.data_ptr(), True, None, None, y.data_ptr(), err.ptr)
    S.sgmf_bn_wgrad(n, h, w, xd.data_ptr(), dyd.data_ptr(), dw.data_ptr(), db.data_ptr(), err.ptr)
    S.sgmf_bn_conv(n, h, w, dyd.data_ptr(), pd.data_ptr(), None, False, xd.data_ptr(), dx.data_ptr(), None, err.ptr)
    err.check()
    b64 = b.astype(np.float64)
    ref = np.maximum(N.conv3x3(x, wt, b64), 0.0)
    scale = N.conv3x3(np.abs(x), np.abs(wt), np.abs(b64))
    assert (np.abs(y.cpu().numpy() - ref) <= 3e-5 * scale).all()
    rw, rb = N.conv3x3_wgrad(x, dy)
    sw, sb = N.conv3x3_wgrad(np.abs(x), np.abs(dy))
    assert (np.abs(dw.cpu().numpy().reshape(rw.shape) - 1.0 - rw) <= 3e-5 * (sw + 1.0)).all()
    assert (np.abs(db.cpu().numpy() - 1.0 - rb) <= 3e-5 * (sb + 1.0)).all()
    # the data gradient, zero where x is not positive
    rx = np.where(x > 0, N.conv3x3_dgrad(dy, wt), 0.0)
    sx = N.conv3x3_dgrad(np.abs(dy), np.abs(wt))
    got = _from_bits(dx.cpu().numpy().view(np.uint16))
    assert (np.abs(got - rx) <= 3e-5 * sx + 2.0 ** -8 * np.abs(rx)).all()
