"""u16 path costs (P2 + the largest cost above 255): the line walks leave the
rows' vectors of odd columns out, in large calls those of odd rows too, and the
winner kernel takes their steps, on the bands across tile edges.  Frames of one
and two columns and rows, odd and even sizes, every lane width with the last
disparity at either end of a lane, P2 at its largest, calls on both sides of the
line in cells; behind the sweep, rows on both sides of the line in columns.
Whole numbers: everything equals the oracle."""
import numpy as np
import pytest

import oracle
from paper_2504_05148_gb300 import scenes
from paper_2504_05148_gb300 import sgmf as S

pytestmark = pytest.mark.gpu


def _run(W, H, D, n, p, band=0, sweep=False, distinct=3, seed=0):
    import torch
    dev = torch.device("cuda:0")
    k = min(n, distinct)
    scs = [scenes.random_small(7000 + seed + i, W, H, D) for i in range(k)]
    pick = torch.arange(n, device=dev) % k
    rep = lambda arrs: torch.from_numpy(np.stack(arrs)).to(dev)[pick].contiguous()
    th, tw = (H + S.BAND_TILE - 1) // S.BAND_TILE, (W + S.BAND_TILE - 1) // S.BAND_TILE
    rng = np.random.default_rng(W + H + D + seed)
    los = [rng.integers(0, D - band + 1, size=(th, tw)).astype(np.int16) for _ in scs] if band else None
    ctx = S.Context(W, H, D, p, max_batch=n, band=band)
    try:
        if sweep:
            S.sgmf_set_tuning(ctx.handle, 4, 128, 1)
        ctx.set_debug(True)
        out = torch.full((n, H, W), -7, dtype=torch.int16, device=dev)
        ins = [rep([getattr(s, a) for s in scs]) for a in ("left", "right", "lidar")]
        if band:
            ctx.compute_banded(*ins, rep(los), out)
        else:
            ctx.compute(*ins, out)
        ctx.sync()
        total, dprime = ctx.stage(S.SGMF_STAGE_SUM), ctx.stage(S.SGMF_STAGE_DPRIME)
        got = out.cpu().numpy()
    finally:
        ctx.close()
    for i, s in enumerate(scs):
        op = oracle.Params(**vars(p))
        if band:
            lo = oracle.expand_tiles(los[i], W, H, S.BAND_TILE)
            o = oracle.compute_banded(s.left, s.right, s.lidar, D, band, lo, op, volumes=i == 0)
        else:
            o = oracle.compute(s.left, s.right, s.lidar, D, op, volumes=i == 0)
        if i == 0:
            want = o.sum
            if band:
                want = np.take_along_axis(want, lo[:, :, None].astype(np.int64) + np.arange(band), axis=2)
            np.testing.assert_array_equal(total.astype(np.int64), want[:, :, :total.shape[2]].astype(np.int64))
            np.testing.assert_array_equal(dprime, o.dprime)
        assert (got[i::k] == o.out).all(), f"frame {i}"


def _frames(cells, W, H, D, band=0):
    dp = band or (64 if D <= 64 else 128 if D <= 128 else 192 if D <= 192 else 256)
    n = -(-cells // (W * H * dp))
    assert 3 <= n <= 4096
    return n


@pytest.mark.parametrize("W,H,D", [(1, 1, 64), (2, 2, 50), (1, 9, 128), (9, 1, 100), (2, 5, 192), (3, 3, 256), (640, 3, 65),
                                   (641, 2, 193), (322, 7, 129)])
@pytest.mark.parametrize("p2", [300, 2048])
def test_small_calls(gpu, W, H, D, p2):
    _run(W, H, D, 2, S.Params(p2=p2))


# eight paths from 25 M cells, four from 50 M
@pytest.mark.parametrize("W,H,D,kw", [
    (2, 200, 64, {}), (201, 1, 57, {}), (99, 2, 128, {}), (64, 33, 100, {}), (1, 130, 192, {}), (41, 40, 169, {}),
    (33, 16, 256, {}), (322, 7, 225, {}), (130, 31, 64, dict(subpixel=1)), (83, 24, 128, dict(num_paths=4)),
    (50, 21, 64, dict(num_paths=4)), (57, 30, 192, dict(num_paths=4)), (60, 29, 250, dict(num_paths=4)),
    (96, 31, 128, dict(consistency=S.SGMF_CHECK_LIDAR, p2=2048))])
def test_large_calls(gpu, W, H, D, kw):
    p = S.Params(**{"p2": 300, **kw})
    _run(W, H, D, _frames(50_000_000 if p.num_paths == 4 else 25_000_000, W, H, D), p, seed=100)


# bands: small calls, and from 100 M cells
@pytest.mark.parametrize("W,H,D,band", [(130, 40, 256, 64), (65, 17, 128, 128), (7, 9, 128, 64), (25, 1, 100, 64), (1, 26, 200, 128)])
@pytest.mark.parametrize("large", [False, True])
@pytest.mark.parametrize("kw", [{}, dict(num_paths=4)])
def test_bands(gpu, W, H, D, band, large, kw):
    if large and W * H < 400:
        W, H = 8 * W + 3, 8 * H + 1
    n = _frames(100_000_000, W, H, D, band) if large else 2
    _run(W, H, D, n, S.Params(p2=300, **kw), band=band, seed=200)


# rows of 700 columns and more as line walks, shorter ones by the row kernel
@pytest.mark.parametrize("W,D", [(699, 64), (700, 64), (701, 100), (902, 192), (1203, 256)])
@pytest.mark.parametrize("kw", [{}, dict(subpixel=1, consistency=S.SGMF_CHECK_STEREO)])
def test_rows_behind_the_sweep(gpu, W, D, kw):
    _run(W, 11, D, 2, S.Params(p2=300, **kw), sweep=True, seed=300)
