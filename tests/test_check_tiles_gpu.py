"""The check kernel's tiles and its list of the pixels that the LiDAR term
decides: frames at, below and above a tile (32 x 32), a list that holds every
pixel (LiDAR alone), some and none, and the output written over d*.  Whole
numbers, so the result equals the definition of Eq. 6 exactly."""
import numpy as np
import pytest

from paper_2504_05148_gb300 import sgmf as S

pytestmark = pytest.mark.gpu


def _want(ds, dp, lidar, p, D):
    H, W = ds.shape
    out = np.full((H, W), -1, np.int16)
    ld = np.where((lidar > 0) & (lidar < D - 0.5), np.rint(lidar), -1).astype(int)
    for y in range(H):
        for x in range(W):
            d = int(ds[y, x])
            st = x - d >= 0 and abs(d - int(dp[y, x - d])) <= p.lr_max_diff
            w = ld[max(y - p.rc, 0):y + p.rc + 1, max(x - p.rc, 0):x + p.rc + 1]
            li = bool(((w >= 0) & (np.abs(w - d) <= p.tc)).any())
            ok = {S.SGMF_CHECK_STEREO_LIDAR: st or li, S.SGMF_CHECK_STEREO: st, S.SGMF_CHECK_LIDAR: li,
                  S.SGMF_CHECK_NONE: True}[p.consistency]
            if ok:
                out[y, x] = d
    return out


@pytest.mark.parametrize("W,H", [(1, 1), (31, 33), (32, 32), (33, 65), (97, 31), (3, 70)])
def test_check_tiles(gpu, W, H):
    import torch
    dev = torch.device("cuda:0")
    D = 64
    rng = np.random.default_rng(W * 100 + H)
    ds = rng.integers(0, D, (H, W)).astype(np.int16)
    dp = rng.integers(0, D, (H, W)).astype(np.int16)
    near = rng.random((H, W)) < 0.5                  # half of the pixels pass the stereo term, where it exists
    for y, x in np.argwhere(near):
        if x - ds[y, x] >= 0:
            dp[y, x - ds[y, x]] = ds[y, x]
    lidar = np.where(rng.random((H, W)) < 0.1, rng.integers(0, D, (H, W)), -1).astype(np.float32)
    for mode in (S.SGMF_CHECK_STEREO_LIDAR, S.SGMF_CHECK_STEREO, S.SGMF_CHECK_LIDAR, S.SGMF_CHECK_NONE):
        for rc in (2, 11):
            p = S.Params(consistency=mode, rc=rc)
            want = _want(ds, dp, lidar, p, D)
            a, b, li = (torch.from_numpy(v).to(dev) for v in (ds, dp, lidar))
            out = torch.full((H, W), 12345, dtype=torch.int16, device=dev)
            for o in (out, a):                       # apart, then in place over d*
                S.sgmf_check_static(W, H, D, p, a.data_ptr(), b.data_ptr(), li.data_ptr(), o.data_ptr(), None)
                torch.cuda.synchronize()
                np.testing.assert_array_equal(o.cpu().numpy(), want, err_msg=f"mode {mode}, rc {rc}")
