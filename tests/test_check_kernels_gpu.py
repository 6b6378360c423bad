"""The check's two kernels, a thread per pixel and the list, on either side of the
rule that picks one: few and many tiles of 32 x 32, a window of few rows and of
more, the LiDAR term alone (the list then holds every pixel) and with the stereo
term; the output apart and in place over d*.  Whole numbers, so the result equals
the definition of Eq. 6 exactly."""
import numpy as np
import pytest

from paper_2504_05148_gb300 import sgmf as S

pytestmark = pytest.mark.gpu


def _want(ds, dp, ld, p, D):
    from scipy.ndimage import maximum_filter
    H, W = ds.shape
    xm = np.arange(W)[None, :] - ds
    dm = np.take_along_axis(dp.astype(int), np.maximum(xm, 0), axis=1)
    stereo = (xm >= 0) & (np.abs(ds - dm) <= p.lr_max_diff)
    lidar = np.zeros((H, W), bool)
    for d in range(D):
        near = maximum_filter(ld == d, size=2 * p.rc + 1, mode="constant", cval=0)
        lidar |= near & (np.abs(ds - d) <= p.tc)
    ok = {S.SGMF_CHECK_STEREO_LIDAR: stereo | lidar, S.SGMF_CHECK_STEREO: stereo, S.SGMF_CHECK_LIDAR: lidar,
          S.SGMF_CHECK_NONE: np.ones((H, W), bool)}[p.consistency]
    return np.where(ok, ds, -1).astype(np.int16)


@pytest.mark.parametrize("W,H", [(1281, 993), (70, 45)])
@pytest.mark.parametrize("rc", [0, 1, 4, 5])
def test_check_kernels(gpu, W, H, rc):
    import torch
    dev = torch.device("cuda:0")
    D = 64
    rng = np.random.default_rng(W + rc)
    ds = rng.integers(0, D, (H, W)).astype(np.int16)
    dp = rng.integers(0, D, (H, W)).astype(np.int16)
    xm = np.arange(W)[None, :] - ds
    y, x = np.nonzero((xm >= 0) & (rng.random((H, W)) < 0.5))   # half of the pixels pass the stereo term, where it exists
    dp[y, xm[y, x]] = ds[y, x]
    lidar = np.where(rng.random((H, W)) < 0.1, rng.integers(0, D, (H, W)), -1).astype(np.float32)
    ld = np.where((lidar > 0) & (lidar < D - 0.5), np.rint(lidar), -1).astype(int)
    for mode in (S.SGMF_CHECK_STEREO_LIDAR, S.SGMF_CHECK_STEREO, S.SGMF_CHECK_LIDAR, S.SGMF_CHECK_NONE):
        p = S.Params(consistency=mode, rc=rc)
        want = _want(ds, dp, ld, p, D)
        a, b, li = (torch.from_numpy(v).to(dev) for v in (ds, dp, lidar))
        out = torch.full((H, W), 12345, dtype=torch.int16, device=dev)
        for o in (out, a):                               # apart, then in place over d*
            S.sgmf_check_static(W, H, D, p, a.data_ptr(), b.data_ptr(), li.data_ptr(), o.data_ptr(), None)
            torch.cuda.synchronize()
            np.testing.assert_array_equal(o.cpu().numpy(), want, err_msg=f"mode {mode}")
