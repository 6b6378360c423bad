"""Behind the sweep the rows are line walks and the winner kernel where a call
has few rows, the row kernel where it has many: frames of one to 260 rows in
calls on either side of the line (12 rows a SM), every lane width, a width of
one pixel and of no whole segment, sub-pixel output and each check.  Every
frame equals the oracle's."""
import numpy as np
import pytest

import oracle
from paper_2504_05148_gb300 import scenes
from paper_2504_05148_gb300 import sgmf as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,H,D,n,kw", [
    (37, 260, 64, 8, {}), (37, 260, 64, 2, {}),                     # many rows; few
    (41, 230, 100, 9, {"subpixel": 1}), (41, 23, 100, 9, {"subpixel": 1}),
    (30, 240, 192, 8, {"consistency": S.SGMF_CHECK_STEREO}), (30, 24, 192, 8, {"consistency": S.SGMF_CHECK_STEREO}),
    (26, 250, 256, 8, {"consistency": S.SGMF_CHECK_LIDAR}), (26, 25, 256, 8, {"consistency": S.SGMF_CHECK_LIDAR}),
    (1, 1, 16, 1, {}), (323, 3, 128, 3, {"consistency": S.SGMF_CHECK_NONE}),
])
def test_rows_behind_the_sweep(gpu, W, H, D, n, kw):
    import torch
    dev = torch.device("cuda:0")
    scs = [scenes.random_small(9950 + i + W, W, H, D) for i in range(n)]
    p = S.Params(**kw)
    ctx = S.Context(W, H, D, p, max_batch=n)
    try:
        S.sgmf_set_tuning(ctx.handle, 4, 128, 1)
        out = torch.empty((n, H, W), dtype=torch.int16, device=dev)
        l, r, li = (torch.from_numpy(np.stack([getattr(s, k) for s in scs])).to(dev) for k in ("left", "right", "lidar"))
        ctx.compute(l, r, li, out)
        ctx.sync()
        got = out.cpu().numpy()
    finally:
        ctx.close()
    for i, s in enumerate(scs):
        want = oracle.compute(s.left, s.right, s.lidar, s.D, oracle.Params(**vars(p)), dumps=False).out
        np.testing.assert_array_equal(got[i], want, err_msg=f"frame {i}")
