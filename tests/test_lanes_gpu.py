"""The full-range aggregation kernels at the edges of their tiles: line walks
around the copy-ahead ring and its unrolled block (16 steps, 4 steps), four
lines a warp, row segments of the winner kernel (one CTA warp per 320 pixels,
four segments a warp), every lane width with the last disparity at either end
of a lane, byte and u16 path costs, four and eight paths.  Cost, S, d*, d' and
the output equal the oracle's bit for bit (whole numbers: no tolerance)."""
import numpy as np
import pytest

import oracle
from paper_2504_05148_gb300 import scenes
from paper_2504_05148_gb300 import sgmf as S

pytestmark = pytest.mark.gpu

# (W, H, D): H around 16 and 20 and W around the segment counts; D at the
# edges of the 8-, 16-, 24- and 32-cell lanes
SHAPES = [(319, 15, 57), (320, 16, 64), (321, 17, 65), (641, 19, 112), (5, 20, 113), (3, 37, 128), (78, 21, 168),
          (1, 33, 169), (1283, 5, 192), (47, 18, 193), (330, 20, 225), (13, 16, 256), (90, 1, 24), (1, 1, 256)]


def _check(scene, params, n=1):
    import torch
    dev = torch.device("cuda:0")
    ctx = S.Context(scene.W, scene.H, scene.D, params, max_batch=n)
    try:
        ctx.set_debug(True)
        rep = lambda a: torch.from_numpy(np.ascontiguousarray(np.stack([a] + [a[::-1]] * (n - 1)))).to(dev)
        out = torch.empty((n, scene.H, scene.W), dtype=torch.int16, device=dev)
        ctx.compute(rep(scene.left), rep(scene.right), rep(scene.lidar), out)
        ctx.sync()
        got = {"cost": ctx.stage(S.SGMF_STAGE_COST), "sum": ctx.stage(S.SGMF_STAGE_SUM),
               "dstar": ctx.stage(S.SGMF_STAGE_DSTAR), "dprime": ctx.stage(S.SGMF_STAGE_DPRIME)}
        outs = out.cpu().numpy()
    finally:
        ctx.close()
    o = oracle.compute(scene.left, scene.right, scene.lidar, scene.D, oracle.Params(**vars(params)), volumes=True)
    for k in ("cost", "sum", "dstar", "dprime"):
        np.testing.assert_array_equal(got[k].astype(np.int64), getattr(o, k).astype(np.int64), err_msg=k)
    np.testing.assert_array_equal(outs[0], o.out)
    for i in range(1, n):          # the frame upside down
        f = [np.ascontiguousarray(a[::-1]) for a in (scene.left, scene.right, scene.lidar)]
        np.testing.assert_array_equal(outs[i], oracle.compute(*f, scene.D, oracle.Params(**vars(params)),
                                                              dumps=False).out, err_msg=f"frame {i}")


@pytest.mark.parametrize("W,H,D", SHAPES)
@pytest.mark.parametrize("p2", [120, 300])
def test_line_and_winner_kernels(gpu, W, H, D, p2):
    _check(scenes.random_small(W * 11 + H * 5 + D, W, H, D), S.Params(p2=p2))


@pytest.mark.parametrize("params", [dict(num_paths=4), dict(subpixel=1), dict(consistency=S.SGMF_CHECK_STEREO),
                                    dict(consistency=S.SGMF_CHECK_LIDAR), dict(consistency=S.SGMF_CHECK_NONE),
                                    dict(num_paths=4, p2=300, subpixel=1)])
def test_winner_kernel_options(gpu, params):
    _check(scenes.random_small(771, 402, 23, 100), S.Params(**params), n=2)


# calls of at least 100 M cells (200 M with four paths) at Dp = 128 and 192: the
# walks store every second row's (column's) vectors.  Small frames in large
# batches put the parities and borders where they can go wrong: one row, two
# columns, odd and even sizes, segments that end on odd columns
@pytest.mark.parametrize("W,H,D,params", [
    (2, 100, 128, {}), (200, 1, 128, {}), (199, 2, 65, {}), (41, 40, 192, {}), (321, 7, 129, {}), (17, 33, 100, {}),
    (640, 9, 128, dict(subpixel=1)), (162, 15, 192, dict(num_paths=4)), (83, 24, 128, dict(num_paths=4)),
    (96, 31, 128, dict(consistency=S.SGMF_CHECK_LIDAR))])
def test_half_stored_vectors(gpu, W, H, D, params):
    import torch
    dev = torch.device("cuda:0")
    p = S.Params(**params)
    dp = 128 if D <= 128 else 192
    n = -(-(200_000_000 if p.num_paths == 4 else 100_000_000) // (W * H * dp))
    assert 3 <= n <= 4096
    scs = [scenes.random_small(8800 + i, W, H, D) for i in range(3)]
    rep = lambda name: torch.from_numpy(np.stack([getattr(s, name) for s in scs])).to(dev)[
        torch.arange(n, device=dev) % 3].contiguous()
    ctx = S.Context(W, H, D, p, max_batch=n)
    try:
        ctx.set_debug(True)
        out = torch.empty((n, H, W), dtype=torch.int16, device=dev)
        ctx.compute(rep("left"), rep("right"), rep("lidar"), out)
        ctx.sync()
        total = ctx.stage(S.SGMF_STAGE_SUM)
        dprime = ctx.stage(S.SGMF_STAGE_DPRIME)
        got = out.cpu().numpy()
    finally:
        ctx.close()
    for i, s in enumerate(scs):
        o = oracle.compute(s.left, s.right, s.lidar, D, oracle.Params(**vars(p)), volumes=i == 0)
        if i == 0:
            np.testing.assert_array_equal(total.astype(np.int64), o.sum.astype(np.int64))
            np.testing.assert_array_equal(dprime, o.dprime)
        assert (got[i::3] == o.out).all(), f"frame {i}"
