"""The row kernel and the check kernel behind the sweep (calls of more than 12 rows
a SM): rows wider than the disparity range, so that slots leave on the way, at every
lane width with the last disparity at the end of a lane and before it, byte and u16
path costs, odd and even widths, with and without the sub-pixel fit; and a batch in
parts whose first part takes them.  Everything equals the oracle; the kernel times
show that these kernels ran."""
import numpy as np
import pytest

import oracle
from paper_2504_05148_gb300 import scenes
from paper_2504_05148_gb300 import sgmf as S

pytestmark = pytest.mark.gpu


def _scenes(W, H, D, n, seed, distinct=3):
    import torch
    dev = torch.device("cuda:0")
    scs = [scenes.random_small(seed + i, W, H, D) for i in range(distinct)]
    pick = torch.arange(n, device=dev) % distinct
    return scs, [torch.from_numpy(np.stack([getattr(s, a) for s in scs])).to(dev)[pick].contiguous()
                 for a in ("left", "right", "lidar")]


@pytest.mark.parametrize("W,D", [(300, 64), (301, 50), (150, 33), (300, 128), (301, 100), (257, 65), (300, 192), (301, 170),
                                 (320, 256), (259, 200), (400, 16)])
@pytest.mark.parametrize("kw", [{}, {"subpixel": 1}, {"p2": 300}, {"p2": 300, "subpixel": 1}])
def test_rows_wider_than_the_range(gpu, W, D, kw):
    import torch
    H, n, p = 40, 64, S.Params(**kw)
    assert H * n > 12 * torch.cuda.get_device_properties(0).multi_processor_count
    scs, ins = _scenes(W, H, D, n, 3000 + W + D)
    ctx = S.Context(W, H, D, p, max_batch=n)
    try:
        S.sgmf_set_tuning(ctx.handle, 4, 128, 1, 0)          # one launch a kernel for the whole batch
        ctx.set_debug(True)
        ctx.set_profiling(True)
        out = torch.full((n, H, W), -7, dtype=torch.int16, device="cuda")
        ctx.compute(*ins, out)
        ctx.sync()
        names = [name for name, _ in ctx.kernel_times()]
        maps = {"sum": S.SGMF_STAGE_SUM, "dstar": S.SGMF_STAGE_DSTAR, "dprime": S.SGMF_STAGE_DPRIME}
        if p.subpixel:
            maps["dsub"] = S.SGMF_STAGE_DSUB
        maps = {k: ctx.stage(v) for k, v in maps.items()}
        got = out.cpu().numpy()
    finally:
        ctx.close()
    assert "consistency" in names and "agg_lines" not in names
    for i, s in enumerate(scs):
        o = oracle.compute(s.left, s.right, s.lidar, D, oracle.Params(**vars(p)), volumes=i == 0)
        if i == 0:
            for k, v in maps.items():
                want = oracle.subpixel(o.sum, o.dstar) if k == "dsub" else getattr(o, k)
                np.testing.assert_array_equal(v.astype(np.int64), want.astype(np.int64), err_msg=k)
        assert (got[i::3] == o.out).all(), f"frame {i}"


@pytest.mark.parametrize("kw", [{}, {"p2": 300, "subpixel": 1}])
def test_parts_by_the_row_kernel(gpu, kw):
    """16 frames of 1242 x 150: a first part of whole sweep waves, whose rows are the
    row kernel's on the second stream, and the rest, whose few rows are walks."""
    import torch
    W, H, D, n, p = 1242, 150, 128, 16, S.Params(**kw)
    scs, ins = _scenes(W, H, D, n, 4100)
    ctx = S.Context(W, H, D, p, max_batch=n)
    try:
        ctx.set_profiling(True)
        got = []
        for parts in (1, 1, 0):                              # twice: the events and the second stream are reused
            S.sgmf_set_tuning(ctx.handle, 4, 128, 1, parts)
            out = torch.full((n, H, W), -7, dtype=torch.int16, device="cuda")
            ctx.compute(*ins, out)
            ctx.sync()
            got.append(out.cpu().numpy())
            names = [name for name, _ in ctx.kernel_times()]
            assert "consistency" in names and ("agg_lines" in names) == bool(parts)
    finally:
        ctx.close()
    for i, s in enumerate(scs):
        want = oracle.compute(s.left, s.right, s.lidar, D, oracle.Params(**vars(p)), dumps=False).out
        for g in got:
            assert (g[i::3] == want).all(), f"frame {i}"
