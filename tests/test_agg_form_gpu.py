"""sgmf_get_agg_form against the kernels that a call launches, and its flags on both
sides of the lines that they follow."""
import pytest

from paper_2504_05148_gb300 import scenes
from paper_2504_05148_gb300 import sgmf as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,H,D,n,kw,sweep", [
    (64, 40, 64, 2, {}, 0), (301, 40, 100, 64, {}, 1), (301, 40, 100, 2, {}, 1), (301, 40, 100, 2, {"p2": 300}, 1),
    (800, 20, 64, 2, {"p2": 300}, 1), (1242, 150, 128, 16, {}, 1), (200, 100, 128, 45, {}, 0), (200, 100, 128, 8, {"p2": 300}, 0),
    (200, 100, 128, 10, {"p2": 300}, 0), (200, 100, 128, 45, {"num_paths": 4}, 0), (200, 100, 128, 10, {"num_paths": 4}, 1)])
def test_form_is_what_runs(gpu, W, H, D, n, kw, sweep):
    import torch
    p = S.Params(**kw)
    s = scenes.random_small(5, W, H, D)
    ins = [torch.from_numpy(a).cuda().expand(n, H, W).contiguous() for a in (s.left, s.right, s.lidar)]
    ctx = S.Context(W, H, D, p, max_batch=n)
    try:
        S.sgmf_set_tuning(ctx.handle, 4, 128, sweep)
        ctx.set_profiling(True)
        ctx.compute(*ins, torch.empty((n, H, W), dtype=torch.int16, device="cuda"))
        ctx.sync()
        names = {name for name, _ in ctx.kernel_times()}
        f = S.sgmf_get_agg_form(ctx.handle, n)
        for bad in (0, n + 1):
            with pytest.raises(S.SgmfError):
                S.sgmf_get_agg_form(ctx.handle, bad)
    finally:
        ctx.close()
    assert f.sweep == ("agg_sweep" in names) == (sweep == 1 and p.num_paths == 8)
    assert (f.row_walks > 0) == ("agg_lines" in names) and (f.row_walks < n) == ("consistency" in names)
    u16 = p.p2 == 300
    cells = n * W * H * (64 if D <= 64 else 128)
    assert f.cost_bytes == 1 + u16 and f.half_rows == (u16 or f.half_lines)
    line = (25e6 if u16 else 100e6) if p.num_paths == 8 else (50e6 if u16 else 200e6)
    assert f.half_lines == (not f.sweep and cells >= line)
