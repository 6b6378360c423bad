"""The box-OR row pass with both radii 0 (one step of 32 pixels holds the window)
and with one of them 0, at widths around a step and every mask width.  Expected:
the maximum filter of the general test; masks are bits, so equality is exact."""
import numpy as np
import pytest

import oracle
from paper_2504_05148_gb300 import scenes
from paper_2504_05148_gb300 import sgmf as S
from test_boxor_gpu import _masks, _want

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,H,D", [(1, 1, 64), (31, 9, 128), (32, 8, 192), (33, 17, 256), (97, 40, 64)])
@pytest.mark.parametrize("rs,rc", [(0, 0), (0, 1), (1, 0)])
def test_radius_zero(gpu, W, H, D, rs, rc):
    s = scenes.random_small(9990 + W, W, H, D, density=0.1)
    box_s, box_c = _masks(s, S.Params(rs=rs, rc=rc))
    dbar = oracle.lidar(s.lidar, D)
    np.testing.assert_array_equal(box_s, _want(dbar, D, rs))
    np.testing.assert_array_equal(box_c, _want(dbar, D, rc))
