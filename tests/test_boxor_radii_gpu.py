"""The column pass by registers (radii up to 8) and its line to the ring (9),
at frames of one, part of one, exactly one, and two row segments and more, one
column past a block, and a row pass over one, three and four chunks of pixels
(radii 0, 20 and 33).  Expected: the maximum filter of the general test; masks
are bits, so equality is exact."""
import numpy as np
import pytest

import oracle
from paper_2504_05148_gb300 import scenes
from paper_2504_05148_gb300 import sgmf as S
from test_boxor_gpu import _masks, _want

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rs", range(10))
def test_column_pass_radii(gpu, rs):
    for i, (W, H, D, rc) in enumerate([(129, 32, 64, 0), (40, 33, 128, 20), (130, 7, 192, 33), (31, 81, 256, 8)]):
        s = scenes.random_small(9900 + 10 * rs + i, W, H, D, density=0.04)
        box_s, box_c = _masks(s, S.Params(rs=rs, rc=rc))
        dbar = oracle.lidar(s.lidar, D)
        np.testing.assert_array_equal(box_s, _want(dbar, D, rs), err_msg=f"{W} x {H}, r_s")
        np.testing.assert_array_equal(box_c, _want(dbar, D, rc), err_msg=f"{W} x {H}, r_c")
