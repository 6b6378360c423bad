"""The work counts behind bench.py's roofline figures follow what the aggregation
stores: every vector, every second one, or the sweep's sums.  CPU only."""
import pytest

import bench
from paper_2504_05148_gb300 import sgmf
from test_abi import _int32_fields

V, N = 1000, 10


def _form(**kw):
    return {"sweep": 0, "row_walks": 1.0, "half_rows": 0, "half_lines": 0, "cost_bytes": 1, **kw}


def test_struct_matches_header():
    assert [f[0] for f in sgmf.sgmf_agg_form._fields_] == _int32_fields("sgmf_agg_form")


# (form, paths, bytes of the walks / of the winner kernel per cell, beside 4 N)
@pytest.mark.parametrize("form,paths,walks,winner", [
    (None, 8, 1 + 8, 8), (_form(), 4, 1 + 4, 4),
    (_form(half_rows=1, half_lines=1), 8, 1 + 4, 4 + 1), (_form(half_rows=1, half_lines=1), 4, 1 + 2, 2 + 1),
    (_form(half_rows=1, cost_bytes=2), 8, 1 + 2 + 12, 2 + 12 + 1),
    (_form(half_rows=1, half_lines=1, cost_bytes=2), 8, 1 + 8, 8 + 1),
    (_form(sweep=1), 8, 1 + 2, 2 + 4), (_form(sweep=1, half_rows=1, cost_bytes=2), 8, 1 + 2, 2 + 4 + 1)])
def test_bytes_follow_the_stored_vectors(form, paths, walks, winner):
    assert bench.algorithmic("agg_lines", V, N, paths, form)["bytes"] == walks * V
    assert bench.algorithmic("agg_rows_wta", V, N, paths, form)["bytes"] == winner * V + 4 * N


def test_every_direction_is_stepped_once():
    """Steps of Eq. 2 (8 operations a cell): the walks take all of them, the winner
    kernel again those whose vectors were left out, the row kernel the rows'."""
    for paths in (4, 8):
        assert bench.algorithmic("agg_lines", V, N, paths)["ops"] == 8 * paths * V
        full = bench.algorithmic("agg_rows_wta", V, N, paths)["ops"]
        half = bench.algorithmic("agg_rows_wta", V, N, paths, _form(half_rows=1, half_lines=1))["ops"]
        assert half - full == 8 * paths / 2 * V
    rows = bench.algorithmic("agg_rows_wta", V, N, 8, _form(sweep=1, row_walks=0.0))
    assert rows["bytes"] == 5 * V + 4 * N
    mixed = bench.algorithmic("agg_rows_wta", V, N, 8, _form(sweep=1, row_walks=0.25))
    wta = bench.algorithmic("agg_rows_wta", V, N, 8, _form(sweep=1))
    assert mixed["bytes"] == 0.25 * wta["bytes"] + 0.75 * rows["bytes"]
    assert bench.algorithmic("agg_lines", V, N, 8, _form(sweep=1, row_walks=0.25))["bytes"] == 0.25 * 3 * V
