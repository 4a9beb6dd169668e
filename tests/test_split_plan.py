"""Where the planner splits rows over the grid: fewer than two outputs per SM, and rows
of at least 65536 iterations.  More outputs need no scratch, so they run at any
scratch or memory budget, alone, batched and served."""
import pytest

from paper_2309_01906_gb300 import binding as hb


@pytest.mark.parametrize("O,split", [(1, True), (200, True), (303, True), (304, False), (500, False), (1823, False), (1824, False)])
@pytest.mark.parametrize("prec,body", [("f32", "load"), ("f32_comp", "dot_bcast"), ("i64", "affine")])
def test_two_outputs_per_sm_are_not_split(O, split, prec, body):
    params = hb.hp_affine_params(3, 5, 7) if body == "affine" else None
    for ext in ([O, 65536], [O, 65537], [O, 16, 300000]):
        n = hb.Nest(ext, 1, "sum", prec, body, params=params)
        d = n.describe()
        n.close()
        assert (d["grid_parts"] > 1) == split and d["team"] == "block", (ext, d)
