"""The kernel that hp_nest_describe names: the launch asks the same questions, so the
table here is of the shapes where they divide.  No GPU."""
import pytest

from paper_2309_01906_gb300 import binding as hb

GRID_CTA = ["grid", "cta"]


@pytest.mark.parametrize("ext,op,prec,body,level_map,kernel", [
    ([1000, 100], "sum", "f32", "load", None, "rect_rows"),
    ([1000, 1021], "sum", "f32_comp", "dot_bcast", None, "rect_rows"),
    ([1000, 31], "sum", "f32", "load", None, "rect_thread_rows"),
    ([1000, 63], "max", "i32", "load", None, "rect_thread_rows"),
    ([1000, 5], "sum", "i64", "dot_bcast", None, "rect_thread_rows"),
    ([1000, 4], "sum", "f32", "load", None, "rect_rows"),
    ([1000, 4], "sum", "f32_comp", "dot_bcast", None, "rect_thread_rows"),
    ([1000, 16], "sum", "f32", "load", None, "rect_lanes"),
    ([1000, 100], "sum", "i64", "affine", None, "rect_lanes"),
    ([1000, 8195], "sum", "i64", "load", None, "rect_flat"),
    ([1, 1 << 20], "sum", "f32_comp", "dot_bcast", None, "rect_flat"),
    ([700, 4092], "sum", "f32", "load", GRID_CTA, "rect_block_pipe"),
    ([700, 4096], "sum", "f32", "load", GRID_CTA, "rect_flat"),
    ([700, 4096], "max", "i64", "load", GRID_CTA, "rect_block_pipe"),
    ([700, 4096], "sum", "f32", "dot_bcast", GRID_CTA, "rect_block_pipe"),
    ([700, 65536], "sum", "f32", "dot_bcast", GRID_CTA, "rect_flat"),
    ([700, 5001], "sum", "f32", "load", ["grid", ("cta", 16, 0)], "rect_block"),
    ([700, 8, 8192], "sum", "f32", "load", ["grid", ("cluster", 4, 0), "cta"], "rect_block_cluster"),
])
def test_rectangular(ext, op, prec, body, level_map, kernel):
    params = hb.hp_affine_params(3, 5, 7) if body == "affine" else None
    n = hb.Nest(ext, 1, op, prec, body, level_map=level_map, params=params)
    assert n.describe()["kernel"] == kernel
    n.close()


@pytest.mark.parametrize("ext,prec,body,level_map,kernel", [
    ([1000, 64], "i8", "load", None, "narrow_warp"), ([20000, 64], "i8", "load", None, "narrow_rows"),
    ([3040, 16], "i8", "load", None, "narrow_warp"), ([3041, 16], "i8", "load", None, "narrow_rows"),
    ([1000, 100], "i8", "dot_bcast", None, "narrow_elements"), ([100000, 100], "i8", "dot_bcast", None, "narrow_rows"),
    ([1000, 777], "i8", "load", None, "narrow_warp"), ([100000, 777], "i8", "load", None, "narrow_rows"),
    ([1000, 777], "i16", "load", None, "narrow_warp"), ([100000, 777], "i16", "load", None, "narrow_warp"),
    ([100, 65536], "i16", "load", GRID_CTA, "narrow_block"),
])
def test_narrow(ext, prec, body, level_map, kernel):
    n = hb.Nest(ext, 1, "sum", prec, body, level_map=level_map)
    assert n.describe()["kernel"] == kernel
    n.close()


@pytest.mark.parametrize("op,ext,kernel", [
    ("compose", [100, 7], "ordered_short"), ("compose", [1000, 31], "ordered_warp"), ("compose", [10000, 31], "ordered_short"),
    ("mat2", [1000, 64], "ordered_warp"), ("mat2", [10000, 64], "ordered_short"), ("last", [10000, 256], "ordered_short"),
    ("last", [30000, 500], "ordered_warp"), ("last", [30000, 1001], "ordered_warp"), ("compose", [4, 1 << 20], "ordered_block"),
])
def test_ordered(op, ext, kernel):
    n = hb.Nest(ext, 1, op, "f32", "load")
    assert n.describe()["kernel"] == kernel
    n.close()
