"""GPU test of the whole-row kernels (outputs that are rows of R consecutive
elements, folded by lanes teams): the bits of the batched executor, which folds
the same plan from its shared-memory ring.  Same per-lane order and same tree,
so the tolerance is zero."""
import numpy as np
import pytest

from paper_2309_01906_gb300 import binding as hb

pytestmark = pytest.mark.gpu

DT = {"f32": "float32", "f32_comp": "float32", "i32": "int32", "i64": "int32"}
OUT = {"f32": "float32", "f32_comp": "float32", "i32": "int32", "i64": "int64"}


def _compare(O, R, op, prec, body, level_map, offset):
    import torch
    g = torch.Generator("cuda").manual_seed(7 * O + R)
    dt = getattr(torch, DT[prec])
    if dt == torch.float32:
        A = torch.randn(O * R + offset, device="cuda", generator=g)
        w = torch.randn(R, device="cuda", generator=g)
    else:
        A = torch.randint(-(1 << 30), 1 << 30, (O * R + offset,), dtype=dt, device="cuda", generator=g)
        w = torch.randint(-1000, 1000, (R,), dtype=dt, device="cuda", generator=g)
    n = hb.Nest([O, R], 1, op, prec, body, level_map=level_map)
    if offset and n.describe()["vec"] == 4:
        n.close()
        return
    ins = [A.data_ptr() + 4 * offset] + ([w.data_ptr()] if body == "dot_bcast" else [])
    s = torch.cuda.current_stream().cuda_stream
    one = torch.full((O + 1,), 9, dtype=getattr(torch, OUT[prec]), device="cuda")
    many = torch.full_like(one, 9)
    n.run(ins, one.data_ptr(), s)
    hb.hp_nest_run_batch([n.handle], [ins], [many.data_ptr()], s)
    torch.cuda.synchronize()
    n.close()
    assert one[O] == 9 and torch.equal(one, many), (O, R, op, prec, body, level_map, offset)


# 5 and 32: the thread rows' range; 4, 33: just outside; 31, 63, 511, 1021: odd rows of each team width
ROWS = [1, 2, 4, 5, 8, 11, 12, 28, 31, 32, 33, 63, 64, 99, 100, 255, 511, 512, 1021, 4000]


@pytest.mark.parametrize("prec,op", [("f32", "sum"), ("f32_comp", "sum"), ("f32", "max"), ("i32", "sum"), ("i64", "min")])
@pytest.mark.parametrize("body", ["load", "dot_bcast"])
def test_rows_equal_the_batched_executor(prec, op, body):
    for R in ROWS:
        # 1, 33, 1000: rows one at a time; 150001: four at a time, with a ragged end
        for O in (1, 33, 1000, 150001 if R <= 100 else 20011):
            for offset in (0, 1):
                _compare(O, R, op, prec, body, None, offset)


@pytest.mark.parametrize("level_map", [["grid", "warp"], ["grid", ("subwarp", 2, 0)], ["grid", ("subwarp", 16, 0)],
                                       ["grid", "seq"], ["grid", ("lane", 4, 0)], ["warp", ("subwarp", 4, 0)]],
                         ids=str)
def test_explicit_lanes_teams(level_map):
    for R in (3, 20, 36, 301):
        for O in (5, 20011):
            _compare(O, R, "sum", "f32_comp", "dot_bcast", level_map, 0)


def test_residuals_of_the_rows_kernels():
    # out + comp is the two-word sum: comp is far below out's last place, and out is hp_nest_run's
    import torch
    for O, R in ((40, 300), (100003, 40), (100003, 20), (100003, 3)):
        A = torch.randn(O * R, device="cuda", generator=torch.Generator("cuda").manual_seed(R))
        n = hb.Nest([O, R], 1, "sum", "f32_comp", "load")
        out, comp = torch.empty(O, device="cuda"), torch.full((O,), float("nan"), device="cuda")
        s = torch.cuda.current_stream().cuda_stream
        n.run_comp([A.data_ptr()], out.data_ptr(), comp.data_ptr(), s)
        torch.cuda.synchronize()
        n.close()
        ref = A.view(O, R).double().sum(1)
        # Dot2: the two-word result errs by at most gamma_R^2 sum|t|
        lim = (R * 2.0 ** -24) ** 2 * 4 * A.view(O, R).abs().double().sum(1) + 1e-30
        assert torch.all((out.double() + comp.double() - ref).abs() <= lim)


@pytest.mark.parametrize("prec,op,body", [("f32", "sum", "load"), ("f32_comp", "sum", "dot_bcast"), ("i64", "max", "dot_bcast")])
def test_blocks_of_several_sets(prec, op, body):
    # enough rows that a warp's block holds several sets of 32; 160001: two, and a ragged last block
    for R in (4, 5, 7, 8, 11, 15):
        for O in (160001, 700003):
            _compare(O, R, op, prec, body, None, 0)
