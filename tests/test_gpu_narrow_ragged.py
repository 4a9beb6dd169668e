"""GPU test of 8- and 16-bit nests whose rows are short or start off 16-byte
boundaries: whole pieces between single loads, several short rows per warp, and
a broadcast operand at any alignment, bit for bit against 64-bit integer sums."""
import numpy as np
import pytest

from paper_2309_01906_gb300 import binding as hb

pytestmark = pytest.mark.gpu


def _run(O, R, prec, op, body, a_off, w_off, level_map=None):
    import torch
    dt, half = (torch.int8, 128) if prec == "i8" else (torch.int16, 32768)
    g = torch.Generator("cuda").manual_seed(O * 31 + R)
    A = torch.randint(-half, half, (O * R + a_off,), dtype=dt, device="cuda", generator=g)
    w = torch.randint(-128, 128, (R + w_off,), dtype=torch.int8, device="cuda", generator=g)
    out = torch.full((O + 1,), 7, dtype=torch.int32, device="cuda")
    ins = [A.data_ptr() + a_off * A.element_size()] + ([w.data_ptr() + w_off] if body == "dot_bcast" else [])
    n = hb.Nest([O, R], 1, op, prec, body, level_map=level_map)
    n.run(ins, out.data_ptr(), torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    n.close()
    a = A[a_off:].cpu().numpy().astype(np.int64).reshape(O, R)
    if op == "sum":
        want = (a * w[w_off:].cpu().numpy().astype(np.int64) if body == "dot_bcast" else a).sum(1)
    else:
        want = a.max(1) if op == "max" else a.min(1)
    got = out.cpu().numpy()
    assert got[O] == 7 and np.array_equal(got[:O], want), (O, R, prec, op, body, a_off, w_off, level_map)


FORMS = [("i8", "sum", "load"), ("i8", "max", "load"), ("i8", "sum", "dot_bcast"), ("i16", "sum", "load"),
         ("i16", "min", "load")]


@pytest.mark.parametrize("prec,op,body", FORMS)
@pytest.mark.parametrize("a_off,w_off", [(0, 0), (1, 0), (0, 3), (9, 16), (13, 7)])
def test_any_row_length_and_alignment(prec, op, body, a_off, w_off):
    # 1 .. 17: less than a granule; 64, 256, 512: whole granules; 512, 1024: the last short rows; both sides of each
    for R in (1, 2, 7, 15, 16, 17, 31, 33, 45, 63, 64, 65, 129, 255, 256, 257, 333, 511, 512, 513, 1000, 1023, 1025, 4099):
        for O in (1, 3, 77, 1500):
            _run(O, R, prec, op, body, a_off, w_off)


@pytest.mark.parametrize("prec,op,body", FORMS)
@pytest.mark.parametrize("level_map", [["grid", ("cta", 4, 0)], ["grid", ("grid", 0, 1000)], ["grid", ("cta", 32, 0)], None])
def test_teams_on_ragged_rows(prec, op, body, level_map):
    for a_off, w_off in ((0, 0), (5, 0), (2, 9)):
        for R in (37, 1001, 40003, 262147):
            _run(9, R, prec, op, body, a_off, w_off, level_map)
