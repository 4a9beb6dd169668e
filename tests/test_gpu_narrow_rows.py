"""GPU test of the kernels that 8- and 16-bit rows of a warp team go to, by their
number: a warp per row (whole pieces or single elements) for few, a warp shared by
short rows for many, around the row counts where one takes over from the other.
Exact against 64-bit sums."""
import pytest

from paper_2309_01906_gb300 import binding as hb

pytestmark = pytest.mark.gpu

FORMS = [("i8", "sum", "load"), ("i8", "max", "load"), ("i8", "sum", "dot_bcast"), ("i16", "sum", "load"),
         ("i16", "min", "load")]


@pytest.mark.parametrize("prec,op,body", FORMS)
@pytest.mark.parametrize("a_off,w_off", [(0, 0), (1, 0), (0, 3), (13, 7)])
def test_few_and_many_rows(prec, op, body, a_off, w_off):
    import torch
    dt, half = (torch.int8, 128) if prec == "i8" else (torch.int16, 32768)
    g = torch.Generator("cuda").manual_seed(a_off * 31 + w_off)
    s = torch.cuda.current_stream().cuda_stream
    rows = (3040, 3041, 12160, 12161, 60000)
    for R in (1, 3, 8, 16, 31, 32, 100, 128, 255, 256, 333, 384, 385, 511, 512, 513, 777, 1023, 1024, 1025):
        A = torch.randint(-half, half, (rows[-1] * R + a_off,), dtype=dt, device="cuda", generator=g)
        w = torch.randint(-128, 128, (R + w_off,), dtype=torch.int8, device="cuda", generator=g)
        a = A[a_off:].view(rows[-1], R)
        if op == "sum":
            want = ((a.int() * w[w_off:].int()) if body == "dot_bcast" else a).sum(1, dtype=torch.int64).int()
        else:
            want = (a.amax(1) if op == "max" else a.amin(1)).int()
        for O in rows:
            out = torch.full((O + 1,), 7, dtype=torch.int32, device="cuda")
            n = hb.Nest([O, R], 1, op, prec, body)
            n.run([A.data_ptr() + a_off * A.element_size()] + ([w.data_ptr() + w_off] if body == "dot_bcast" else []),
                  out.data_ptr(), s)
            torch.cuda.synchronize()
            n.close()
            assert out[O] == 7 and torch.equal(out[:O], want[:O]), (O, R, prec, op, body, a_off, w_off)
