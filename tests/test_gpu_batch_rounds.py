"""GPU test of the batched executor's lanes teams: windows that hold one round of
a team's rows, two, or more take different folds of the same order and tree, and
rows that wrap around the end of the shared-memory ring take others than rows
that do not.  The bits are those of one launch per nest, so the tolerance is
zero."""
import pytest

from paper_2309_01906_gb300 import binding as hb

pytestmark = pytest.mark.gpu

LENGTHS = [3, 8, 20, 33, 100, 255, 512, 1021, 2047, 4095]
OUTPUTS = [1, 2, 7, 33, 300]


@pytest.mark.parametrize("prec,op,body", [("f32", "sum", "load"), ("f32_comp", "sum", "dot_bcast"), ("i64", "sum", "load"),
                                          ("i32", "max", "dot_bcast")])
def test_rounds_equal_single_launches(prec, op, body):
    import torch
    s = torch.cuda.current_stream().cuda_stream
    g = torch.Generator("cuda").manual_seed(5)
    nests, ins, one, many = [], [], [], []
    for R in LENGTHS:
        for O in OUTPUTS:
            if prec[0] == "f":
                A, w = torch.randn(O * R, device="cuda", generator=g), torch.randn(R, device="cuda", generator=g)
            else:
                A = torch.randint(-(1 << 30), 1 << 30, (O * R,), dtype=torch.int32, device="cuda", generator=g)
                w = torch.randint(-1000, 1000, (R,), dtype=torch.int32, device="cuda", generator=g)
            nests.append(hb.Nest([O, R], 1, op, prec, body))
            ins.append([A, w] if body == "dot_bcast" else [A])
            out = torch.full((O + 1,), 9, dtype=torch.int64 if prec == "i64" else A.dtype, device="cuda")
            one.append(out)
            many.append(out.clone())
            nests[-1].run([t.data_ptr() for t in ins[-1]], out.data_ptr(), s)
    hb.hp_nest_run_batch([n.handle for n in nests], [[t.data_ptr() for t in i] for i in ins], [t.data_ptr() for t in many], s)
    torch.cuda.synchronize()
    for k, n in enumerate(nests):
        n.close()
        assert one[k][-1] == 9 and torch.equal(one[k], many[k]), (LENGTHS[k // len(OUTPUTS)], OUTPUTS[k % len(OUTPUTS)])
