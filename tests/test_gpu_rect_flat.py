"""GPU test of the contiguous block kernel and of the combine of grid parts: the
bits of the batched executor, which folds the same plan from its shared-memory
ring and combines an output's parts in one thread.  Same per-thread order, same
trees, so the tolerance is zero."""
import pytest

from paper_2309_01906_gb300 import binding as hb

pytestmark = pytest.mark.gpu

# CTA teams (whole vectors or not, one step or many); grid parts: fewer than a
# group of 8 chains, than 32 chains, more than 32, and ragged last parts
SHAPES = [(33, 4099), (5, 8195), (700, 5001), (2000, 4100), (1, 65536), (1, 70001), (3, (1 << 18) + 4), (30, 262147),
          (100, 65537), (300, 65540), (700, 65537), (1, (1 << 20) + 1), (1, 5000004)]


@pytest.mark.parametrize("prec,op", [("f32", "sum"), ("f32_comp", "sum"), ("f32", "min"), ("i32", "max"), ("i64", "sum")])
@pytest.mark.parametrize("body", ["load", "dot_bcast"])
def test_flat_blocks_equal_the_batched_executor(prec, op, body):
    import torch
    s = torch.cuda.current_stream().cuda_stream
    for O, R in SHAPES:
        g = torch.Generator("cuda").manual_seed(O + R)
        if prec[0] == "f":
            A, w = torch.randn(O * R, device="cuda", generator=g), torch.randn(R, device="cuda", generator=g)
        else:
            A = torch.randint(-(1 << 30), 1 << 30, (O * R,), dtype=torch.int32, device="cuda", generator=g)
            w = torch.randint(-1000, 1000, (R,), dtype=torch.int32, device="cuda", generator=g)
        ins = [A.data_ptr()] + ([w.data_ptr()] if body == "dot_bcast" else [])
        n = hb.Nest([O, R], 1, op, prec, body)
        assert n.describe()["team"] == "block"
        one = torch.full((O + 1,), 9, dtype=torch.int64 if prec == "i64" else A.dtype, device="cuda")
        many = torch.full_like(one, 9)
        n.run(ins, one.data_ptr(), s)
        hb.hp_nest_run_batch([n.handle], [ins], [many.data_ptr()], s)
        torch.cuda.synchronize()
        n.close()
        assert one[O] == 9 and torch.equal(one, many), (O, R)


@pytest.mark.parametrize("prec", ["f32", "f32_comp", "i64"])
def test_long_rows_leave_the_pipeline(prec):
    import torch
    s = torch.cuda.current_stream().cuda_stream
    # around the first row length that leaves it, and tails of one to three more steps of 1024 elements
    for O, R in [(700, 4092), (700, 4096), (701, 4100), (333, 5120), (91, 6148), (90, 7164), (90, 8188), (33, 8192)]:
        g = torch.Generator("cuda").manual_seed(O + R)
        A = torch.randn(O * R, device="cuda", generator=g) if prec[0] == "f" else \
            torch.randint(-(1 << 30), 1 << 30, (O * R,), dtype=torch.int32, device="cuda", generator=g)
        n = hb.Nest([O, R], 1, "sum", prec, "load", level_map=["grid", "cta"])
        assert n.describe()["pipe"] == 1
        one = torch.full((O + 1,), 9, dtype=torch.int64 if prec == "i64" else A.dtype, device="cuda")
        many = torch.full_like(one, 9)
        n.run([A.data_ptr()], one.data_ptr(), s)
        hb.hp_nest_run_batch([n.handle], [[A.data_ptr()]], [many.data_ptr()], s)
        torch.cuda.synchronize()
        n.close()
        assert one[O] == 9 and torch.equal(one, many), (O, R)
