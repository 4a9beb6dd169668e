"""GPU test of a nest whose input changes its alignment from run to run: another
kernel takes rows that do not start on 16 bytes, with a launch of its own size."""
import pytest

from paper_2309_01906_gb300 import binding as hb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("body", ["load", "dot_bcast"])
@pytest.mark.parametrize("O,R", [(100000, 31), (7, 31), (3, 63), (50001, 63), (20000, 7), (5, 101)])
def test_alignment_alternates(O, R, body):
    import torch
    g = torch.Generator("cuda").manual_seed(R)
    A = torch.randint(-9, 10, (O * R + 8,), device="cuda", generator=g).int()
    w = torch.randint(-9, 10, (R,), device="cuda", generator=g).int()
    s = torch.cuda.current_stream().cuda_stream
    n = hb.Nest([O, R], 1, "sum", "i32", body)
    for k in (0, 1, 0, 4, 3, 0, 2, 1):
        out = torch.full((O + 1,), 7, dtype=torch.int32, device="cuda")
        n.run([A.data_ptr() + 4 * k] + ([w.data_ptr()] if body == "dot_bcast" else []), out.data_ptr(), s)
        a = A[k:k + O * R].view(O, R)
        assert out[O] == 7 and torch.equal(out[:O], (a * w if body == "dot_bcast" else a).sum(1, dtype=torch.int32)), k
    n.close()
