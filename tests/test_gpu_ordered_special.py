"""GPU test of ordered reductions on signed zeros, infinities and NaN: a row gives
the same bits in a nest of few rows (a warp each) and of many (rows share a
warp), also where joining an identity shows (-0, infinite matrix entries)."""
import pytest

from paper_2309_01906_gb300 import binding as hb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("op,floats,n_out", [("compose", 1, 2), ("mat2", 4, 4), ("last", 1, 1)])
@pytest.mark.parametrize("R", [1, 2, 5, 7, 8, 9, 16, 31, 32, 50, 64, 100, 127, 128])
def test_few_and_many_rows_agree(op, floats, n_out, R):
    import torch
    g = torch.Generator("cuda").manual_seed(R)
    special = torch.tensor([0.0, -0.0, 1.0, -1.0, float("inf"), -float("inf"), float("nan"), 1e-40, 2.0], device="cuda")
    rows, few = 4000, 12
    ins = []
    for _ in range(2 if op == "compose" else 1):
        t = torch.randint(0, special.numel(), (few, R * floats), device="cuda", generator=g)
        v = special[t]
        v[:4] = torch.where(v[:4].isfinite(), v[:4], -0.0)      # rows without infinities: zeros and their signs
        v[4:8] = torch.where(v[4:8].isnan(), 1.0, v[4:8])
        ins.append(v.repeat(rows // few + 1, 1)[:rows].contiguous())
    s = torch.cuda.current_stream().cuda_stream
    outs = []
    for O in (few, rows):
        out = torch.full((O, n_out), 7.0, device="cuda")
        n = hb.Nest([O, R], 1, op, "f32", "load")
        kernel = n.describe()["kernel"]
        n.run([t.data_ptr() for t in ins], out.data_ptr(), s)
        torch.cuda.synchronize()
        n.close()
        outs.append((kernel, out))
    if op != "mat2" or R <= 64:      # 16 pieces of 4 matrices
        assert outs[1][0] == "ordered_short" and (R <= 16 or outs[0][0] == "ordered_warp")
    a, b = outs[0][1], outs[1][1]
    for k in range(rows // few):
        c = b[k * few:(k + 1) * few]
        assert torch.equal(a.isnan(), c.isnan()) and torch.equal(a.nan_to_num(nan=0.0).view(torch.int32), c.nan_to_num(nan=0.0).view(torch.int32)), k
