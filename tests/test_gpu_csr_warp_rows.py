"""GPU test of CSR rows that take a warp or 8 lanes each, around the row counts at
which a unit of work holds 1, 2, 4 (and 8) of them per team (760 CTAs with a unit
each, 8 for long rows).  Small integers, so FP32 sums are exact."""
import numpy as np
import pytest

from paper_2309_01906_gb300 import binding as hb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,ln", [(9, 67), (12159, 600), (12161, 67), (24319, 67), (24321, 300), (97279, 520), (97281, 520),
                                     (97296, 67), (194561, 67), (1, 20), (33, 64), (48639, 64), (48641, 64), (97279, 50),
                                     (97281, 50), (194559, 20), (194561, 20), (389121, 5)])
@pytest.mark.parametrize("fuse", [0, 1])
def test_rows_per_team(rows, ln, fuse):
    import torch
    g = torch.Generator("cuda").manual_seed(rows)
    cols = 2000
    off = torch.arange(rows + 1, device="cuda") * ln
    col = torch.randint(0, cols, (rows * ln,), dtype=torch.int32, device="cuda", generator=g)
    val, x = (torch.randint(-2, 3, (k,), device="cuda", generator=g).float() for k in (rows * ln, cols))
    y, h = torch.full((rows,), 7.0, device="cuda"), torch.full((cols,), -1, dtype=torch.int64, device="cuda")
    s = torch.cuda.current_stream().cuda_stream
    n = hb.Nest(csr_rows=rows, red_level=1, op="sum", prec="f32", body="csr_gather",
                params=hb.hp_csr_params(rows * ln, cols, 0, fuse, cols))
    for _ in range(2):
        n.run([t.data_ptr() for t in (off, col, val, x, h)], y.data_ptr(), s)
        assert n.check(s) == 0
        assert torch.equal(y, (val * x[col.long()]).view(rows, ln).sum(1))
        if fuse:
            assert torch.equal(h, torch.bincount(col, minlength=cols))
    n.close()
