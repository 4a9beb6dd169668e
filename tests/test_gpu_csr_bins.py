"""GPU test of the fused histogram with many more bins than rows (its clear has to
reach every bin, by more CTAs than the rows take): exact counts, run after run."""
import numpy as np
import pytest

from paper_2309_01906_gb300 import binding as hb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,bins", [(1, 12287), (1, 12288), (1, 12289), (3, 1 << 20), (300, (1 << 22) + 77), (1, 1 << 24)])
def test_more_bins_than_rows(rows, bins):
    import torch
    g = np.random.Generator(np.random.PCG64(bins))
    off = np.arange(rows + 1, dtype=np.int64) * 50
    nnz = int(off[-1])
    col = g.integers(0, bins, nnz).astype(np.int32)
    val = g.integers(-2, 3, nnz).astype(np.float32)
    ins = [torch.from_numpy(t).cuda() for t in (off, col, val)] + [torch.ones(bins, device="cuda")]
    y, h = torch.empty(rows, device="cuda"), torch.empty(bins, dtype=torch.int64, device="cuda")
    s = torch.cuda.current_stream().cuda_stream
    n = hb.Nest(csr_rows=rows, red_level=1, op="sum", prec="f32", body="csr_gather",
                params=hb.hp_csr_params(nnz, bins, 0, 1, bins))
    for _ in range(2):
        h.fill_(-1)
        t0, t1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        t0.record()
        n.run([t.data_ptr() for t in ins] + [h.data_ptr()], y.data_ptr(), s)
        t1.record()
        assert n.check(s) == 0
        assert np.array_equal(h.cpu().numpy(), np.bincount(col, minlength=bins))
        assert np.array_equal(y.cpu().numpy(), val.reshape(rows, 50).sum(1))
    # 2^24 bins are 134 MB: 20 us at HBM's rate, 2000 us by one CTA
    assert t0.elapsed_time(t1) < 0.5
    n.close()
