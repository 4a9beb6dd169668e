"""GPU test of the CSR work kernel at the edges of its units (2048, 256 and 32
rows of the three short classes, single rows and chunks of the long ones), run
after run on one nest (the kernel clears its own counters).  Values and x are
small integers whose row sums stay below 2^24, so FP32 sums are exact."""
import numpy as np
import pytest

from paper_2309_01906_gb300 import binding as hb

pytestmark = pytest.mark.gpu

SHAPES = {
    "thread_rows": [3] * 2047, "thread_rows_unit": [3] * 2048, "thread_rows_more": [4] * 2049 + [0] * 5,
    "lane_rows": [40] * 255, "lane_rows_unit": [5] * 256, "lane_rows_more": [64] * 257,
    "warp_rows": [100] * 31, "warp_rows_unit": [65] * 32, "warp_rows_more": [2048] * 33,
    "cta_rows": [2049, 16384, 3001], "one_chunk_more": [16385], "long_rows": [65536, 40000, 49152, 49153],
    "all": [1, 70, 20000, 0, 5, 3000, 2, 16385, 64, 2048] * 23,
    "combine_kernel": [65536] * 131,       # more chunk slots than the last CTA folds itself
}


@pytest.mark.parametrize("prec", ["f32", "f32_comp"])
@pytest.mark.parametrize("shape", SHAPES)
def test_units_of_every_class(shape, prec):
    import torch
    lens = np.asarray(SHAPES[shape], np.int64)
    g = np.random.Generator(np.random.PCG64(lens.size))
    off = np.concatenate([[0], np.cumsum(lens)])
    nnz, n_cols = int(off[-1]), 5000
    col = g.integers(0, n_cols, nnz).astype(np.int32)
    val = g.integers(-2, 3, nnz).astype(np.float32)
    x = g.integers(-2, 3, n_cols).astype(np.float32)
    csum = np.concatenate([[0], np.cumsum(val.astype(np.int64) * x[col].astype(np.int64))])
    want = (csum[off[1:]] - csum[off[:-1]]).astype(np.float32)
    bins = (n_cols >> 4) + 1
    d = [torch.from_numpy(t).cuda() for t in (off, col, val, x)]
    s = torch.cuda.current_stream().cuda_stream
    for fuse in (0, 1):
        n = hb.Nest(csr_rows=lens.size, red_level=1, op="sum", prec=prec, body="csr_gather",
                    params=hb.hp_csr_params(nnz, n_cols, 4, fuse, bins))
        for _ in range(3):
            y = torch.full((lens.size,), 7.0, device="cuda")
            h = torch.full((bins,), -1, dtype=torch.int64, device="cuda")
            n.run([t.data_ptr() for t in d] + [h.data_ptr()], y.data_ptr(), s)
            assert n.check(s) == 0
            assert np.array_equal(y.cpu().numpy(), want)
            if fuse:
                assert np.array_equal(h.cpu().numpy(), np.bincount(col >> 4, minlength=bins))
        n.close()
