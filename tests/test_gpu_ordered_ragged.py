"""GPU test of ordered reductions over rows of any length and alignment: short
rows that share a warp, and rows read as shifted granules.  The maps have
a = +-1 and small integer b, so every FP32 operation is exact and the result must
be the recurrence's bit for bit; last-valid copies values."""
import numpy as np
import pytest

from paper_2309_01906_gb300 import binding as hb

pytestmark = pytest.mark.gpu

# pieces of 8 (and 32 aligned values): one piece, two, a power of two of them, one round of a warp and more
LENGTHS = [1, 3, 7, 8, 9, 15, 16, 17, 32, 33, 63, 64, 65, 127, 128, 129, 255, 256, 257, 1000, 1001, 1027, 40003]


def _place(v, offset):
    import torch
    buf = torch.zeros(v.size + offset, dtype=torch.float32, device="cuda")
    buf[offset:] = torch.from_numpy(v.reshape(-1)).cuda()
    return buf, buf.data_ptr() + 4 * offset


def _run(op, O, R, ins, n_out):
    import torch
    out = torch.full((O * n_out + 1,), 7.0, device="cuda")
    n = hb.Nest([O, R], 1, op, "f32", "load")
    n.run([p for _, p in ins], out.data_ptr(), torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    n.close()
    got = out.cpu().numpy()
    assert got[O * n_out] == 7.0
    return got[:O * n_out].reshape(O, n_out)


@pytest.mark.parametrize("off_a,off_b", [(0, 0), (1, 1), (2, 3), (0, 1), (4, 3)])
def test_compose_exact_at_any_alignment(off_a, off_b):
    for R in LENGTHS:
        for O in (1, 5, 37):
            g = np.random.Generator(np.random.PCG64(R * 41 + O))
            a = g.choice([-1.0, 1.0], (O, R)).astype(np.float32)
            b = g.integers(-8, 9, (O, R)).astype(np.float32)
            got = _run("compose", O, R, [_place(a, off_a), _place(b, off_b)], 2)
            suffix = np.cumprod(a[:, ::-1].astype(np.int64), axis=1)[:, ::-1]     # product of a[x:]
            later = np.concatenate([suffix[:, 1:], np.ones((O, 1), np.int64)], axis=1)
            assert np.array_equal(got[:, 0], suffix[:, 0]) and np.array_equal(got[:, 1], (later * b).sum(1)), (R, O)


@pytest.mark.parametrize("offset", [0, 1, 2, 3])
def test_last_valid_at_any_alignment(offset):
    for R in LENGTHS:
        for O in (1, 5, 37):
            g = np.random.Generator(np.random.PCG64(R * 43 + O))
            v = g.standard_normal((O, R)).astype(np.float32)
            v[g.random((O, R)) < 0.97] = np.nan
            got = _run("last", O, R, [_place(v, offset)], 1)[:, 0]
            valid = ~np.isnan(v)
            want = np.where(valid.any(1), v[np.arange(O), R - 1 - np.argmax(valid[:, ::-1], axis=1)],
                            np.float32(np.nan))
            assert np.array_equal(got, want, equal_nan=True), (R, O)
