"""GPU test of ordered reductions around the row counts where short rows begin to
share a warp (12, 18 or 24 rows per SM), and where ragged rows begin to be read as shifted granules (4
rows of 64 iterations, 18 rows per SM of 8).  a = +-1 and small integers, so every FP32
operation is exact; last-valid copies values."""
import pytest

from paper_2309_01906_gb300 import binding as hb

pytestmark = pytest.mark.gpu

LENGTHS = (1, 2, 7, 8, 9, 15, 16, 17, 31, 32, 50, 63, 64, 65, 100, 127, 128, 129, 255)
ROWS = (1, 3, 4, 5, 1824, 1825, 2736, 2737, 3648, 3649)


def _check(op, O, R, ins, want):
    import torch
    out = torch.full((want.numel() + 1,), 7.0, device="cuda")
    n = hb.Nest([O, R], 1, op, "f32", "load")
    n.run([t.data_ptr() for t in ins], out.data_ptr(), torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    n.close()
    assert out[-1] == 7.0 and torch.equal(out[:-1].nan_to_num(nan=-99.0), want.reshape(-1).nan_to_num(nan=-99.0)), (op, O, R)


@pytest.mark.parametrize("offset", [0, 1, 4])
def test_few_and_many_rows(offset):
    import torch
    g = torch.Generator("cuda").manual_seed(offset)
    for R in LENGTHS:
        for O in ROWS:
            buf = [torch.randint(-8, 9, (O * R + offset,), device="cuda", generator=g).float() for _ in range(2)]
            a, b = buf[0][offset:].sign_(), buf[1][offset:]
            a[a == 0] = 1.0
            suffix = a.view(O, R).flip(1).cumprod(1).flip(1)
            later = torch.cat([suffix[:, 1:], torch.ones(O, 1, device="cuda")], 1)
            _check("compose", O, R, [a, b], torch.stack([suffix[:, 0], (later * b.view(O, R)).sum(1)], 1))
            v = b.clone() if offset == 0 else b
            v[torch.rand(O * R, device="cuda", generator=g) < 0.9] = float("nan")
            m = v.view(O, R)
            at = torch.where(m.isnan(), -1, torch.arange(R, device="cuda")).amax(1)
            _check("last", O, R, [v], torch.where(at < 0, float("nan"), m.gather(1, at.clamp(min=0)[:, None])[:, 0]))
            if offset % 4 == 0:   # products of [[1, k], [0, 1]]
                k = torch.randint(-8, 9, (O, R), device="cuda", generator=g).float()
                one, zero = torch.ones_like(k), torch.zeros_like(k)
                mat = torch.stack([one, k, zero, one], 2).reshape(-1)
                _check("mat2", O, R, [mat], torch.stack([one[:, 0], k.sum(1), zero[:, 0], one[:, 0]], 1))
