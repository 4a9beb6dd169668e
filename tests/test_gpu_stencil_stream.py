"""GPU test of the register-streamed stencil kernels: the same bits as the tiled
kernel (a map with an explicit tile), for every radius and step count that has a
streamed kernel, on 16-byte rows and on others, with ragged edges and with
infinities and NaN in the input.  Both run the same FMA chains, so the tolerance
is zero."""
import numpy as np
import pytest

from paper_2309_01906_gb300 import binding as hb

pytestmark = pytest.mark.gpu

STREAMED = [(r, t) for r in (1, 2, 3, 4) for t in range(1, 9) if r < 4 or t <= 5]


def _run(st, buf, out_offset, n):
    import torch
    out = torch.full((n + out_offset + 1,), 7.0, dtype=torch.float32, device="cuda")
    s = torch.cuda.current_stream().cuda_stream
    st.run(buf.data_ptr(), out.data_ptr() + 4 * out_offset, s)
    assert st.check(s) == 0
    assert out[n + out_offset].item() == 7.0 and torch.all(out[:out_offset] == 7.0)
    return out[out_offset:out_offset + n].view(torch.int32)


@pytest.mark.parametrize("r,T", STREAMED)
def test_streamed_equals_tiled(r, T):
    import torch
    g = np.random.Generator(np.random.PCG64(100 * r + T))
    c = g.uniform(-0.5, 0.5, (2 * r + 1) ** 2).astype(np.float32).tolist()
    # one point, one column, one short row, less and more than one warp's columns and strip, ragged and whole
    for ny, nx in [(1, 1), (9, 1), (1, 130), (5, 64), (61, 127), (130, 260), (300, 517), (1030, 388)]:
        A = g.uniform(-1.0, 1.0, ny * nx).astype(np.float32)
        A[g.integers(0, ny * nx, 2)] = [np.inf, np.nan]
        buf = torch.from_numpy(A).cuda()
        auto, tiled = hb.Stencil(ny, nx, r, c, T), hb.Stencil(ny, nx, r, c, T, tile=(16, 64))
        assert tiled.describe()["kernel"] == "stencil_tile"
        if (r, T) != (1, 1) or nx % 4:
            assert auto.describe()["kernel"] == "stencil_stream"
        want = _run(tiled, buf, 0, ny * nx)
        for out_offset in (0, 1):      # 1: the output is not 16-byte aligned
            assert torch.equal(_run(auto, buf, out_offset, ny * nx), want), (ny, nx, out_offset)
        auto.close()
        tiled.close()


@pytest.mark.parametrize("r,T", [(1, 2), (2, 7), (3, 8), (4, 2), (4, 5)])
def test_column_group_edges(r, T):
    import torch
    g = np.random.Generator(np.random.PCG64(1000 * r + T))
    c = g.uniform(-0.5, 0.5, (2 * r + 1) ** 2).astype(np.float32).tolist()
    probe = hb.Stencil(64, 64, r, c, T)
    cols = probe.describe()["warp_columns"]
    probe.close()
    # one group more from 121 columns on, and again every `cols`; the inner groups overlap by the ghost columns
    for nx in (119, 120, 121, 124, 120 + cols, 121 + cols, 123 + cols, 120 + 2 * cols, 122 + 2 * cols):
        A = g.uniform(-1.0, 1.0, 37 * nx).astype(np.float32)
        buf = torch.from_numpy(A).cuda()
        auto, tiled = hb.Stencil(37, nx, r, c, T), hb.Stencil(37, nx, r, c, T, tile=(16, 64))
        assert auto.describe()["kernel"] == "stencil_stream"
        want = _run(tiled, buf, 0, 37 * nx)
        assert torch.equal(_run(auto, buf, 0, 37 * nx), want), nx
        auto.close()
        tiled.close()


@pytest.mark.parametrize("r,T", [(3, 8), (4, 2)])
def test_long_array_of_one_tile_width(r, T):
    import torch
    g = np.random.Generator(np.random.PCG64(7 * r + T))
    c = g.uniform(-0.5, 0.5, (2 * r + 1) ** 2).astype(np.float32).tolist()
    A = torch.from_numpy(g.uniform(-1.0, 1.0, 8000 * 128).astype(np.float32)).cuda()
    auto, tiled = hb.Stencil(8000, 128, r, c, T), hb.Stencil(8000, 128, r, c, T, tile=(16, 64))
    assert auto.describe()["kernel"] == "stencil_tile"
    assert torch.equal(_run(auto, A, 0, 8000 * 128), _run(tiled, A, 0, 8000 * 128))
    auto.close()
    tiled.close()
