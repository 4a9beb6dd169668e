"""GPU test of a nest's first run on a stream that does not wait for the default
one, while the default stream still has work queued: what the first run finds on
the device (counters, tickets, row lists, tables) is ready whatever the stream.
Values are small integers, so every result is exact.  Scratch is allocated from
memory that held other values before."""
import numpy as np
import pytest

from paper_2309_01906_gb300 import binding as hb

pytestmark = pytest.mark.gpu


def _ints(g, n, dtype):
    import torch
    return torch.randint(-3, 4, (n,), device="cuda", generator=g).to(dtype)


def _csr(fuse):
    import torch
    lens = np.asarray([1, 70, 20000, 0, 5, 3000, 2, 16385, 64, 2048] * 11, np.int64)
    rng = np.random.Generator(np.random.PCG64(3))
    off = np.concatenate([[0], np.cumsum(lens)])
    nnz, cols = int(off[-1]), 4000
    col = rng.integers(0, cols, nnz).astype(np.int32)
    val, x = rng.integers(-2, 3, nnz).astype(np.float32), rng.integers(-2, 3, cols).astype(np.float32)
    csum = np.concatenate([[0], np.cumsum(val.astype(np.int64) * x[col].astype(np.int64))])
    want = torch.from_numpy((csum[off[1:]] - csum[off[:-1]]).astype(np.float32))
    ins = [torch.from_numpy(t).cuda() for t in (off, col, val, x)] + [torch.empty(cols, dtype=torch.int64, device="cuda")]
    n = hb.Nest(csr_rows=lens.size, red_level=1, op="sum", prec="f32", body="csr_gather",
                params=hb.hp_csr_params(nnz, cols, 0, fuse, cols))
    return n, ins, torch.empty(lens.size, device="cuda"), want


def _split(kind):
    import torch
    g = torch.Generator("cuda").manual_seed(11)
    O, R = 3, (1 << 20) + 5
    if kind == "narrow":
        a = _ints(g, O * R, torch.int8)
        n = hb.Nest([O, R], 1, "sum", "i8", "load", level_map=["grid", ("grid", 0, 1 << 14)])
        return n, [a], torch.empty(O, dtype=torch.int32, device="cuda"), a.view(O, R).sum(1, dtype=torch.int32).cpu()
    if kind == "last":
        a = torch.full((O * R,), float("nan"), device="cuda")
        a.view(O, R)[:, 77777] = torch.arange(1.0, O + 1, device="cuda")
        n = hb.Nest([O, R], 1, "last", "f32", "load", level_map=["grid", ("grid", 0, 1 << 14)])
        return n, [a], torch.empty(O, device="cuda"), torch.arange(1.0, O + 1)
    a = _ints(g, O * R, torch.int32)
    n = hb.Nest([O, R], 1, "sum", "i32", "load", level_map=["grid", ("grid", 0, 1 << 14)])
    return n, [a], torch.empty(O, dtype=torch.int32, device="cuda"), a.view(O, R).sum(1, dtype=torch.int32).cpu()


@pytest.mark.parametrize("kind", ["csr", "csr_hist", "narrow", "last", "rect", "batch"])
def test_first_run_on_a_stream_of_its_own(kind):
    import torch
    n, ins, out, want = _csr(kind == "csr_hist") if kind.startswith("csr") else _split("rect" if kind == "batch" else kind)
    junk = [torch.full((1 << 18,), -1, dtype=torch.int32, device="cuda") for _ in range(8)]
    torch.cuda.synchronize()
    del junk
    torch.cuda.empty_cache()
    side = torch.cuda.Stream()             # created non-blocking
    torch.cuda._sleep(1 << 28)             # the default stream is busy for about 0.1 s
    for _ in range(2):
        out.record_stream(side)
        if kind == "batch":
            hb.hp_nest_run_batch([n.handle], [[t.data_ptr() for t in ins]], [out.data_ptr()], side.cuda_stream)
        else:
            n.run([t.data_ptr() for t in ins], out.data_ptr(), side.cuda_stream)
        side.synchronize()
        with torch.cuda.stream(side):
            got = out.cpu()
            out.fill_(0)
        assert torch.equal(got, want)
    assert n.check(side.cuda_stream) == 0
    torch.cuda.synchronize()
    n.close()


@pytest.mark.parametrize("kind", ["csr", "csr_hist", "narrow", "last", "rect"])
def test_first_run_inside_a_capture(kind):
    """A relaxed capture may hold a nest's first run: what it finds is ready at once, not only after a replay."""
    import torch
    n, ins, out, want = _csr(kind == "csr_hist") if kind.startswith("csr") else _split(kind)
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(side):
        graph = torch.cuda.CUDAGraph()
        graph.capture_begin(capture_error_mode="relaxed")
        n.run([t.data_ptr() for t in ins], out.data_ptr(), side.cuda_stream)
        graph.capture_end()
        for replay in (False, True, True, False, True):
            out.fill_(7)
            if replay:
                graph.replay()
            else:
                n.run([t.data_ptr() for t in ins], out.data_ptr(), side.cuda_stream)
            side.synchronize()
            assert torch.equal(out.cpu(), want)
    assert n.check(side.cuda_stream) == 0
    del graph
    n.close()
