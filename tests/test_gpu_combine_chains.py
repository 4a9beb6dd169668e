"""GPU test of the combine of partials against its restatement on the host: part g
adds to chain g mod 32 from +0, and the 32 chains join in a butterfly, neighbours
first.  Both device forms: by a warp (split rectangular nests) and by one thread
(long CSR rows, in the work kernel's last CTA and in a kernel of its own).  The
partials are what the same folds give as outputs of their own, so FP32 sums have
to agree bit for bit; compensated sums run on small integers, exactly."""
import numpy as np
import pytest

from paper_2309_01906_gb300 import binding as hb

pytestmark = pytest.mark.gpu

PARTS = [2, 7, 8, 9, 15, 16, 17, 23, 24, 25, 31, 32, 33, 40, 63, 64, 65, 127, 300, 608, 1000]
CHUNK = 16384


def _chains(parts):
    c = np.zeros(32, np.float32)
    for g, p in enumerate(parts):
        c[g % 32] = c[g % 32] + p
    while c.size > 1:
        c = c[0::2] + c[1::2]
    return c[0]


def _run(n, ins, out):
    import torch
    s = torch.cuda.current_stream().cuda_stream
    n.run([t.data_ptr() for t in ins], out.data_ptr(), s)
    assert n.check(s) == 0
    torch.cuda.synchronize()
    n.close()
    return out.cpu().numpy()


@pytest.mark.parametrize("G", PARTS)
def test_split_rows(G):
    import torch
    g = torch.Generator("cuda").manual_seed(G)
    O, tile = 5, 1024
    A = torch.randn(O * G * tile, device="cuda", generator=g)
    parts = _run(hb.Nest([O * G, tile], 1, "sum", "f32", "load", level_map=["grid", "cta"]), [A], torch.empty(O * G, device="cuda"))
    got = _run(hb.Nest([O, G * tile], 1, "sum", "f32", "load", level_map=["grid", ("grid", 0, tile)]), [A], torch.empty(O, device="cuda"))
    want = np.array([_chains(p) for p in parts.reshape(O, G)], np.float32)
    assert np.array_equal(got, want), G
    # compensated, the last part ragged
    R = (G - 1) * tile + 100
    B = torch.randint(-50, 51, (O, R), device="cuda", generator=g)
    n = hb.Nest([O, R], 1, "sum", "f32_comp", "load", level_map=["grid", ("grid", 0, tile)])
    assert n.describe()["grid_parts"] == G
    got = _run(n, [B.float()], torch.empty(O, device="cuda"))
    assert np.array_equal(got, B.sum(1).float().cpu().numpy()), G


@pytest.mark.parametrize("copies", [1, 5])       # 5: more chunk slots than the last CTA folds itself
@pytest.mark.parametrize("prec", ["f32", "f32_comp"])
def test_long_csr_rows(prec, copies):
    import torch
    chunks = [2, 7, 8, 9, 15, 16, 17, 24, 25, 31, 32, 33, 70] * copies
    lens = np.array([(c - 1) * CHUNK + 1 + 1009 * (i % 16) for i, c in enumerate(chunks)], np.int64)
    off = np.concatenate([[0], np.cumsum(lens)])
    nnz, cols = int(off[-1]), 4096
    assert (2 * (nnz // CHUNK) + 2 > 1024) == (copies > 1)
    g = torch.Generator("cuda").manual_seed(copies)
    col = torch.randint(0, cols, (nnz,), dtype=torch.int32, device="cuda", generator=g)
    if prec == "f32":
        val, x = torch.randn(nnz, device="cuda", generator=g), torch.randn(cols, device="cuda", generator=g)
    else:
        val, x = (torch.randint(-2, 3, (k,), device="cuda", generator=g).float() for k in (nnz, cols))

    def csr(offsets):
        n = hb.Nest(csr_rows=offsets.size - 1, red_level=1, op="sum", prec=prec, body="csr_gather",
                    params=hb.hp_csr_params(nnz, cols, 0, 0, 0))
        return _run(n, [torch.from_numpy(offsets).cuda(), col, val, x], torch.empty(offsets.size - 1, device="cuda"))

    got = csr(off)
    if prec == "f32_comp":
        total = torch.cat([torch.zeros(1, device="cuda", dtype=torch.float64), (val * x[col.long()]).double().cumsum(0)]).cpu().numpy()
        assert np.array_equal(got, (total[off[1:]] - total[off[:-1]]).astype(np.float32))
        return
    # the partials: every chunk a row of its own, which the CTA class folds as a chunk is folded (a
    # ragged last one may belong to a shorter class, so these rows are whole chunks)
    lens = np.array([c * CHUNK for c in chunks], np.int64)
    off = np.concatenate([[0], np.cumsum(lens)])
    nnz = int(off[-1])
    col, val = torch.cat([col, col])[:nnz], torch.cat([val, val])[:nnz]
    got, parts = csr(off), csr(np.arange(nnz // CHUNK + 1, dtype=np.int64) * CHUNK)
    first = np.concatenate([[0], np.cumsum(chunks)])
    want = np.array([_chains(parts[a:b]) for a, b in zip(first[:-1], first[1:])], np.float32)
    assert np.array_equal(got, want)
