"""GPU test of grid parts in the batched executor: the warp that takes an output's
last ticket reads parts that other CTAs wrote.  Many outputs in a few parts
each, and parts that arrive in bursts; one nest listed many times.  Integers, so
every run is exact."""
import pytest

from paper_2309_01906_gb300 import binding as hb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("levels", ["one", "two"])
def test_parts_of_many_outputs(levels):
    import torch
    s = torch.cuda.current_stream().cuda_stream
    g = torch.Generator("cuda").manual_seed(2)
    nests, ins, outs, want = [], [], [], []
    for O, R, tile in [(4000, 4096, 1024), (997, 16384, 4096), (64, 65536, 2048), (1, 1 << 20, 4096), (3001, 2050, 1025)]:
        A = torch.randint(-(1 << 30), 1 << 30, (O, R), dtype=torch.int32, device="cuda", generator=g)
        if levels == "one":
            nests.append(hb.Nest([O, R], 1, "sum", "i64", "load", level_map=["grid", ("grid", 0, tile)]))
        else:
            nests.append(hb.Nest([O, R // tile, tile], 1, "sum", "i64", "load", level_map=["grid", ("grid", 0, 1), "cta"]))
        assert nests[-1].describe()["grid_parts"] == (R // tile if R % 4 == 0 or levels == "two" else 2)
        ins.append(A)
        want.append(A.sum(1, dtype=torch.int64))
        outs.append(torch.empty(O, dtype=torch.int64, device="cuda"))
    for _ in range(20):
        for t in outs:
            t.fill_(7)
        hb.hp_nest_run_batch([n.handle for n in nests], [[t.data_ptr()] for t in ins], [t.data_ptr() for t in outs], s)
        torch.cuda.synchronize()
        for t, w in zip(outs, want):
            assert torch.equal(t, w)
    for n in nests:
        n.close()


def test_one_nest_listed_many_times():
    """The entries of one nest run at the same time on different inputs: each has its own parts."""
    import torch
    s = torch.cuda.current_stream().cuda_stream
    g = torch.Generator("cuda").manual_seed(4)
    for O, R, level_map in [(300, 65536, None), (1, 1 << 20, None), (7, 5000, ["grid", ("grid", 0, 625)])]:
        n = hb.Nest([O, R], 1, "sum", "i64", "load", level_map=level_map)
        assert n.describe()["grid_parts"] > 1
        ins = [torch.randint(-(1 << 30), 1 << 30, (O, R), dtype=torch.int32, device="cuda", generator=g) for _ in range(8)]
        outs = [torch.empty(O, dtype=torch.int64, device="cuda") for _ in ins]
        for _ in range(5):
            for t in outs:
                t.fill_(7)
            hb.hp_nest_run_batch([n.handle] * 8, [[t.data_ptr()] for t in ins], [t.data_ptr() for t in outs], s)
            torch.cuda.synchronize()
            for t, o in zip(ins, outs):
                assert torch.equal(o, t.sum(1, dtype=torch.int64))
        n.close()
