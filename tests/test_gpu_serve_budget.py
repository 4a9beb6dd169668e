"""GPU test of a server's memory budget: a request is admitted when its inputs,
outputs and the scratch of four teams per SM fit, whatever parts the planner cuts."""
import pytest

from paper_2309_01906_gb300 import binding as hb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("O", [1, 100, 200, 303, 304, 1000])
def test_budget_of_exactly_one_request(O):
    import torch
    R = 300000
    A = torch.randint(-9, 10, (O, R), device="cuda").float()
    out = torch.zeros(O, device="cuda")
    parts = -(-608 // O) if O < 304 else 0
    need = 4 * (O * R + O) + (4 * O * min(parts, R // 16384) + 4 * O if parts else 0)
    n = hb.Nest([O, R], 1, "sum", "f32", "load")
    torch.cuda.synchronize()
    for budget, fits in ((need, True), (need - 1, False)):
        server = hb.hp_serve_create(budget, 4, 1)
        try:
            if fits:
                assert hb.hp_serve_poll(server, hb.hp_serve_submit(server, n.handle, [A.data_ptr()], out.data_ptr()), -1) == hb.HP_OK
                assert torch.equal(out, A.sum(1))
            else:
                with pytest.raises(hb.HPError):
                    hb.hp_serve_submit(server, n.handle, [A.data_ptr()], out.data_ptr())
        finally:
            hb.hp_serve_destroy(server)
    n.close()
