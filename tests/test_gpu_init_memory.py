"""lbm_init_fields and lbm_net_warm_start hold no device memory beyond the context's arena once
they return: the arena is all that lbm_arena_bytes and lbm_batch_arena_bytes count, and all that
a caller who passes one gives.  A second context of the same kind makes the call, so that nothing
but the call's own memory is new; what would be held is at least 16 bytes a node (33 MB)."""
import pytest

pytestmark = pytest.mark.gpu

GRID = (128, 128, 128)


def _fields():
    import torch
    x = torch.linspace(-0.5, 0.5, GRID[0], device="cuda", dtype=torch.float64)
    T = x.expand(GRID[2], GRID[1], GRID[0]).contiguous()
    return torch.zeros_like(T), torch.zeros_like(T), torch.zeros_like(T), T


def _kept(call):
    import torch
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    call()
    torch.cuda.synchronize()
    return before - torch.cuda.mem_get_info()[0]


@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("torch_arena", [True, False])
def test_rounds_keep_no_memory(precision, torch_arena):
    import torch
    import paper_1710_04751_gb300 as lbm
    from paper_1710_04751_gb300 import net
    fields = _fields()
    pred = torch.zeros((16 ** 3, 4), device="cuda")
    calls = (lambda s: s.set_fields(*fields, iterations=2), lambda s: net.warm_start(s, pred, 16, 2))
    first = lbm.LBM(GRID, 15, Ra=1e4, precision=precision, torch_arena=torch_arena)
    for call in calls:
        call(first)
    for call in calls:
        sim = lbm.LBM(GRID, 15, Ra=1e4, precision=precision, torch_arena=torch_arena)
        assert _kept(lambda: call(sim)) < 4 << 20
        sim.close()
    first.close()


def test_rounds_of_batch_members_keep_no_memory():
    import paper_1710_04751_gb300 as lbm
    fields = _fields()
    b = lbm.Batch([{"grid": GRID, "Ra": 1e4, "Pr": 0.71}] * 2, lattice=15, Ma=0.05)
    one = lbm.LBM(GRID, 15, Ra=1e4)
    one.set_fields(*fields, iterations=2)
    assert _kept(lambda: [b.member(i).set_fields(*fields, iterations=2) for i in range(b.count)]) < 4 << 20
    b.close()
    one.close()
