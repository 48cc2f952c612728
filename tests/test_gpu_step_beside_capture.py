"""lbm_step on a stream of its own while the same thread captures another stream in the global mode
(torch.cuda.graph's): the steps run at once, and the capture is not disturbed, whether the context
has its graphs of runs already or makes them then."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

RUNS = (8, 8, 8, 6, 6, 6, 6, 5, 5)


@pytest.mark.parametrize("before", [0, 3])
def test_steps_beside_a_capture(before):
    import torch
    import paper_1710_04751_gb300 as lbm
    kw = dict(Ra=2e3, precision=lbm.FP32, noise_amp=0.1, residual_interval=0)
    a, b = lbm.LBM((12, 9, 7), 15, stream=torch.cuda.Stream(), **kw), lbm.LBM((12, 9, 7), 15, **kw)
    for _ in range(before):
        a.step(8)
    a.synchronize()
    x = torch.zeros(1000, device="cuda")
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        x.add_(1)
        for n in RUNS:
            a.step(n)
        x.add_(1)
    a.synchronize()
    assert x.sum() == 0
    g.replay()
    assert (x == 2).all()
    b.step(8 * before + sum(RUNS))
    assert a.steps_done == b.steps_done
    for p, q in zip(a.get_populations(), b.get_populations()):
        assert np.array_equal(p, q)
    a.close()
    b.close()
