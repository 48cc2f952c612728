"""lbm_step in short runs of equal and changing lengths (the run graphs) against one long call:
the same states, step counts and residuals, in every storage form, odd and even run lengths,
with and without residual checks."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1, 2, 3])
@pytest.mark.parametrize("interval", [0, 7, 20])
def test_runs_of_steps_equal_one_call(precision, interval):
    import paper_1710_04751_gb300 as lbm
    kw = dict(Ra=2e3, precision=precision, noise_amp=0.1, residual_interval=interval)
    runs = [5] * 4 + [6] * 3 + [5, 5, 130, 130, 4, 4, 4, 3, 3, 1, 1, 20, 20, 20]
    a, b = lbm.LBM((12, 9, 7), 15, **kw), lbm.LBM((12, 9, 7), 15, **kw)
    for n in runs:
        a.step(n)
    b.step(sum(runs))
    assert a.steps_done == b.steps_done == sum(runs)
    assert a.residual() == b.residual()
    for x, y in zip(a.get_populations(), b.get_populations()):
        assert np.array_equal(x, y)
    a.close()
    b.close()


def test_runs_recorded_into_the_callers_graph():
    import torch
    import paper_1710_04751_gb300 as lbm
    kw = dict(Ra=2e3, precision=lbm.FP32, noise_amp=0.1, residual_interval=0)
    st = torch.cuda.Stream()
    a, b = lbm.LBM((12, 9, 7), 15, stream=st, **kw), lbm.LBM((12, 9, 7), 15, **kw)
    for _ in range(3):
        a.step(8)  # by now a graph of the library's own
    a.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        a.step(8)
        a.step(6)
        a.step(6)
    with torch.cuda.stream(st):
        g.replay()
        g.replay()
    b.step(24 + 2 * 20)
    for x, y in zip(a.get_populations(), b.get_populations()):
        assert np.array_equal(x, y)
    a.step(8)
    b.step(8)
    for x, y in zip(a.get_populations(), b.get_populations()):
        assert np.array_equal(x, y)
    a.close()
    b.close()


def test_runs_of_a_new_length_do_not_wait_for_the_old_ones():
    import paper_1710_04751_gb300 as lbm
    kw = dict(Ra=2e3, precision=lbm.FP32, noise_amp=0.1, residual_interval=0)
    a, b = lbm.LBM((96, 96, 96), 15, **kw), lbm.LBM((96, 96, 96), 15, **kw)
    runs = [100, 100, 100, 90, 90, 80, 80, 80, 100, 100]
    a.set_timeout(1e-9)  # any wait for the GPU would run out
    for n in runs:
        a.step(n)
    a.set_timeout(600.0)
    a.synchronize()
    a.step(80)
    b.step(sum(runs) + 80)
    for x, y in zip(a.get_populations(), b.get_populations()):
        assert np.array_equal(x, y)
    a.close()
    b.close()
