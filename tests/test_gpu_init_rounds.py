"""The fused rounds of lbm_init_fields (one step and the reimposition in one kernel, cavities at
the paper's unit higher-order rates in FP64 and FP32) against the rounds as two kernels, and
the resampling behind lbm_net_warm_start against the oracle's.

FP64: the two-kernel rounds are reached by moving one unit rate by 2^-50, which changes a moment
by 2^-50 of itself; both forms round each of the `rounds` updates of values below 1 a few times:
1e-13 covers 4 rounds of some hundred roundings of 2^-53.  FP32: against the FP64 rounds, within
1e-5 of max(|p|, rest weight), the single-precision parity bound of the step itself."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

GRIDS = [(2, 2, 2), (5, 4, 3), (33, 7, 5), (130, 3, 4), (64, 5, 6)]


def _run(grid, lattice, precision, nudge, e4_mode, rounds):
    import torch
    import paper_1710_04751_gb300 as lbm
    p = lbm.derive_params(grid, lattice, 2e3, 0.71, 0.05 * math.sqrt(3.0), e4_mode=e4_mode)
    p.heat_source = 2e-4
    p.ext_force[0], p.ext_force[1], p.ext_force[2] = 1e-4, -2e-4, 5e-5
    p.T_hot, p.T_cold = 0.6, -0.4
    if nudge:
        p.omega_f[14] = 1.0 + 2.0 ** -50
    sim = lbm.LBM(grid, lattice, params=p, precision=precision)
    g = torch.Generator().manual_seed(11)
    shape = (grid[2], grid[1], grid[0])
    u = [(0.03 * torch.randn(shape, generator=g, dtype=torch.float64)).cuda() for _ in range(3)]
    T = (torch.rand(shape, generator=g, dtype=torch.float64) - 0.5).cuda()
    rho = (1 + 0.02 * torch.randn(shape, generator=g, dtype=torch.float64)).cuda()
    sim.set_fields(*u, T, rho=rho, iterations=rounds)
    out = sim.get_populations()
    sim.close()
    return out


@pytest.mark.parametrize("grid", GRIDS)
@pytest.mark.parametrize("lattice,e4_mode", [(15, 0), (15, 1), (7, 0)])
def test_fused_rounds_equal_two_kernel_rounds(grid, lattice, e4_mode):
    two = _run(grid, lattice, 0, True, e4_mode, 4)
    one = _run(grid, lattice, 0, False, e4_mode, 4)
    for a, b in zip(one, two):
        assert np.abs(a - b).max() <= 1e-13
    single = _run(grid, lattice, 1, False, e4_mode, 4)
    for a, b, w in zip(single, two, (1 / 72, 1 / 72 if lattice == 15 else 1 / 8)):
        assert (np.abs(a - b) <= 1e-5 * np.maximum(np.abs(b), w)).all()


@pytest.mark.parametrize("m,grid", [(1, (3, 4, 5)), (2, (2, 3, 70)), (5, (129, 4, 3)), (16, (16, 16, 16)),
                                    (9, (4, 18, 17))])
def test_resampling_at_the_edges_of_its_tiles(m, grid):
    import torch
    import paper_1710_04751_gb300 as lbm
    from oracle import nn_oracle as nno
    from paper_1710_04751_gb300 import net
    sim = lbm.LBM(grid, 15, Ra=1e3, precision=lbm.FP64)
    pred = np.random.default_rng(m).uniform(-1, 1, (m ** 3, 4)).astype(np.float32)
    net.warm_start(sim, torch.as_tensor(pred).cuda(), m)
    f = sim.fields()
    U0 = sim.params()["U0"]
    ref = nno.trilinear(pred.astype(np.float64), m, *grid)
    Fz = 0.5 * sim.params()["gbeta"] * f["T"]  # lbm_fields takes half the force off the momentum
    for got, want in ((f["ux"], U0 * ref[..., 0]), (f["uy"], U0 * ref[..., 1]),
                      (f["uz"] + Fz / f["rho"], U0 * ref[..., 2]), (f["T"], 0.5 * ref[..., 3])):
        assert np.abs(got - want).max() <= 1e-13
    sim.close()
