"""lbm_net_targets (one pass, float-pair sums in the single-precision forms) against the FP64
fields of lbm_fields, for every storage form, both scalar lattices, odd grids, sources and
forces, a misaligned output and non-finite populations.

Tolerance: the FP32 result may round differently by one unit in the last place
(2^-23 |value|); the pair sums carry 2^-44 of the summed magnitudes (below 4 for the
populations of one node), divided by U0 for the velocities."""
import ctypes
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

GRIDS = [(2, 1, 1), (5, 4, 3), (33, 17, 9), (70, 3, 3), (64, 16, 2)]


def _reference(sim):
    f = sim.fields()
    u0 = sim.params()["U0"]
    return np.stack([f["ux"] / u0, f["uy"] / u0, f["uz"] / u0, 2.0 * f["T"]], -1).reshape(-1, 4), u0


def _check(got, ref, u0):
    tol = 2.0 ** -23 * np.abs(ref) + 4 * 2.0 ** -44 * np.array([1 / u0, 1 / u0, 1 / u0, 2.0])
    assert (np.abs(got.astype(np.float64) - ref) <= tol).all()


@pytest.mark.parametrize("grid", GRIDS)
@pytest.mark.parametrize("lattice", [15, 7])
@pytest.mark.parametrize("precision", [0, 1, 2, 3])
def test_targets_equal_the_fp64_fields(grid, lattice, precision):
    import paper_1710_04751_gb300 as lbm
    from paper_1710_04751_gb300 import net
    p = lbm.derive_params(grid, lattice, 1e3, 0.71, 0.05 * math.sqrt(3.0))
    p.heat_source = 1e-3
    p.ext_force[0], p.ext_force[1], p.ext_force[2] = 1e-4, -2e-4, 3e-4
    p.T_hot, p.T_cold = 0.7, -0.4
    sim = lbm.LBM(grid, lattice, params=p, precision=precision, noise_amp=0.3, seed=5)
    sim.step(7)
    ref, u0 = _reference(sim)
    _check(net.targets(sim).cpu().numpy(), ref, u0)
    sim.close()


def test_targets_into_a_misaligned_buffer():
    import torch
    import paper_1710_04751_gb300 as lbm
    from paper_1710_04751_gb300 import net
    sim = lbm.LBM((13, 7, 5), 15, Ra=1e3, noise_amp=0.2)
    sim.step(3)
    buf = torch.full((4 * sim.ncell + 2,), 7.0, device="cuda")
    sim._check(net._lib().lbm_net_targets(sim._ctx, ctypes.c_void_p(buf.data_ptr() + 4)))
    out = buf.cpu().numpy()
    assert out[0] == 7.0 and out[-1] == 7.0
    assert np.array_equal(out[1:-1].reshape(-1, 4), net.targets(sim).cpu().numpy())
    sim.close()


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan, 3.0e38])
def test_targets_of_non_finite_populations(value):
    import paper_1710_04751_gb300 as lbm
    from paper_1710_04751_gb300 import net
    sim = lbm.LBM((8, 6, 4), 15, Ra=1e3, noise_amp=0.2)
    f, g = sim.get_populations_native()
    f[3, 1, 2, 3] = value
    g[9, 2, 4, 5] = value
    f[:, 3, 1, 1] = 0.0
    sim.set_populations_native(f, g)
    with np.errstate(all="ignore"):
        ref = _reference(sim)[0].astype(np.float32)
    assert np.array_equal(net.targets(sim).cpu().numpy()[~np.isfinite(ref)], ref[~np.isfinite(ref)], equal_nan=True)
    assert (np.isfinite(net.targets(sim).cpu().numpy()) == np.isfinite(ref)).all()
    sim.close()
