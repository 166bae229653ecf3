"""States at the limits of what the step takes.  Bars of the parity tests (FP64: 1e-10 in L1, 1e-8 at
most).

The M1 closure where |F| exceeds cE by so much that |F|^2 / (cE)^2 overflows: cold cells lie at the
energy floor (1e-300 by default) or in the Wien tail, and a flux can reach them a step before its
energy does.  The closure keeps its clamped value there.

Cells whose pressure is negative (total energy below the kinetic energy: strong rarefactions, or a
snapshot): the sound speed of such a face state is NaN, and the wave speeds come from the averages
alone until the interaction's floor restores the pressure."""
import numpy as np
import pytest

from paper_1806_07390_gb300 import workloads as W
from tests import helpers as H
from tests.test_gpu_kernel_sizes import random_case
from tests.test_gpu_parity import FP64_L1, FP64_MAX, fxmod, run_gpu, run_oracle  # noqa: F401

pytestmark = pytest.mark.gpu


# f^2 = (|F| / cE)^2 just below and above 2^1022 and far past the largest double
@pytest.mark.parametrize("energy", [1e-152, 1e-156, 1e-250, 1e-300])
@pytest.mark.parametrize("shape", [(24,), (13, 12), (9, 8, 7)])
def test_flux_far_above_the_free_streaming_limit(fxmod, shape, energy):  # noqa: F811
    pb, s = random_case(shape, 3, "fp64")
    N, G, NG = pb.ncell, pb.ngroups, 2 + pb.dims
    E = s[NG * N:(NG + G) * N].reshape(pb.shape + (G,))
    # a block of cells wide enough that the reconstruction leaves face states of its value
    E[tuple(slice(1, 7) for _ in pb.shape) + (1,)] = energy
    got, st, _ = run_gpu(fxmod, pb, state=s)
    ref, rst = run_oracle(pb, state=s)
    assert np.all(np.isfinite(ref))
    assert st == 0 and rst == 0
    H.assert_parity(pb, got, ref, FP64_L1, FP64_MAX)


def test_fronts_that_meet_in_cold_gas(fxmod):  # noqa: F811
    # radiation at T = 1 runs from both sides into 31 cells of gas and radiation at T = 0.004, whose
    # upper group holds 1e-197
    pb, _ = W.sod_1d(n=64, ngroups=4, precision="fp64")
    pb.bc_lo = pb.bc_hi = ("periodic",) * 3
    pb.kappa0, pb.kap_rho_exp, pb.kap_T_exp, pb.kap_eps_exp, pb.sigma0 = 1.0, 0, 0, 0, 0.0
    pb.c_light, pb.nsteps = 20.0, 45
    pb.dt = 0.4 / 64 / pb.c_light
    prim = np.zeros((4, 64))
    prim[0], prim[1], prim[3] = 1.0, 0.004, 1.0
    prim[3, 16:47] = 0.004
    got, st, _ = run_gpu(fxmod, pb, prim)
    ref, rst = run_oracle(pb, prim)
    assert np.all(np.isfinite(ref))
    assert st == 0 and rst == 0
    H.assert_parity(pb, got, ref, FP64_L1, FP64_MAX)


# Isolated cells inside the grid (beside a boundary their ghosts would repeat them, and two such states
# leave no wave speeds at all) that hold nine tenths of their kinetic energy, or all but one part in 1e12.
# The local Lax-Friedrichs solver has no speeds of its own for them, in the oracle either.
@pytest.mark.parametrize("precision,part", [("fp64", 0.9), ("fp64", 1.0 - 1e-12), ("fp32", 0.9), ("fp32n64", 0.9)])
@pytest.mark.parametrize("shape,solver", [((50,), "hllc"), ((23, 19), "hllc"), ((23, 19), "hlle"), ((9, 8, 7), "hllc")])
def test_cells_with_negative_pressure(fxmod, shape, solver, precision, part):  # noqa: F811
    pb, s = random_case(shape, 2, precision, steps=1)
    pb.riemann = solver
    N, D = pb.ncell, pb.dims
    cells = np.arange(N).reshape(pb.shape)[tuple(slice(2, -2, 3) for _ in pb.shape)].reshape(-1)
    ke = 0.5 * sum(s[(1 + q) * N:(2 + q) * N] ** 2 for q in range(D)) / s[:N]
    s[(1 + D) * N + cells] = part * ke[cells]
    ref, rst = run_oracle(pb, state=s)
    assert np.all(np.isfinite(ref)) and rst == 0
    got, st, _ = run_gpu(fxmod, pb, state=s)
    assert np.all(np.isfinite(got)) and st == 0
    if precision == "fp64":
        H.assert_parity(pb, got, ref, FP64_L1, FP64_MAX)
    else:
        H.assert_parity(pb, got, ref, 1e-4, natural=True)


# Gas far colder than the upper groups' band edges (eps/T up to 1e6): their Planck energies are 0 in FP32.
# The radiation heats it by several orders of magnitude within the step.
@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp32n64"])
@pytest.mark.parametrize("G", [1, 15, 16])
def test_gas_far_below_the_groups(fxmod, G, precision):  # noqa: F811
    pb, prim = W.kh_2d(nx=24, ny=20, ngroups=G, nsteps=2, precision=precision)
    prim = np.array(prim)
    prim[1] = prim[0] * 10.0 ** np.random.default_rng(4).uniform(-5.0, -3.0, pb.ncell)
    prim[-1] = 0.3
    ref, rst = run_oracle(pb, prim)
    assert np.all(np.isfinite(ref)) and rst == 0
    got, st, _ = run_gpu(fxmod, pb, prim)
    assert np.all(np.isfinite(got)) and st == 0
    if precision == "fp64":
        H.assert_parity(pb, got, ref, FP64_L1, FP64_MAX)
    else:
        H.assert_parity(pb, got, ref, 1e-4, natural=True)
