"""The step's and the adjoint's kernels at the sizes where their tiles, lanes and size rules change:
one cell more or less than a tile, odd, single and the most groups, both sides of each rule, against
the oracle.  The bars are those of the parity tests (FP64: 1e-10 in L1, 1e-8 at most; FP32 forms 1e-4
of each field's natural scale; gradients 1e-6 against the oracle's tangents)."""
import numpy as np
import pytest

import oracle
from paper_1806_07390_gb300 import workloads as W
from tests import helpers as H
from tests.test_gpu_adjoint import _random_tangent, gpu_adjoint
from tests.test_gpu_parity import FP64_L1, FP64_MAX, fxmod, run_gpu, run_oracle  # noqa: F401

pytestmark = pytest.mark.gpu


def random_case(shape, G, precision, steps=2, vterms=0):
    """A generic state (no two cells alike) with open, mirrored and periodic sides."""
    D = len(shape)
    if D == 1:
        pb, _ = W.sod_1d(n=shape[0], ngroups=G, precision=precision)
    elif D == 2:
        pb, _ = W.blobs_2d(shape=shape, ngroups=G, precision=precision)
    else:
        pb, _ = W.lognormal_3d(shape=shape, ngroups=G, precision=precision)
    pb.bc_lo = ("reflect", "outflow", "periodic")
    pb.bc_hi = ("outflow", "reflect", "periodic")
    pb.nsteps, pb.vterms, pb.c_light = steps, vterms, 5.0
    pb.dt = 0.3 / max(shape) / pb.c_light
    return pb, W.random_state(pb, seed=17, flux_frac=0.6)


# smallest grid; one group and the most; tile and chunk edges (20 x 8-lane and 256-thread tiles),
# more groups than a block's tasks hold once in 3-d; 1 to 16 lanes per cell of the FP64 interaction and
# both sides of its last step (152 x 224 cells); small and large gas-face tiles (520 x 160,
# 33 x 20 x 21, 161 x 18 x 19)
@pytest.mark.parametrize("shape,G,precision", [
    ((4,), 1, "fp64"), ((33,), 32, "fp64"), ((34049,), 2, "fp64"), ((161,), 17, "fp32"),
    ((4, 4), 32, "fp64"), ((129, 7), 3, "fp64"), ((45, 9), 7, "fp64"), ((152, 224), 2, "fp64"), ((152, 225), 3, "fp64"),
    ((4, 5), 1, "fp32"), ((21, 33), 15, "fp32"), ((41, 19), 16, "fp32n64"), ((520, 160), 1, "fp32"),
    ((19, 23), 32, "fp32"), ((4, 4, 4), 1, "fp32"), ((17, 9, 5), 13, "fp32"), ((7, 18, 6), 20, "fp32n64"),
    ((9, 5, 8), 32, "fp32"), ((6, 5, 7), 32, "fp64"), ((33, 20, 21), 2, "fp32"), ((161, 18, 19), 1, "fp64"),
])
def test_step_at_the_edges_of_tiles_and_rules(fxmod, shape, G, precision):  # noqa: F811
    pb, s = random_case(shape, G, precision)
    got, st, _ = run_gpu(fxmod, pb, state=s)
    ref, rst = run_oracle(pb, state=s)
    assert st == 0 and rst == 0
    if precision == "fp64":
        H.assert_parity(pb, got, ref, FP64_L1, FP64_MAX)
    else:
        H.assert_parity(pb, got, ref, 1e-4, natural=True)


@pytest.mark.parametrize("shape,G,precision", [((30, 11), 1, "fp32"), ((13, 35), 31, "fp32"),
                                               ((9, 8, 7), 17, "fp32n64"), ((65,), 3, "fp64")])
def test_velocity_terms_at_the_edges_of_lanes(fxmod, shape, G, precision):  # noqa: F811
    pb, s = random_case(shape, G, precision, vterms=1)
    got, st, _ = run_gpu(fxmod, pb, state=s)
    ref, rst = run_oracle(pb, state=s)
    assert st == 0 and rst == 0
    if precision == "fp64":
        H.assert_parity(pb, got, ref, FP64_L1, FP64_MAX)
    else:
        H.assert_parity(pb, got, ref, 1e-4, natural=True)


@pytest.mark.parametrize("nr,nth,G,precision", [(21, 9, 1, "fp32"), (40, 35, 19, "fp32"), (13, 8, 5, "fp64")])
def test_spherical_step_at_the_edges_of_tiles(fxmod, nr, nth, G, precision):  # noqa: F811
    pb, prim = W.spherical_2d(nr=nr, nth=nth, ngroups=G, nsteps=2, precision=precision)
    got, st, _ = run_gpu(fxmod, pb, prim)
    ref, rst = run_oracle(pb, prim)
    assert st == 0 and rst == 0
    if precision == "fp64":
        H.assert_parity(pb, got, ref, FP64_L1, FP64_MAX)
    else:
        H.assert_parity(pb, got, ref, 1e-4, natural=True)


# blocks of 256 / G faces: one group (256 faces), group counts that leave threads over, the most
@pytest.mark.parametrize("shape,G", [((9,), 1), ((40,), 12), ((23, 17), 1), ((14, 13), 7), ((7, 6), 32), ((6, 5, 4), 3)])
def test_adjoint_at_the_edges_of_blocks(fxmod, shape, G):  # noqa: F811
    pb, s = random_case(shape, G, "fp64")
    J, gs, gr, dk, after = gpu_adjoint(fxmod, pb, s, 3, 2)
    assert np.array_equal(after, s)
    t = _random_tangent(pb, s, 1)
    dkap = 0.3 * pb.kappa0
    _, Jr, dJ, _, _ = oracle.run_objective(pb, s, pb.dt, 3, tangent=t, dkappa0=dkap)
    assert abs(J - Jr) <= 1e-12 * abs(Jr)
    got = float(gs @ t) + dk * dkap
    assert abs(got - dJ) <= 1e-6 * abs(dJ), (got, dJ)


# after two steps only cells near the upper x boundary have adjoints: of the warps of one block (32 cells
# of rows of 40, 4 per warp) some have cells to work on and some have none, and kappa0's partial is
# the block's sum over both
@pytest.mark.parametrize("shape,G,couple", [((40, 9), 2, 1), ((40, 9), 2, 0), ((67,), 20, 1)])
def test_adjoint_where_warps_of_a_block_are_idle(fxmod, shape, G, couple):  # noqa: F811
    pb, s = random_case(shape, G, "fp64")
    pb.couple = couple
    J, gs, gr, dk, _ = gpu_adjoint(fxmod, pb, s, 2, 1)
    g = gs[:pb.ncell].reshape(pb.shape)
    assert np.all(g[..., :20] == 0.0) and np.all(g[..., -1] != 0.0)
    t = _random_tangent(pb, s, 1)
    dkap = 0.3 * pb.kappa0
    _, Jr, dJ, _, _ = oracle.run_objective(pb, s, pb.dt, 2, tangent=t, dkappa0=dkap)
    assert abs(J - Jr) <= 1e-12 * abs(Jr)
    got = float(gs @ t) + dk * dkap
    assert abs(got - dJ) <= 1e-6 * abs(dJ), (got, dJ)
    _, _, dJk, _, _ = oracle.run_objective(pb, s, pb.dt, 2, tangent=np.zeros_like(t), dkappa0=dkap)
    assert abs(dk * dkap - dJk) <= 1e-6 * abs(dJk), (dk * dkap, dJk)


# A Cartesian grid's coefficients depend on its cell width alone: moved by 2^20 widths of the domain, the same
# state gives the same step and the same gradient, bit for bit.
@pytest.mark.parametrize("shape,G,precision", [((75,), 3, "fp64"), ((45, 37), 2, "fp64"), ((9, 11, 7), 2, "fp64"),
                                               ((45, 37), 3, "fp32n64")])
def test_step_and_gradient_do_not_depend_on_the_origin(fxmod, shape, G, precision):  # noqa: F811
    pb, s = random_case(shape, G, precision)
    got, J = [], []
    for x0 in (0.0, 2.0 ** 20):
        pb.x_lo, pb.x_hi = (x0,) * 3, (x0 + 1.0,) * 3
        state, st, _ = run_gpu(fxmod, pb, state=s)
        assert st == 0
        j, gs, _, dk, _ = gpu_adjoint(fxmod, pb, s, 2, 1)
        got.append((state, gs))
        J.append((j, dk))
    np.testing.assert_array_equal(got[0][0], got[1][0])
    # (the adjoint's atomic sums come in any order)
    np.testing.assert_allclose(got[0][1], got[1][1], rtol=0.0, atol=(1e-13 if precision == "fp64" else 1e-5) * np.max(np.abs(got[0][1])))
    np.testing.assert_allclose(J[0], J[1], rtol=1e-12 if precision == "fp64" else 1e-5)


def test_face_buffer_past_32_bit_offsets(fxmod):  # noqa: F811
    # 3-d with the velocity terms: the face buffer's third direction begins past 2^32 elements on the largest
    # grids that are accepted (236e6 cells; 71 GB here).  A state of period 8 along z steps like the small
    # grid of one period.
    import torch
    pb, s = random_case((4, 24, 8), 1, "fp32", steps=1, vterms=1)
    pb.bc_lo, pb.bc_hi = ("reflect", "outflow", "periodic"), ("outflow", "reflect", "periodic")
    pb.dt = 0.3 / 24 / pb.c_light
    pb.x_lo, pb.x_hi = (0.0,) * 3, (1.0, 1.0, 1.0)
    ref, st, _ = run_gpu(fxmod, pb, state=s)
    assert st == 0
    reps = 306875
    pb.n, pb.x_hi = (4, 24, 8 * reps), (1.0, 1.0, float(reps))
    assert 8 * (5 * 24 + 4 * 25) * 8 * reps >= 2 ** 32
    fields = torch.from_numpy(s.astype(np.float32)).cuda().reshape(9, 1, -1)
    g = fxmod.Grid(pb)
    state = fields.expand(9, reps, fields.shape[2]).contiguous().reshape(-1)
    g.upload(state)
    g.step(pb.dt, 1)
    assert g.status() == 0
    g.download(state)
    g.close()
    out, want = state.reshape(9, reps, -1), torch.from_numpy(ref).cuda().to(torch.float32).reshape(9, -1)
    for v in range(9):
        scale = float(want[v].abs().max())
        assert float((out[v] - want[v]).abs().max()) <= 1e-5 * scale, v
