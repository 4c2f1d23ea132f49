"""The range of the squared residual inside a FP32-inner CG solve on any-size
grids: r.r is summed in FP64 from the first term on, so that a solve whose
residuals square below the FP32 range takes the course of the same solve in
ordinary units.

The adjoint system A lambda = G*(K : W) is linear in W and K scales out of
lambda: with K times 2^46 and W times 2^-107 the right-hand side is 2^-61
times the unscaled one (about 1e-18, its squares within FP32), every vector
of the solve is a power of two times its unscaled counterpart, and the
residual ends near 1e-24, whose squares are zero in FP32.  Powers of two
round alike, so iterations and gradients agree up to the last bits of the
dot product p.Kp (its FP32 products lose theirs below 2^-126): one iteration
and ten times the solve's relative residual of 1e-6."""
import numpy as np
import pytest

from paper_1901_06531_gb300 import inputs

from gpu_util import lib, neohooke_two_phase

pytestmark = pytest.mark.gpu

MASK = np.array([0, 0, 0, 1, 0, 0, 1, 1, 0], np.uint8)


@pytest.mark.parametrize("shape", [(36, 24, 18), (72, 54, 12)])
def test_small_units_take_the_same_course(shape):
    mf = lib()
    nx, ny, nz = shape
    cell = (nz, ny, nx)
    ph, params = neohooke_two_phase(cell, 3)
    W = np.array([0.3, -0.2, 0.5, 0.1, 0.4, -0.1, 0.2, 0.6, -0.3])
    got = []
    for kscale, wscale in ((1.0, 1.0), (2.0 ** 46, 2.0 ** -107)):
        ctx = mf.Context(nx, ny, nz, mf.MF_FP32_INNER)
        ctx.set_material(mf.MF_NEOHOOKE, kscale * params, ph)
        ctx.set_F(inputs.random_F(cell, 6, 0.02))
        J, grad, its = ctx.adjoint(MASK, np.zeros(9), wscale * W, tol_cg=1e-200, cg_rel=1e-6)
        got.append((grad / wscale, its))
    (g0, i0), (g1, i1) = got
    assert i0 > 10 and abs(i1 - i0) <= 1
    assert np.max(np.abs(g1 - g0)) <= 1e-5 * np.max(np.abs(g0))


def test_solve_on_a_larger_grid_against_fp64():
    """Partial sums of several hundred planes: the FP32-inner solve ends within
    its field tolerance of 1e-8 of the plain FP64 one."""
    mf = lib()
    nx, ny, nz = 72, 54, 36
    ph, params = neohooke_two_phase((nz, ny, nx), 5)
    m, t = inputs.fix_rotation(*inputs.history_uniaxial_stress_ramp(2, 0.05))
    got = []
    for prec in (mf.MF_FP64, mf.MF_FP32_INNER):
        ctx = mf.Context(nx, ny, nz, prec)
        ctx.set_material(mf.MF_NEOHOOKE, params, ph)
        out = ctx.solve(m, t, 1e-10, 1e-12, cg_rel=1e-4)
        got.append((ctx.get_fields()[0], out["Fbar"]))
    assert np.max(np.abs(got[1][0] - got[0][0])) < 1e-8
    assert np.max(np.abs(got[1][1] - got[0][1])) < 1e-9
