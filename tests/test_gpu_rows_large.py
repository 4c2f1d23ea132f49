"""The FP32 tangent pass fused with the x transform on 256 x 256 planes under
the SVK law: the operator against the oracle within its element-wise bound, a
solve whose groups of rows outnumber the resident blocks (each block walks
over several groups and refills its buffers) against the plain FP64 solve of
the same cell within the FP32-inner field tolerance of 1e-8."""
import numpy as np
import pytest

from oracle import materials as omat, solver as osolver
from paper_1901_06531_gb300 import inputs

from gpu_util import fp32_operator_error, lib, polycrystal

pytestmark = pytest.mark.gpu

MASK = np.array([0, 0, 0, 1, 1, 0, 1, 1, 1], np.uint8)
SHAPE = (16, 256, 256)


def test_svk_operator_on_the_largest_plane():
    import torch
    mf = lib()
    ph, params, R = polycrystal(SHAPE, 5, 4)
    ctx = mf.Context(256, 256, 16, mf.MF_FP32_INNER)
    ctx.set_material(mf.MF_SVK_CUBIC, params, ph, rot=R)
    F = inputs.random_F(SHAPE, 6, 0.05)
    ctx.set_F(F)
    ctx.constitutive()
    x = inputs.random_field(SHAPE, 7).astype(np.float32)
    xt = torch.as_tensor(x.reshape(-1), device="cuda")
    y = torch.full_like(xt, float("nan"))
    ctx.matvec(xt, y, MASK)
    _, K = omat.Material(ph, omat.SVK_CUBIC, params, R).PK(F)
    fp32_operator_error(y.cpu().numpy().reshape(x.shape), osolver.matvec(K, x.astype(np.float64), MASK))


def test_svk_solve_on_the_largest_plane():
    mf = lib()
    ph, params, R = polycrystal(SHAPE, 5, 4)
    m, t = inputs.fix_rotation(*inputs.history_uniaxial_stress_ramp(1, 0.2))
    got = []
    for prec in (mf.MF_FP64, mf.MF_FP32_INNER):
        ctx = mf.Context(256, 256, 16, prec)
        ctx.set_material(mf.MF_SVK_CUBIC, params, ph, rot=R)
        if prec == mf.MF_FP64:
            ctx.set_inexact_newton(1)
        ctx.solve(m, t, 1e-10, 1e-12, cg_rel=1e-4)
        got.append(ctx.get_fields()[0])
        del ctx
    assert np.max(np.abs(got[1] - got[0])) < 1e-8
