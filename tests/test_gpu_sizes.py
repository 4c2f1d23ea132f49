"""The any-size transform kernels against the oracle at sizes where they can
go wrong: every pair of stage radices, one to three passes per axis, odd half
lengths and odd nz, partial z-pass tiles, planes near the shared-memory limit.
FP64 operator and residual to 1e-12
relative (one application, no iteration), the FP32 operator within its
element-wise bound, both as in the operator tests."""
import numpy as np
import pytest

from oracle import materials as omat, solver as osolver
from paper_1901_06531_gb300 import inputs

from gpu_util import fp32_operator_error, lib, neohooke_two_phase, rel

pytestmark = pytest.mark.gpu

# (nx, ny, nz), with the passes (stage radices) of nx, ny / 2 and nz
SHAPES = [
    (4, 6, 2),        # 4 | 3 | 2: one stage each
    (6, 4, 3),        # 2x3 | 2 | 3
    (18, 12, 27),     # 2x3, 3 | 2x3 | 3x3, 3
    (24, 18, 16),     # 4x2, 3 | 3x3 | 4x4
    (36, 54, 6),      # 4, 3x3 | 3x3, 3 | 2x3
    (54, 8, 81),      # 2x3, 3x3 | 4 | 3x3, 3x3
    (72, 24, 12),     # 4x2, 3x3 | 4x3 | 4x3
    (162, 4, 9),      # 2x3, 3x3, 3 (three passes along x) | 2 | 3x3
    (4, 162, 4),      # odd ny / 2 = 81
    (8, 16, 243),     # 4x2 | 4x2 | 3x3, 3x3, 3
    (16, 16, 54),     # 4x4 | 4x2 | 2x3, 3x3
    (64, 32, 4),      # 4, 4x4 | 4x4 | 4
    (256, 6, 4),      # 4x4, 4x4 | 3 | 4
    (128, 192, 2),    # the largest plane shared memory takes
    (96, 144, 2),     # 4x4, 2x3 | 4x2, 3x3 | 2
]
MASK = np.array([0, 0, 0, 1, 1, 0, 1, 1, 1], np.uint8)


@pytest.mark.parametrize("shape", SHAPES)
def test_operator_and_residual(shape):
    import torch
    mf = lib()
    nx, ny, nz = shape
    cell = (nz, ny, nx)
    ph, params = neohooke_two_phase(cell, nx + ny + nz)
    om = omat.Material(ph, omat.NEOHOOKE, params)
    F = inputs.random_F(cell, 3, 0.05)
    x = inputs.random_field(cell, 4)
    P, K = om.PK(F)
    pbar = np.array([0, 0, 0, 0.01, 0.02, 0, 0.0, 0.0, -0.01])
    ref = osolver.matvec(K, x, MASK)
    refb = osolver.residual(P, MASK, pbar)
    for prec, dt in ((mf.MF_FP64, torch.float64), (mf.MF_FP32_INNER, torch.float32)):
        ctx = mf.Context(nx, ny, nz, prec)
        ctx.set_material(mf.MF_NEOHOOKE, params, ph)
        ctx.set_F(F)
        ctx.constitutive()
        xt = torch.as_tensor(x.reshape(-1), dtype=dt, device="cuda")
        y = torch.full_like(xt, float("nan"))
        ctx.matvec(xt, y, MASK)
        got = y.cpu().numpy().astype(np.float64).reshape(ref.shape)
        if prec == mf.MF_FP64:
            assert rel(got, ref) < 1e-12
        else:
            x32 = x.astype(np.float32).astype(np.float64)
            fp32_operator_error(got, osolver.matvec(K, x32, MASK))
        b = torch.full((9 * nx * ny * nz,), float("nan"), dtype=torch.float64, device="cuda")
        ctx.residual(MASK, pbar, b)
        assert rel(b.cpu().numpy().reshape(refb.shape), refb) < 1e-12


@pytest.mark.parametrize("shape", [(18, 12, 27), (6, 4, 3), (24, 18, 16)])
def test_caller_fields_need_only_their_own_alignment(shape):
    """Fields of a caller that start 8 bytes off a 16-byte boundary: the
    residual without a context reads and writes them there, with the bits of
    the aligned call."""
    import torch
    mf = lib()
    nx, ny, nz = shape
    n9 = 9 * nx * ny * nz
    P = torch.as_tensor(inputs.random_field((nz, ny, nx), 5).reshape(-1), device="cuda")
    pbar = np.linspace(-0.1, 0.1, 9)
    aligned = torch.empty(n9, dtype=torch.float64, device="cuda")
    mf.residual_noalloc(nx, ny, nz, P, MASK, pbar, aligned)
    Pu = torch.empty(n9 + 1, dtype=torch.float64, device="cuda")[1:]
    Pu.copy_(P)
    bu = torch.full((n9 + 2,), float("nan"), dtype=torch.float64, device="cuda")
    mf.residual_noalloc(nx, ny, nz, Pu, MASK, pbar, bu[1:n9 + 1])
    assert torch.equal(bu[1:n9 + 1], aligned)
    assert bu[0].isnan() and bu[-1].isnan()


def test_cg_on_any_size_grids():
    """The residual update and the dot products inside a solve (the inverse
    pass with the CG update): FP64 and FP32-inner solves reach the oracle."""
    mf = lib()
    nx, ny, nz = 18, 12, 9
    ph, params = neohooke_two_phase((nz, ny, nx), 2)
    m, t = inputs.fix_rotation(*inputs.history_uniaxial_stress_ramp(2, 0.05))
    r = osolver.solve(omat.Material(ph, omat.NEOHOOKE, params), m, t, 1e-10, 1e-12)
    for prec, tol in ((mf.MF_FP64, 1e-10), (mf.MF_FP32_INNER, 1e-8)):
        ctx = mf.Context(nx, ny, nz, prec)
        ctx.set_material(mf.MF_NEOHOOKE, params, ph)
        out = ctx.solve(m, t, 1e-10, 1e-12, cg_rel=1e-4)
        F, _ = ctx.get_fields()
        assert np.max(np.abs(F.reshape(r["F"].shape) - r["F"])) < tol
        assert rel(out["Fbar"], r["Fbar"]) < 1e-9
