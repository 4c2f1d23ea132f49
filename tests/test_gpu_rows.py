"""The FP32 tangent pass fused with the x transform (split x-y planes): the
operator and a solve on it, for both laws, with and without a voxel scale, on
the smallest and the largest plane it serves, against the same cell on the
other kernels.  Operators agree within twice the element-wise FP32 bound
(each side within c log2(N) eps32 max|y| of the exact product), converged
fields within twice the FP32-inner field tolerance of 1e-8."""
import numpy as np
import pytest

from oracle import materials as omat, solver as osolver
from paper_1901_06531_gb300 import inputs

from gpu_util import EPS32, fp32_operator_error, lib, neohooke_two_phase, polycrystal

pytestmark = pytest.mark.gpu

MASK = np.array([0, 0, 0, 1, 1, 0, 1, 1, 1], np.uint8)


def cell(mf, shape, law, scale):
    nx, ny, nz = shape
    ctx = mf.Context(nx, ny, nz, mf.MF_FP32_INNER)
    zyx = (nz, ny, nx)
    sc = inputs.lognormal_scale(zyx, 0.3, 5) if scale else None
    if law == "nh":
        ph, params = neohooke_two_phase(zyx, 4)
        ctx.set_material(mf.MF_NEOHOOKE, params, ph, scale=sc)
    else:
        ph, params, R = polycrystal(zyx, 5, 4)
        ctx.set_material(mf.MF_SVK_CUBIC, params, ph, rot=R, scale=sc)
    return ctx


@pytest.mark.parametrize("law", ["nh", "svk"])
@pytest.mark.parametrize("scale", [False, True])
def test_operator_of_split_and_fused_planes(law, scale):
    import torch
    mf = lib()
    shape = (32, 32, 16)
    F = inputs.random_F(shape[::-1], 6, 0.05)
    x = torch.as_tensor(inputs.random_field(shape[::-1], 7).reshape(-1), dtype=torch.float32, device="cuda")
    got = []
    for split in (0, 1):
        ctx = cell(mf, shape, law, scale)
        ctx.set_xy_split(split)
        ctx.set_F(F)
        ctx.constitutive()
        y = torch.full_like(x, float("nan"))
        ctx.matvec(x, y, MASK)
        got.append(y.cpu().numpy().astype(np.float64))
    bound = 2 * 2 * np.log2(x.numel() / 9) * EPS32 * np.max(np.abs(got[0]))
    assert np.max(np.abs(got[1] - got[0])) <= bound


def test_operator_on_the_largest_plane():
    import torch
    mf = lib()
    shape = (256, 256, 16)
    zyx = shape[::-1]
    ph, params = neohooke_two_phase(zyx, 4)
    ctx = cell(mf, shape, "nh", False)
    F = inputs.random_F(zyx, 6, 0.05)
    ctx.set_F(F)
    ctx.constitutive()
    x = inputs.random_field(zyx, 7).astype(np.float32)
    xt = torch.as_tensor(x.reshape(-1), device="cuda")
    y = torch.full_like(xt, float("nan"))
    ctx.matvec(xt, y, MASK)
    _, K = omat.Material(ph, omat.NEOHOOKE, params).PK(F)
    fp32_operator_error(y.cpu().numpy().reshape(x.shape), osolver.matvec(K, x.astype(np.float64), MASK))


@pytest.mark.parametrize("law", ["nh", "svk"])
def test_solve_on_split_planes(law):
    mf = lib()
    m, t = inputs.fix_rotation(*inputs.history_uniaxial_stress_ramp(2, 0.05 if law == "nh" else 0.2))
    got = []
    for split in (0, 1):
        ctx = cell(mf, (32, 32, 16), law, False)
        ctx.set_xy_split(split)
        out = ctx.solve(m, t, 1e-10, 1e-12, cg_rel=1e-4)
        got.append((ctx.get_fields()[0], out))
    assert np.max(np.abs(got[0][0] - got[1][0])) < 2e-8
    assert np.max(np.abs(got[0][1]["Fbar"] - got[1][1]["Fbar"])) < 2e-9
