"""The kernels that mf_time_kernels times are those of a CG iteration."""
import numpy as np
import pytest

from paper_1901_06531_gb300 import inputs

from gpu_util import lib, neohooke_two_phase

pytestmark = pytest.mark.gpu

MASK = np.array([0, 0, 0, 1, 1, 0, 1, 1, 1], np.uint8)


@pytest.mark.parametrize("n,split", [(256, 1), (32, 1), (32, 0)])
def test_time_kernels_times_the_kernels_of_an_iteration(n, split):
    """Launches of one repetition: on split planes the fused tangent and row
    pass, the column pass, the z-pass and the two inverse passes; on others
    the tangent pass and three transform passes."""
    mf = lib()
    shape = (16, n, n)
    ph, params = neohooke_two_phase(shape, 3)
    ctx = mf.Context(n, n, 16, mf.MF_FP32_INNER)
    ctx.set_material(mf.MF_NEOHOOKE, params, ph)
    ctx.set_xy_split(split)
    ctx.constitutive()
    for graph in (False, True):
        before = mf.kernel_launches()
        ms = ctx.time_kernels(MASK, reps=3, graph=graph)
        assert mf.kernel_launches() - before == 3 * (5 if split else 4)
        assert np.all(np.isfinite(ms))
        if not graph:
            assert np.all(ms > 0)
    # the stop flag and the CG vectors are left as a solve can use them
    ctx.set_F(None)
    m, t = inputs.fix_rotation(*inputs.history_uniaxial_stress_ramp(1, 0.05))
    assert ctx.solve(m, t, 1e-8, 1e-10)["newton"][0] > 0
