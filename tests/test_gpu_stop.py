"""After a CG solve has stopped, the kernels of an iteration that was already
queued return without touching memory: the loop body holds two iterations, so
a solve that stops in the first one leaves the second to return at once.

Checked on the fused FP32 plane kernels of every plane size (their row
transform has one stage on 16 and 32 squared planes, two on the others)
through the buffers those kernels write: a solve of one iteration from the
right-hand side G*(K : W) leaves K : p and its projected spectrum in the
workspace, where an operator application to p = G*(K : W) leaves the same
values.  A forward pass that runs after the stop would have put the
unprojected, unscaled spectrum there, N times larger."""
import numpy as np
import pytest

from paper_1901_06531_gb300 import inputs

from gpu_util import lib, neohooke_two_phase

pytestmark = pytest.mark.gpu

MASK = np.array([0, 0, 0, 1, 0, 0, 1, 1, 0], np.uint8)   # no rigid rotation left free


@pytest.mark.parametrize("n", [16, 32, 48, 64, 96])
def test_no_pass_writes_after_the_stop(n):
    import torch
    mf = lib()
    shape = (16, n, n)
    ctx = mf.Context(n, n, 16, mf.MF_FP32_INNER)
    ph, params = neohooke_two_phase(shape, 3)
    ctx.set_material(mf.MF_NEOHOOKE, params, ph)
    ctx.autotune()
    ctx.set_F(inputs.random_F(shape, 6, 0.02))
    ctx.constitutive()
    W = np.array([0.3, -0.2, 0.5, 0.1, 0.4, -0.1, 0.2, 0.6, -0.3])
    w = torch.as_tensor(np.repeat(W, ctx.N), dtype=torch.float32, device="cuda")
    p, y = torch.empty_like(w), torch.empty_like(w)
    ctx.matvec(w, p, MASK)
    snap = lambda: ctx.workspace[:ctx.workspace.numel() // 4 * 4].view(torch.float32).clone()  # noqa: E731
    ctx.matvec(w, y, MASK)
    a = snap()
    ctx.matvec(p, y, MASK)
    want = snap()
    where = (a.view(torch.int32) != want.view(torch.int32)).nonzero().reshape(-1)
    # K : p and the spectrum, 9N floats each, but for the spectrum's zeros in
    # both: y-Nyquist rows, and where kx or ky is zero one component of three
    # (together 2/n of it)
    assert 16 * ctx.N < where.numel() <= 18 * ctx.N
    try:
        ctx.adjoint(MASK, np.zeros(9), W, tol_cg=1e-30, cg_rel=1e-6, max_cg=1)
    except mf.MixFFTError as e:
        assert e.status == mf.MF_NOT_CONVERGED
    got = snap()
    err = (got[where] - want[where]).abs().max().item()
    # FP32 rounding of the two applications, against a factor of N
    assert err <= 1e-4 * want[where].abs().max().item()
