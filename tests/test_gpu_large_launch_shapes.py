"""The line-resident x passes with four line groups a warp, against the FP64 oracle.

Grids of more than 9728 line groups take that shape: a warp reuses its line buffers
from group to group and prefetches the next one's rows, and problems that share a
velocity loop inside the solute kernel. Line lengths that reach it on grids of up to
512 x 512 lines: 64 and more voxels in FP32, 16 and more in FP64. Two iterations of
each solver, both symbol sets; tolerances as in the parity tests, and the three-load
solute solve, whose loads share launches, against single ones.
"""
import numpy as np
import pytest
import torch

from oracle import acm_oracle as O
from paper_2312_15554_gb300 import inputs as I

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def relerr(a, b):
    return float(np.abs(np.asarray(a) - b).max() / np.abs(b).max())


@pytest.mark.parametrize("shape,fp64", [((512, 512, 16), True), ((512, 256, 32), True), ((512, 256, 64), True),
                                        ((512, 512, 64), False), ((512, 256, 128), False), ((128, 256, 512), False)])
def test_x_passes_with_four_groups_a_warp(lib, shape, fp64):
    lanes = {16: 2, 32: 4, 64: 4} if fp64 else {64: 2, 128: 4, 512: 16}
    assert shape[0] * shape[1] // (32 // lanes[shape[2]]) >= 9728
    H = I.random_indicator(shape, 0.35, 21)
    Hd = torch.as_tensor(H, device=DEV)
    dt = torch.float64 if fp64 else torch.float32
    pr = lib.FP64 if fp64 else lib.FP32
    tol = 1e-10 if fp64 else 1e-5
    g = [1.0, 0.25, -0.5]
    pen = dict(eps=0.0, max_iter=2, alpha0=250.0, beta0=180.0, b0=300.0)
    R = O.stokes(H, g, O.StokesParams(adaptive=False, **pen))
    ctx = lib.acm_ctx(shape)
    u = torch.zeros((3,) + shape, dtype=dt, device=DEV)
    lam = torch.zeros_like(u)
    _, _, rep = lib.acm_stokes(ctx, Hd, g, lib.stokes_params(adaptive=0, precision=pr, **pen), None, None, u, None, lam)
    assert relerr(u.cpu().numpy(), R.state.u) < tol
    assert relerr(lam.cpu().numpy(), R.state.lam) < tol
    np.testing.assert_allclose(rep.res[:6], R.residuals[-1], rtol=1e-8 if fp64 else 2.5e-4)
    uo = R.state.u / np.abs(R.state.u).max()
    ud = torch.as_tensor(uo, dtype=dt, device=DEV)
    for deriv in (O.CENTRAL, O.EXACT):
        prm = lib.advdiff_params(eps=0.0, max_iter=2, precision=pr, deriv=deriv)
        chi = torch.zeros((3,) + shape, dtype=dt, device=DEV)
        one = torch.zeros(shape, dtype=dt, device=DEV)
        lib.acm_advdiff_tensor(ctx, Hd, ud, 10.0, prm, chi)
        for j in range(3):
            lib.acm_advdiff(ctx, Hd, ud, 10.0, [1.0 if c == j else 0.0 for c in range(3)], prm, one)
            assert float((chi[j] - one).abs().max()) <= (1e-12 if fp64 else 1e-6) * float(one.abs().max())
        Rc = O.advdiff(H, uo, 10.0, [0.0, 0.0, 1.0], O.AdvDiffParams(eps=0.0, max_iter=2, deriv=deriv))
        assert relerr(one.cpu().numpy(), Rc.chi) < tol
    ctx.close()
