"""Every launch shape of the line-resident x passes against the FP64 oracle.

The x passes pick warps per block, line groups per warp and a split by
component from the number of line groups of the grid, and FP64 lines below 256
voxels are split over more lanes than FP32 ones. The grids here give one, two,
four and eight warps a block with one group each, with and without the
component split, in both precisions. Tolerances as in the parity tests: FP64
1e-10, FP32 fields 1e-5 of the largest magnitude.
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


@pytest.mark.parametrize("fp64", [True, False])
@pytest.mark.parametrize("shape", [(8, 16, 128), (16, 8, 256), (128, 128, 16), (128, 128, 32), (128, 256, 32),
                                   (128, 128, 64)])
def test_x_passes_match_oracle_at_every_launch_shape(lib, shape, fp64):
    H = I.random_indicator(shape, 0.35, 21)
    dt = torch.float64 if fp64 else torch.float32
    pr = lib.FP64 if fp64 else lib.FP32
    tol = 1e-10 if fp64 else 1e-5
    g = [1.0, 0.25, -0.5]
    pen = dict(alpha0=250.0, beta0=180.0, b0=300.0)
    R = O.stokes(H, g, O.StokesParams(eps=0.0, adaptive=False, max_iter=3, **pen))
    Hd = torch.as_tensor(H, device=DEV)
    ctx = lib.acm_ctx(shape)
    u = torch.zeros((3,) + shape, dtype=dt, device=DEV)
    lam = torch.zeros_like(u)
    s, K, rep = lib.acm_stokes(ctx, Hd, g, lib.stokes_params(eps=0.0, adaptive=0, max_iter=3, precision=pr, **pen),
                               None, None, u, None, lam)
    assert relerr(u.cpu().numpy(), R.state.u) < tol
    assert relerr(lam.cpu().numpy(), R.state.lam) < tol
    np.testing.assert_allclose(rep.res[:6], R.residuals[-1], rtol=1e-8 if fp64 else 2.5e-4)
    uo = R.state.u / np.abs(R.state.u).max()
    Rc = O.advdiff(H, uo, 10.0, [0.5, 1.0, -0.25], O.AdvDiffParams(eps=0.0, max_iter=3))
    chi = torch.zeros(shape, dtype=dt, device=DEV)
    lib.acm_advdiff(ctx, Hd, torch.as_tensor(uo, dtype=dt, device=DEV), 10.0, [0.5, 1.0, -0.25],
                    lib.advdiff_params(eps=0.0, max_iter=3, precision=pr), chi, None)
    assert relerr(chi.cpu().numpy(), Rc.chi) < tol
    ctx.close()
