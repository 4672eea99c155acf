"""The strided passes at every line length and tile shape against the FP64 oracle.

Lines of 8 to 512 points along both strided axes (one, two and three exchange
stages), pencil counts below, at and above a tile's width, column counts that
fill tiles and leave the Nyquist column a tile of its own or share one with
others. Tolerances as in the parity tests: FP64 1e-12 for a transform and 1e-10
for fields, FP32 2e-6 and 1e-5, of the largest magnitude.
"""
import numpy as np
import pytest
import torch

from oracle import acm_oracle as O
from paper_2312_15554_gb300 import inputs as I

pytestmark = pytest.mark.gpu

DEV = "cuda:0"

SHAPES = [(512, 8, 8), (8, 512, 8), (512, 8, 64), (32, 8, 16), (8, 32, 64), (16, 16, 16), (128, 16, 64), (64, 8, 256),
          (8, 256, 32), (256, 8, 16)]


def relerr(a, b):
    return float(np.abs(np.asarray(a) - b).max() / np.abs(b).max())


@pytest.mark.parametrize("fp64", [True, False])
@pytest.mark.parametrize("shape", SHAPES)
def test_strided_passes_match_oracle(lib, shape, fp64):
    dt = torch.float64 if fp64 else torch.float32
    pr = lib.FP64 if fp64 else lib.FP32
    ctx = lib.acm_ctx(shape)
    x = I.random_field(shape, 11)
    ref = O.fft3(x)[..., : shape[2] // 2 + 1]
    xin = torch.as_tensor(x, dtype=dt, device=DEV)
    out = torch.zeros(shape[:2] + (shape[2] // 2 + 1, 2), dtype=dt, device=DEV)
    lib.acm_fft_r2c(ctx, xin, out, fp64)
    got = out.cpu().numpy()
    assert relerr(got[..., 0] + 1j * got[..., 1], ref) < (1e-12 if fp64 else 2e-6)
    back = torch.zeros(shape, dtype=dt, device=DEV)
    lib.acm_fft_c2r(ctx, out, back, fp64)
    assert relerr(back.cpu().numpy(), x) < (1e-12 if fp64 else 2e-6)

    H = I.random_indicator(shape, 0.35, 22)
    Hd = torch.as_tensor(H, device=DEV)
    g = [1.0, 0.25, -0.5]
    tol = 1e-10 if fp64 else 1e-5
    pen = dict(alpha0=250.0, beta0=180.0, b0=300.0)
    R = O.stokes(H, g, O.StokesParams(eps=0.0, adaptive=False, max_iter=3, **pen))
    u = torch.zeros((3,) + shape, dtype=dt, device=DEV)
    p = torch.zeros(shape, dtype=dt, device=DEV)
    s, K, rep = lib.acm_stokes(ctx, Hd, g, lib.stokes_params(eps=0.0, adaptive=0, max_iter=3, precision=pr, **pen),
                               None, None, u, p, None)
    assert relerr(u.cpu().numpy(), R.state.u) < tol
    assert relerr(p.cpu().numpy(), R.p) < tol
    np.testing.assert_allclose(rep.res[:6], R.residuals[-1], rtol=1e-8 if fp64 else 2.5e-4)
    uo = R.state.u / np.abs(R.state.u).max()
    Rc = O.advdiff(H, uo, 10.0, [0.5, 1.0, -0.25], O.AdvDiffParams(eps=0.0, max_iter=3))
    chi = torch.zeros(shape, dtype=dt, device=DEV)
    grad = torch.zeros((3,) + shape, dtype=dt, device=DEV)
    lib.acm_advdiff(ctx, Hd, torch.as_tensor(uo, dtype=dt, device=DEV), 10.0, [0.5, 1.0, -0.25],
                    lib.advdiff_params(eps=0.0, max_iter=3, precision=pr), chi, grad)
    assert relerr(chi.cpu().numpy(), Rc.chi) < tol
    assert relerr(grad.cpu().numpy(), Rc.grad_chi) < tol
    ctx.close()
