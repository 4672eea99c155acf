"""Planes of 32 lines with rows of 8 to 32 voxels, in the calls that transform real
fields by blocks of up to 64 lines: warm starts, the gradient form of K, and
transforms of arrays off the alignment of a pair. Tolerances as in the parity tests.
"""
import numpy as np
import pytest
import torch

from oracle import acm_oracle as O
from paper_2312_15554_gb300 import inputs as I

pytestmark = pytest.mark.gpu

DEV = "cuda:0"
SHAPES = [(1, 32, 8), (1, 32, 16), (1, 32, 32), (1, 32, 64), (1, 64, 8)]


def relerr(a, b):
    return float(np.abs(np.asarray(a) - b).max() / np.abs(b).max())


@pytest.mark.parametrize("fp64", [True, False])
@pytest.mark.parametrize("shape", SHAPES)
def test_warm_start_matches_oracle(lib, shape, fp64):
    H = I.disk_pack(shape[1], shape[2], 0.6, 2.0, 3)
    u0 = 0.01 * I.random_field((3,) + shape, 3)
    l0 = I.random_field((3,) + shape, 4) * H[None]
    g = [0.3, 1.0, -0.5]
    pen = dict(eps=0.0, max_iter=5, alpha0=250.0, beta0=180.0, b0=300.0)
    R = O.stokes(H, g, O.StokesParams(adaptive=False, **pen), init=O.warm_state(H, u0, l0))
    dt = torch.float64 if fp64 else torch.float32
    ctx = lib.acm_ctx(shape)
    u = torch.zeros((3,) + shape, dtype=dt, device=DEV)
    lam = torch.zeros_like(u)
    p = torch.zeros(shape, dtype=dt, device=DEV)
    lib.acm_stokes(ctx, torch.as_tensor(H, device=DEV), g,
                   lib.stokes_params(adaptive=0, precision=lib.FP64 if fp64 else lib.FP32, **pen),
                   torch.as_tensor(u0, dtype=dt, device=DEV), torch.as_tensor(l0, dtype=dt, device=DEV), u, p, lam)
    ctx.close()
    tol = 1e-10 if fp64 else 1e-5
    assert relerr(u.cpu().numpy(), R.state.u) < tol
    assert relerr(lam.cpu().numpy(), R.state.lam) < tol
    assert relerr(p.cpu().numpy(), R.p) < tol


@pytest.mark.parametrize("shape", SHAPES)
def test_gradient_form_matches_oracle(lib, shape):
    H = I.disk_pack(shape[1], shape[2], 0.6, 2.0, 3)
    pen = dict(eps=0.0, max_iter=20, alpha0=250.0, beta0=180.0, b0=300.0)
    Km, Kg, _ = O.permeability_tensor(H, O.StokesParams(adaptive=False, **pen))
    ctx = lib.acm_ctx(shape)
    u3 = torch.zeros((3, 3) + shape, dtype=torch.float64, device=DEV)
    _, K, Kgrad, _ = lib.acm_stokes_tensor(ctx, torch.as_tensor(H, device=DEV),
                                           lib.stokes_params(adaptive=0, precision=lib.FP64, **pen), u3, grad_form=True)
    ctx.close()
    assert relerr(K, Km) < 1e-9
    assert relerr(Kgrad, Kg) < 1e-9


@pytest.mark.parametrize("fp64", [True, False])
@pytest.mark.parametrize("shape", SHAPES)
def test_unaligned_transform_pair_matches_oracle(lib, shape, fp64):
    dt = torch.float64 if fp64 else torch.float32
    x = I.random_field(shape, 40)
    ref = O.fft3(x)[..., : shape[2] // 2 + 1]

    def buf(n):
        # one element in front and one behind, to see stores outside the array
        b = torch.full((n + 2,), 7.0, dtype=dt, device=DEV)
        return b, b[1:n + 1]
    (_, xin), (bs, spec), (bb, back) = buf(x.size), buf(2 * ref.size), buf(x.size)
    xin.copy_(torch.as_tensor(x.ravel(), dtype=dt))
    ctx = lib.acm_ctx(shape)
    lib.acm_fft_r2c(ctx, xin, spec, fp64, 1)
    lib.acm_fft_c2r(ctx, spec, back, fp64, 1)
    ctx.close()
    got = spec.cpu().numpy().reshape(ref.shape + (2,))
    tol = 1e-12 if fp64 else 2e-6
    assert relerr(got[..., 0] + 1j * got[..., 1], ref) < tol
    assert relerr(back.cpu().numpy().reshape(shape), x) < tol
    for b in (bs, bb):
        assert float(b[0]) == float(b[-1]) == 7.0
