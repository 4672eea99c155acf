"""Plane cells whose y forward, Green step and y inverse run as one pass, and the bare
transforms that read and write the caller's arrays.

Planes of 32 to 512 lines and narrow and wide rows against the FP64 oracle, left to
the grid and tuned (both y passes on row segments) and mixed (three passes); the
transform pair on device arrays, on arrays off the alignment of a complex element, on
host arrays, and with several fields. Tolerances as in the parity tests.
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
@pytest.mark.parametrize("tiles", ["grid", "segments", "mixed"])
@pytest.mark.parametrize("shape", [(1, 32, 8), (1, 64, 16), (1, 128, 128), (1, 256, 64), (1, 512, 32)])
def test_plane_pass_matches_oracle(lib, shape, tiles, fp64):
    H = I.disk_pack(shape[1], shape[2], 0.6, 2.5, 3)
    g = [0.3, 1.0, -0.5]
    dt = torch.float64 if fp64 else torch.float32
    kw = dict(eps=0.0, max_iter=8, alpha0=250.0, beta0=180.0, b0=300.0)
    R = O.stokes(H, g, O.StokesParams(adaptive=False, **kw))
    ctx = lib.acm_ctx(shape)
    if tiles != "grid":
        t = lib.acm_get_tiles(ctx, fp64)
        t["y_fwd_stokes"] = -8 if fp64 else -16
        if tiles == "segments":
            t["y_inv_stokes"] = t["y_fwd_stokes"]
        try:
            lib.acm_set_tiles(ctx, t, fp64)
        except lib.AcmError:
            assert shape[1] not in (64, 128, 256)
    u = torch.zeros((3,) + shape, dtype=dt, device=DEV)
    p = torch.zeros(shape, dtype=dt, device=DEV)
    s, K, rep = lib.acm_stokes(ctx, torch.as_tensor(H, device=DEV), g, lib.stokes_params(
        adaptive=0, precision=lib.FP64 if fp64 else lib.FP32, **kw), None, None, u, p, None)
    ctx.close()
    tol = 1e-10 if fp64 else 1e-5
    assert relerr(u.cpu().numpy(), R.state.u) < tol
    assert relerr(p.cpu().numpy(), R.p) < tol
    np.testing.assert_allclose(rep.res[:6], R.residuals[-1], rtol=1e-8 if fp64 else 2.5e-4)


@pytest.mark.parametrize("fp64", [True, False])
@pytest.mark.parametrize("where", ["device", "unaligned", "host"])
@pytest.mark.parametrize("shape", [(16, 32, 64), (1, 32, 512), (512, 8, 8), (32, 16, 256)])
def test_transform_pair_on_every_kind_of_array(lib, shape, where, fp64):
    dt = torch.float64 if fp64 else torch.float32
    nb = 2
    x = np.stack([I.random_field(shape, 40 + b) for b in range(nb)])
    ref = np.stack([O.fft3(f)[..., : shape[2] // 2 + 1] for f in x])
    off = 1 if where == "unaligned" else 0
    dev = "cpu" if where == "host" else DEV

    def buf(n):
        return torch.zeros(n + off, dtype=dt, device=dev)[off:]
    xin, spec, back = buf(x.size), buf(2 * ref.size), buf(x.size)
    xin.copy_(torch.as_tensor(x.ravel(), dtype=dt))
    ctx = lib.acm_ctx(shape)
    lib.acm_fft_r2c(ctx, xin, spec, fp64, nb)
    got = spec.cpu().numpy().reshape(ref.shape + (2,))
    tol = 1e-12 if fp64 else 2e-6
    assert relerr(got[..., 0] + 1j * got[..., 1], ref) < tol
    lib.acm_fft_c2r(ctx, spec, back, fp64, nb)
    assert relerr(back.cpu().numpy().reshape(x.shape), x) < tol
    ctx.close()
