"""The guessed right-hand side of the Stokes x pass in FP32, in batches and across the
change of precision, and device loops whose cap their iterations a turn do not divide.

Penalties are products of the same factors on both sides, so a run follows the oracle's
to rounding as long as no comparison of Eq. 22 is closer than FP32 resolves (2.5e-4 of a
residual, the tolerance of the parity tests); each case asserts that margin first.
"""
import numpy as np
import pytest
import torch

from oracle import acm_oracle as O
from paper_2312_15554_gb300 import inputs as I

pytestmark = pytest.mark.gpu

DEV = "cuda:0"
SHAPE = (8, 16, 32)
G = [0.0, 1.0, 0.5]
START = dict(alpha0=150.0, beta0=400.0)


def oracle(H, g, n, b0, psi_min_frac):
    R = O.stokes(H, g, O.StokesParams(adaptive=True, eps=0.0, max_iter=n, b0=b0, psi_min_frac=psi_min_frac, **START))
    r = np.array(R.residuals)
    with np.errstate(all="ignore"):
        ratio = r[:, 0::2] / r[:, 1::2]
        tau = np.array(O.StokesParams().tau)
        margin = np.nanmin(np.minimum(np.abs(ratio / tau - 1), np.abs(1 / (ratio * tau) - 1)))
    assert margin > 1e-3
    assert np.any(np.diff(R.penalties[:, 2]) != 0)
    return R


def relerr(a, b):
    return float(np.abs(np.asarray(a) - b).max() / np.abs(b).max())


CASES = [(2.0, 1e-3), (2.0e4, 0.05), (2.0e3, 0.5), (300.0, 0.9)]


@pytest.mark.parametrize("device_loop", [0, 1])
@pytest.mark.parametrize("b0,psi_min_frac", CASES)
def test_fp32_follows_the_oracle(lib, b0, psi_min_frac, device_loop):
    H = I.sphere_pack(SHAPE, 0.5, 3.0, 5)[0]
    R = oracle(H, G, 30, b0, psi_min_frac)
    ctx = lib.acm_ctx(SHAPE)
    u = torch.zeros((3,) + SHAPE, device=DEV)
    lam = torch.zeros_like(u)
    lib.acm_stokes(ctx, torch.as_tensor(H, device=DEV), G, lib.stokes_params(
        eps=0.0, max_iter=30, adaptive=1, b0=b0, psi_min_frac=psi_min_frac, device_loop=device_loop, check_every=4,
        **START), None, None, u, None, lam)
    hist = lib.acm_history(ctx, 0)
    ctx.close()
    np.testing.assert_allclose(hist[:, 12:15], R.penalties, rtol=1e-12)
    assert relerr(u.cpu().numpy(), R.state.u) < 1e-5
    assert relerr(lam.cpu().numpy(), R.state.lam) < 1e-5


# the FP32 phase of these ends after 10, 5 and 4 iterations, while b changes
@pytest.mark.parametrize("device_loop", [0, 1])
@pytest.mark.parametrize("b0,psi_min_frac,eps32", [(2.0e4, 0.05, 0.498), (2.0, 1e-3, 0.1), (2.0e3, 0.5, 0.4)])
def test_guess_does_not_outlive_the_precision(lib, b0, psi_min_frac, eps32, device_loop):
    H = I.sphere_pack(SHAPE, 0.5, 3.0, 5)[0]
    R = oracle(H, G, 30, b0, psi_min_frac)
    ctx = lib.acm_ctx(SHAPE)
    u = torch.zeros((3,) + SHAPE, dtype=torch.float64, device=DEV)
    lam = torch.zeros_like(u)
    _, _, rep = lib.acm_stokes(ctx, torch.as_tensor(H, device=DEV), G, lib.stokes_params(
        eps=0.0, eps32=eps32, max_iter=30, adaptive=1, b0=b0, psi_min_frac=psi_min_frac, device_loop=device_loop,
        check_every=4, precision=lib.FP32_THEN_FP64, **START), None, None, u, None, lam)
    hist = lib.acm_history(ctx, 0)
    ctx.close()
    assert rep.iters == 30 and 20 <= rep.iters_fp64 <= 26
    np.testing.assert_allclose(hist[:, 12:15], R.penalties, rtol=1e-12)
    assert relerr(u.cpu().numpy(), R.state.u) < 1e-5
    assert relerr(lam.cpu().numpy(), R.state.lam) < 1e-5


@pytest.mark.parametrize("b0,psi_min_frac", CASES[:2])
def test_every_problem_of_a_batch_keeps_its_own_guess(lib, b0, psi_min_frac):
    Hs = [I.sphere_pack(SHAPE, 0.5, 3.0, 5)[0], I.sphere_pack((16, 16, 16), 0.35, 2.5, 8)[0],
          I.sphere_pack(SHAPE, 0.7, 2.0, 9)[0]]
    n = 24
    batch = lib.acm_batch([H.shape for H in Hs])
    lib.acm_batch_history_enable(batch, n)
    u = [torch.zeros((3, 3) + H.shape, device=DEV) for H in Hs]
    lib.acm_batch_stokes(batch, [torch.as_tensor(H, device=DEV) for H in Hs], lib.stokes_params(
        eps=0.0, max_iter=n, adaptive=1, b0=b0, psi_min_frac=psi_min_frac, **START), u)
    for i, H in enumerate(Hs):
        for j in range(3):
            R = oracle(H, [1.0 if c == j else 0.0 for c in range(3)], n, b0, psi_min_frac)
            hist = lib.acm_batch_history(batch, i, j)
            np.testing.assert_allclose(hist[:, 12:15], R.penalties, rtol=1e-12)
            assert relerr(u[i][j].cpu().numpy(), R.state.u) < 1e-5
    batch.close()


@pytest.mark.parametrize("cap", [1, 3, 5, 7, 13, 16, 17, 25, 30])
def test_unrolled_loops_stop_at_their_cap(lib, cap):
    """Up to four iterations run per turn of the device loop; the host loop launches one
    by one. Same iterations, same fields."""
    H = torch.as_tensor(I.sphere_pack(SHAPE, 0.5, 3.0, 5)[0], device=DEV)
    uin = torch.as_tensor(0.1 * I.random_field((3,) + SHAPE, 9), dtype=torch.float32, device=DEV)
    out = {}
    for loop in (0, 1):
        ctx = lib.acm_ctx(SHAPE)
        u = torch.zeros((3,) + SHAPE, device=DEV)
        p = torch.zeros(SHAPE, device=DEV)
        chi = torch.zeros(SHAPE, device=DEV)
        _, _, r = lib.acm_stokes(ctx, H, G, lib.stokes_params(eps=0.0, max_iter=cap, adaptive=1, device_loop=loop,
                                                              check_every=3), None, None, u, p, None)
        h = lib.acm_history(ctx, 0)
        _, _, _, rs = lib.acm_advdiff(ctx, H, uin, 5.0, [1.0, 0.0, 0.0], lib.advdiff_params(
            eps=0.0, max_iter=cap, device_loop=loop, check_every=3), chi)
        assert r.iters == rs.iters == cap and h.shape[0] == cap
        out[loop] = [u.cpu().numpy(), p.cpu().numpy(), chi.cpu().numpy(), h]
        ctx.close()
    for a, b in zip(out[0], out[1]):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("fp64", [False, True])
@pytest.mark.parametrize("n1", [32, 64, 128, 256, 512])
def test_plane_cells_run_one_strided_pass(lib, n1, fp64):
    """Left to the grid, or with both y passes on row segments, a plane's y forward, Green
    step and y inverse are one launch; with mixed choices they are three."""
    shape = (1, n1, 16)
    H = torch.as_tensor(I.disk_pack(n1, 16, 0.6, 2.5, 3), device=DEV)
    u = torch.zeros((3,) + shape, dtype=torch.float64 if fp64 else torch.float32, device=DEV)
    ctx = lib.acm_ctx(shape)
    base = lib.acm_get_tiles(ctx, fp64)
    seg = -8 if fp64 else -16
    choices = [(base, 0)]
    if n1 in (64, 128, 256):
        choices += [({**base, "y_fwd_stokes": seg, "y_inv_stokes": seg}, 0), ({**base, "y_fwd_stokes": seg}, 6)]
    for tiles, want in choices:
        lib.acm_set_tiles(ctx, tiles, fp64)
        lib.acm_profile_read(ctx)
        lib.acm_stokes(ctx, H, G, lib.stokes_params(eps=0.0, max_iter=6, adaptive=0, device_loop=0,
                                                    precision=lib.FP64 if fp64 else lib.FP32), u=u)
        n = {k: v[1] for k, v in lib.acm_profile_read(ctx).items()}
        assert (n["y_fwd_stokes"], n["z_stokes"], n["y_inv_stokes"]) == (want, 6, want)
    ctx.close()
