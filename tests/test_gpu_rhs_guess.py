"""The right-hand side that the Stokes x pass forms with a guessed penalty b.

The guess repeats the last change of Eq. 22; it is wrong whenever b starts, stops or
turns its change, or reaches psi_min. Runs that start far above and far below the
balance, with a clamp close by, pass through all of these; penalties and fields
follow the FP64 oracle (tolerances of the adaptive parity test) in both loops.
"""
import numpy as np
import pytest
import torch

from oracle import acm_oracle as O
from paper_2312_15554_gb300 import inputs as I

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.mark.parametrize("device_loop", [0, 1])
@pytest.mark.parametrize("b0,psi_min_frac", [(2.0, 1e-3), (2.0e4, 0.05), (2.0e3, 0.5), (300.0, 0.9)])
def test_guessed_right_hand_sides_follow_the_oracle(lib, b0, psi_min_frac, device_loop):
    H = I.sphere_pack((16, 16, 16), 0.5, 3.0, 5)[0]
    g = [0.0, 1.0, 0.5]
    kw = dict(eps=0.0, max_iter=45, alpha0=150.0, beta0=400.0, b0=b0, psi_min_frac=psi_min_frac)
    R = O.stokes(H, g, O.StokesParams(adaptive=True, **kw))
    b = R.penalties[:, 2]
    assert len(set(np.sign(np.diff(b)))) >= 2        # b changes in some iterations and not, or otherwise, in others
    ctx = lib.acm_ctx(H.shape)
    u = torch.zeros((3,) + H.shape, dtype=torch.float64, device=DEV)
    lam = torch.zeros_like(u)
    s, K, rep = lib.acm_stokes(ctx, torch.as_tensor(H, device=DEV), g, lib.stokes_params(
        adaptive=1, precision=lib.FP64, device_loop=device_loop, check_every=7, **kw), None, None, u, None, lam)
    hist = lib.acm_history(ctx, 0)
    ctx.close()
    assert rep.iters == 45
    np.testing.assert_allclose(hist[:, 12:15], R.penalties, rtol=1e-12)
    assert np.abs(u.cpu().numpy() - R.state.u).max() < 1e-9 * np.abs(R.state.u).max()
    assert np.abs(lam.cpu().numpy() - R.state.lam).max() < 1e-9 * np.abs(R.state.lam).max()
