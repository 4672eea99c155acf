"""Batches of many distinct cell shapes.

The device-resident loop watches the stop flags of a bounded number of shapes;
batches of more run host-launched. One batch on each side of that bound, and
one past the four shapes the loop once had room for: every cell as in a solve
of its own (the launches are the same ones, so to the FP32 rounding of K).
"""
import itertools

import numpy as np
import pytest
import torch

from paper_2312_15554_gb300 import inputs as I

pytestmark = pytest.mark.gpu

DEV = "cuda:0"

SHAPES = [s for s in itertools.product((8, 16, 32), repeat=3)]


@pytest.mark.parametrize("nshapes", [5, 16, 17, 27])
def test_batch_of_many_shapes_matches_single_cells(lib, nshapes):
    shapes = SHAPES[:nshapes] + SHAPES[:2]
    Hs = [torch.as_tensor(I.random_indicator(sh, 0.4, 60 + i), device=DEV) for i, sh in enumerate(shapes)]
    prm = lib.stokes_params(eps=0.0, adaptive=1, max_iter=9)
    batch = lib.acm_batch(shapes)
    u = [torch.zeros((3, 3) + sh, device=DEV) for sh in shapes]
    _, K, reps = lib.acm_batch_stokes(batch, Hs, prm, u)
    batch.close()
    for i, sh in enumerate(shapes):
        ctx = lib.acm_ctx(sh)
        u1 = torch.zeros((3, 3) + sh, device=DEV)
        _, K1, _, r1 = lib.acm_stokes_tensor(ctx, Hs[i], prm, u1)
        ctx.close()
        assert [r.iters for r in reps[i]] == [r.iters for r in r1] == [9, 9, 9]
        np.testing.assert_allclose(K[i], K1, rtol=1e-6, atol=1e-6 * np.abs(K1).max())
        assert float((u[i] - u1).abs().max()) <= 1e-6 * float(u1.abs().max())


def test_refused_history_leaves_the_batch_usable(lib):
    """A history that does not fit device memory is refused, and the next solve does not
    write the records of the one before it (the device loop is captured anew)."""
    shapes = [(16, 16, 16), (8, 16, 32)]
    Hs = [torch.as_tensor(I.random_indicator(sh, 0.4, 90 + i), device=DEV) for i, sh in enumerate(shapes)]
    prm = lib.stokes_params(eps=0.0, adaptive=1, max_iter=8)
    batch = lib.acm_batch(shapes)
    lib.acm_batch_history_enable(batch, 8)
    _, K0, _ = lib.acm_batch_stokes(batch, Hs, prm)
    h0 = lib.acm_batch_history(batch, 1, 2)
    with pytest.raises(lib.AcmError):
        lib.acm_batch_history_enable(batch, 2**31 - 1)   # about a terabyte
    _, K1, _ = lib.acm_batch_stokes(batch, Hs, prm)
    np.testing.assert_array_equal(K0, K1)
    assert lib.acm_batch_history(batch, 1, 2).shape[0] == 0
    lib.acm_batch_history_enable(batch, 8)
    lib.acm_batch_stokes(batch, Hs, prm)
    np.testing.assert_array_equal(lib.acm_batch_history(batch, 1, 2), h0)
    batch.close()
