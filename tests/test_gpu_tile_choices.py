"""The tile choices of the strided passes within their two sets.

The choices of one set (the row segments -W, or the positive widths) differ in the
columns a block takes only: fields agree bit for bit. FP32 lines of 128 and 256 points
have a segment of 4 columns, the width a pass of a small grid picks by itself, so that
the tuner can pick it there.
"""
import numpy as np
import pytest
import torch

from paper_2312_15554_gb300 import inputs as I

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def _fields(lib, ctx, H, uin, fp64):
    dt = torch.float64 if fp64 else torch.float32
    pr = lib.FP64 if fp64 else lib.FP32
    u = torch.zeros((3,) + H.shape, dtype=dt, device=DEV)
    p = torch.zeros(H.shape, dtype=dt, device=DEV)
    chi = torch.zeros(H.shape, dtype=dt, device=DEV)
    Hd = torch.as_tensor(H, device=DEV)
    lib.acm_stokes(ctx, Hd, [1.0, 0.3, -0.5], lib.stokes_params(eps=0.0, adaptive=0, max_iter=4, precision=pr), u=u, p=p)
    lib.acm_advdiff(ctx, Hd, uin, 10.0, [1.0, 0.0, 0.5], lib.advdiff_params(eps=0.0, max_iter=4, precision=pr), chi)
    return [x.cpu().numpy() for x in (u, p, chi)]


@pytest.mark.parametrize("fp64", [False, True])
@pytest.mark.parametrize("shape", [(64, 128, 32), (256, 64, 16), (128, 256, 16), (512, 8, 32), (8, 512, 32), (1, 128, 64)])
def test_choices_of_one_set_agree_bit_for_bit(lib, shape, fp64):
    H = (I.disk_pack(shape[1], shape[2], 0.5, 3.0, 3) if shape[0] == 1 else I.sphere_pack(shape, 0.5, 2.5, 3)[0])
    uin = torch.as_tensor(0.1 * I.random_field((3,) + shape, 9) * (1 - H)[None],
                          dtype=torch.float64 if fp64 else torch.float32, device=DEV)
    ctx = lib.acm_ctx(shape)
    base = lib.acm_get_tiles(ctx, fp64)
    for k in base:
        n = shape[1] if k.startswith("y") else shape[0]
        seen = {True: [], False: []}
        ref = {}
        for w in (-16, -8, -4, 2, 4, 8, 16, 32):
            try:
                lib.acm_set_tiles(ctx, {**base, k: w}, fp64)
            except lib.AcmError:
                continue
            seen[w < 0].append(w)
            if w < 0 and shape[0] == 1:
                # on a plane both y passes change their rounding together (one pass does their work)
                lib.acm_set_tiles(ctx, {**base, **{j: w for j in base if j.startswith("y")}}, fp64)
            got = _fields(lib, ctx, H, uin, fp64)
            for a, b in zip(ref.setdefault(w < 0, got), got):
                np.testing.assert_array_equal(a, b, err_msg=f"{k} {w}")
        segments = ([-8, -4] if fp64 else [-16, -8] + ([-4] if n > 64 else [])) if n in (64, 128, 256) else []
        assert seen[True] == segments, (k, n)
        assert base[k] in seen[False]
    ctx.close()


def test_tuned_small_grid_picks_among_its_candidates(lib):
    shape = (256, 32, 64)
    ctx = lib.acm_ctx(shape)
    t = lib.acm_autotune(ctx, False)
    assert t["z_stokes"] in (-16, -8, -4)
    lib.acm_set_tiles(ctx, t, False)
    assert lib.acm_get_tiles(ctx, False) == t
    ctx.close()
