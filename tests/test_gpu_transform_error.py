"""How far the bare transforms are from the exact ones.

Relative L2 error of r2c and c2r of seeded normal fields against transforms in
extended precision. The bounds are the errors of the block-phase real transforms
with tabulated twiddles (every twiddle of a line one rounded root, no product of
roots), measured on these inputs, plus half a per cent for their printed digits:
passes that regroup the arithmetic may not lose accuracy to it.
"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

DEV = "cuda:0"

# shape: (r2c, c2r)
FP32 = {
    (16, 16, 32): (1.204e-07, 1.219e-07), (16, 16, 64): (1.282e-07, 1.375e-07),
    (16, 16, 128): (1.320e-07, 1.420e-07), (16, 16, 256): (1.362e-07, 1.452e-07),
    (16, 16, 512): (1.424e-07, 1.471e-07), (64, 64, 64): (1.522e-07, 1.617e-07),
    (64, 64, 128): (1.550e-07, 1.657e-07), (32, 64, 256): (1.563e-07, 1.655e-07),
}
FP64 = {
    (16, 16, 8): (1.896e-16, 1.950e-16), (16, 16, 16): (2.100e-16, 2.123e-16),
    (16, 16, 32): (2.362e-16, 2.165e-16), (16, 16, 64): (2.669e-16, 2.336e-16),
    (16, 16, 128): (2.709e-16, 2.462e-16), (16, 16, 256): (2.827e-16, 2.637e-16),
    (16, 16, 512): (2.949e-16, 2.898e-16), (64, 64, 64): (3.419e-16, 3.130e-16),
    (64, 64, 128): (3.416e-16, 3.219e-16), (32, 64, 256): (3.420e-16, 3.221e-16),
}


def _err(a, b):
    d = np.abs(a.astype(b.dtype) - b)
    return float(np.sqrt((d ** 2).sum() / (np.abs(b) ** 2).sum()))


def transform_errors(lib, shape, fp64):
    """(r2c, c2r), the mean over four seeds (two on the larger fields)."""
    dt = torch.float64 if fp64 else torch.float32
    out = []
    ctx = lib.acm_ctx(shape)
    for seed in range(2 if max(shape[:2]) > 16 else 4):
        x = np.random.default_rng(seed).standard_normal(shape).astype(np.float64 if fp64 else np.float32)
        ref = np.fft.rfftn(x.astype(np.longdouble))
        spec = torch.zeros(ref.shape + (2,), dtype=dt, device=DEV)
        back = torch.zeros(shape, dtype=dt, device=DEV)
        lib.acm_fft_r2c(ctx, torch.as_tensor(x, device=DEV), spec, fp64)
        s = spec.cpu().numpy()
        rs = np.stack([ref.real, ref.imag], -1).astype(x.dtype)   # the input of c2r: the rounded exact spectrum
        refb = np.fft.irfftn(rs[..., 0].astype(np.longdouble) + 1j * rs[..., 1].astype(np.longdouble), s=shape,
                             axes=(0, 1, 2))
        lib.acm_fft_c2r(ctx, torch.as_tensor(rs, device=DEV), back, fp64)
        out.append((_err(s[..., 0] + 1j * s[..., 1], ref), _err(back.cpu().numpy(), refb)))
    ctx.close()
    return np.mean(out, axis=0)


@pytest.mark.parametrize("shape", list(FP32))
def test_fp32_transforms_are_as_accurate_as_tabulated_twiddles(lib, shape):
    r2c, c2r = transform_errors(lib, shape, False)
    assert r2c <= 1.005 * FP32[shape][0]
    assert c2r <= 1.005 * FP32[shape][1]


@pytest.mark.parametrize("shape", list(FP64))
def test_fp64_transforms_lose_no_accuracy(lib, shape):
    """Another order of the arithmetic rounds independently: the relative spread of an RMS
    over n values is 1/sqrt(2 n), that of two of them 1/sqrt(n), and three of those are
    allowed beside the printed digits."""
    n = (2 if max(shape[:2]) > 16 else 4) * np.prod(shape)
    tol = 1.0 + 3.0 / np.sqrt(n) + 0.0005
    r2c, c2r = transform_errors(lib, shape, True)
    assert r2c <= tol * FP64[shape][0]
    assert c2r <= tol * FP64[shape][1]
