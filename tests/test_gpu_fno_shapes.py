"""The network's pruned transforms and weight gradients at the edges of their range.

Every line length along axis 2 up to 512, kept modes up to the whole spectrum
(2 modes = n0 = n1, modes = n2 / 2), every width, batches that leave the channel
mix a ragged last block, against the FP64 oracle on the same BF16-rounded
parameters. The bounds are those of the other network tests: BF16 storage, 2e-2.
"""
import numpy as np
import pytest
import torch

from oracle import fno_oracle as F
from paper_2312_15554_gb300 import inputs as I

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.mark.parametrize("shape,width,modes,layers,B", [((8, 8, 8), 32, 4, 2, 3), ((16, 8, 128), 16, 4, 1, 2),
                                                       ((8, 8, 256), 4, 3, 1, 1), ((8, 16, 512), 8, 4, 1, 2),
                                                       ((64, 8, 16), 16, 4, 2, 1), ((16, 32, 16), 32, 8, 1, 5),
                                                       ((128, 8, 32), 8, 1, 2, 2)])
def test_network_matches_oracle_at_the_edges_of_its_shapes(lib, shape, width, modes, layers, B):
    rng = np.random.Generator(np.random.PCG64(5))
    theta = F.init_params(width, modes, layers, 5)
    theta = torch.as_tensor(theta + 0.05 * rng.standard_normal(theta.size), dtype=torch.float32)
    theta = theta.to(torch.bfloat16).to(torch.float64).numpy()
    Hs = np.stack([I.random_indicator(shape, 0.4, 30 + b) for b in range(B)])
    tgt = 0.5 * rng.standard_normal((B, 6) + shape)
    fno = lib.acm_fno(shape, width, modes, layers, max_batch=B)
    fno.set_params(theta.astype(np.float32))
    Hd = torch.as_tensor(Hs, device=DEV)
    out = torch.zeros((B, 6) + shape, dtype=torch.float32, device=DEV)
    fno.forward(Hd, out)
    grad = torch.zeros(fno.num_params, dtype=torch.float32, device=DEV)
    loss = fno.backward(Hd, torch.as_tensor(tgt, dtype=torch.float32, device=DEV), grad)
    out, g = out.cpu().numpy(), grad.cpu().numpy().astype(np.float64)
    L_ref, g_ref = 0.0, np.zeros_like(g)
    for b in range(B):
        o, cache = F.forward(theta, Hs[b], width, modes, layers)
        np.testing.assert_allclose(out[b], o, atol=2e-2 * np.abs(o).max())
        Lb, dout = F.loss_and_grad_out(o, tgt[b], Hs[b])
        L_ref += Lb / B
        g_ref += F.backward(theta, Hs[b], cache, dout / B, width, modes, layers)
    assert loss == pytest.approx(L_ref, rel=2e-2)
    assert g @ g_ref / (np.linalg.norm(g) * np.linalg.norm(g_ref)) > 0.999
    assert np.linalg.norm(g - g_ref) / np.linalg.norm(g_ref) < 2e-2
    fno.close()
