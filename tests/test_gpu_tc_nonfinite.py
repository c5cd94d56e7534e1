"""The tensor-core flow's LeakyReLU of infinities: slope 0 times -inf is NaN, as on the FP32 path."""
import types

import numpy as np
import pytest

from gpu_util import require_gpu

pytestmark = pytest.mark.gpu


# one and two configurations per block; conv1 in single sites, in pairs, with a pass for the images
@pytest.mark.parametrize("B", [4, 200])
@pytest.mark.parametrize("nd,L,width", [(2, 8, 8), (2, 16, 16), (2, 16, 32), (2, 32, 32), (3, 8, 16)])
def test_slope_zero_of_minus_infinity(nd, L, width, B):
    torch, P = require_gpu()
    shape = types.SimpleNamespace(nd=nd, L=L, n_layers=1, hidden=(width, width), c1=width, c2=width, ksize=3,
                                  use_final_tanh=True, leaky_slope=0.0)
    T = 3 ** nd
    # positive weights, no biases: a field of -3e38 overflows to -inf at every site and channel
    w = np.concatenate([np.full(width * T, 0.5), np.zeros(width), np.full(width * width * T, 0.5), np.zeros(width),
                        np.full(2 * width * T, 0.5), np.zeros(2)])
    flow = P.Flow(shape, w, precision="bf16")
    z = torch.full((B, L ** nd), -3e38, device="cuda")
    phi = flow.sample(B, z=z, phi4=(-4.0, 6.0)).phi
    n = torch.arange(L ** nd, device="cuda")
    updated = sum(n // L ** i % L for i in range(nd)) % 2 == 1
    assert torch.isnan(phi[:, updated]).all() and torch.equal(phi[:, ~updated], z[:, ~updated])
    assert P.device_status() == P._abi.GF_EDEVICE          # (reported once, then clear)
    assert P.device_status() == 0
