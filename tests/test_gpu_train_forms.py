"""Training's two forms of the forward pass and the recompute: layer by layer (small batches
of lattices that do not fit a CTA whole) and fused with a slice ring."""
import numpy as np
import pytest

import gf_inputs as gi
import oracle
from gpu_util import LOGW_RTOL, require_gpu

pytestmark = pytest.mark.gpu

# lattices that go through a slice ring: G < L, slices recomputed at the wrap, several
# weight stages a layer; a batch of 40 is below half of the SMs (layer by layer), 80 and
# 200 above (fused; 200: a second configuration on some SMs)
SHAPES = [(2, 64, 16, 3), (2, 48, 32, 2), (3, 12, 24, 2), (3, 14, 32, 1), (3, 16, 8, 3)]
PHI4 = (-4.0, 8.0)


@pytest.mark.parametrize("nd,L,width,layers", SHAPES)
def test_forms_agree(nd, L, width, layers):
    torch, P = require_gpu()
    shape = gi.FlowShape(nd, L, layers, width, width)
    flow = P.Flow(shape, gi.init_weights(shape, seed=L))
    # every sum has one order in both forms: equal to the bit
    small = [flow.forward_train(40, seed=5, counter0=3 + 40 * i)[:2] for i in range(2)]
    for B in (80, 200):
        phi, logq, _ = flow.forward_train(B, seed=5, counter0=3)
        for i, (p, q) in enumerate(small):
            assert torch.equal(phi[40 * i:40 * i + 40], p) and torch.equal(logq[40 * i:40 * i + 40], q)
    # the weight gradients are FP32 sums over the batch in another grouping
    parts = [flow.train_step(40, PHI4, seed=5, counter0=3 + 40 * i) for i in range(2)]
    loss, grad = flow.train_step(80, PHI4, seed=5, counter0=3)
    mean = (parts[0][1].double() + parts[1][1].double()) / 2
    assert (grad.double() - mean).norm() <= 1e-5 * mean.norm()
    # FP64 means of the same 80 numbers
    want = (parts[0][0] + parts[1][0]).item() / 2
    assert abs(loss.item() - want) <= 1e-13 * max(abs(want), 1)
    # and the sampler's log w = -(S + log q) of the same configurations
    ref = -flow.sample(80, seed=5, counter0=3, phi4=PHI4).logw.mean().item()
    assert abs(loss.item() - ref) <= LOGW_RTOL * max(abs(ref), 1)
    assert P.device_status() == 0


@pytest.mark.parametrize("nd,L,width", [(3, 16, 8), (2, 48, 16)])
def test_fused_ring_gradient_matches_the_oracle(nd, L, width):
    _, P = require_gpu()
    shape, B = gi.FlowShape(nd, L, 2, width, width), 80
    w = gi.init_weights(shape, seed=L)
    z = oracle.prior(shape.V, B, seed=5, counter0=3, f32=True)
    ref_loss, ref = oracle.flow_loss_grad(shape, w.astype(np.float32).astype(np.float64), *PHI4, z)
    loss, grad = P.Flow(shape, w).train_step(B, PHI4, seed=5, counter0=3)
    assert abs(loss.item() - ref_loss) <= LOGW_RTOL * max(abs(ref_loss), 1)
    # the FP32 gradient's stated tolerance: relative L2 1e-3
    assert np.linalg.norm(grad.double().cpu().numpy() - ref) <= 1e-3 * np.linalg.norm(ref)
