"""The reverse pass's kernels over widths, lattices and unit sizes, against the
oracle gradient, and the recompute path's fallback."""
import numpy as np
import pytest

import gf_inputs as gi
import oracle
from gpu_util import require_gpu

pytestmark = pytest.mark.gpu

# every width in 2D and 3D, the smallest lattices, odd unit counts, one lattice
# whose units take a single staging buffer and whose weights stay in global memory
SHAPES = [(2, 2, 8, 3), (2, 4, 32, 2), (2, 6, 16, 5), (2, 10, 24, 3), (2, 16, 8, 2), (2, 20, 32, 2), (2, 64, 16, 1),
          (3, 2, 16, 4), (3, 4, 8, 3), (3, 4, 24, 2), (3, 6, 32, 2), (3, 10, 16, 1), (3, 16, 32, 1)]


@pytest.mark.parametrize("nd,L,width,B", SHAPES)
def test_gradient_matches_the_oracle(nd, L, width, B):
    torch, P = require_gpu()
    shape = gi.FlowShape(nd, L, 3, width, width)
    w = gi.init_weights(shape, seed=L)
    w32 = w.astype(np.float32).astype(np.float64)
    m2, lam = -4.0, 8.0
    z = oracle.prior(shape.V, B, seed=5, counter0=3, f32=True)
    ref_loss, ref = oracle.flow_loss_grad(shape, w32, m2, lam, z)
    flow = P.Flow(shape, w)
    loss, grad = flow.train_step(B, (m2, lam), seed=5, counter0=3)
    g = grad.double().cpu().numpy()
    assert abs(loss.item() - ref_loss) <= 1e-4 * max(abs(ref_loss), 1)
    # the FP32 gradient's stated tolerance: relative L2 1e-3
    assert np.linalg.norm(g - ref) <= 1e-3 * np.linalg.norm(ref)
    # same result again, and from a batch that is one of several units per CTA
    loss2, grad2 = flow.train_step(B, (m2, lam), seed=5, counter0=3)
    assert torch.equal(grad, grad2) and torch.equal(loss, loss2)
    if L ** nd <= 400:
        lb, gb = flow.train_step(700, (m2, lam), seed=5, counter0=3)
        parts = [flow.train_step(n, (m2, lam), seed=5, counter0=3 + at) for at, n in ((0, 300), (300, 400))]
        mean = (parts[0][1].double() * 300 + parts[1][1].double() * 400) / 700
        # FP32 sums over 700 configurations in another grouping
        assert (gb.double() - mean).norm() <= 1e-5 * mean.norm()
    assert P.device_status() == 0
