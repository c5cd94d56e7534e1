"""GPU tests of the general network's kernel (gf_flow_variant.cu): sites per
thread, channel groups of 4 and 8, weight stages of several chunks or none, and
CTA sizes, at the sizes where they change."""
import pytest

import gf_inputs as gi
from gpu_util import assert_logw_close, assert_sites_close, require_gpu

pytestmark = pytest.mark.gpu

SHAPES = [
    (2, 2, 3, (9, 3), 7),            # taps that wrap more than once
    (2, 6, 2, (12, 20), 3),          # L not a multiple of 4; groups of 8 and of 4
    (2, 4, 2, (65, 64), 3),          # rows longer than a pass; several chunks per tap row
    (2, 16, 2, (16, 16, 8), 5),      # several chunks, two passes of the head's sites
    (2, 48, 2, (3,), 3),             # four sites per thread, sums over more sites than threads
    (2, 16, 2, (111,), 3),           # no room for a stage: weights through L1
    (2, 12, 2, (), 5),               # no hidden layer
    (3, 6, 2, (131,), 3),            # 3D, no room for a stage
    (3, 6, 2, (12, 20), 3),
    (3, 12, 1, (4, 8), 3),
    (3, 4, 2, (7, 1), 5),
]


@pytest.mark.parametrize("nd,L,layers,hidden,ksize", SHAPES)
def test_oracle_and_batch_independence(orc, nd, L, layers, hidden, ksize):
    """Against the FP64 oracle at the plain path's tolerances; then every
    configuration of larger batches (other CTA sizes and splits) to the bit."""
    torch, P = require_gpu()
    shape = gi.FlowShape(nd, L, layers, hidden_sizes=hidden, ksize=ksize)
    w = gi.init_weights(shape, seed=13)
    flow = P.Flow(shape, w)
    m2, lam = -4.0, 8.0
    out = flow.sample(5, seed=9, phi4=(m2, lam), return_z=True)
    ref = orc.flow_sample(shape, w, m2, lam, 5, seed=9)
    assert_sites_close(out.phi.cpu().numpy(), ref["phi"])
    for k in ("logq", "S", "logw"):
        assert_logw_close(getattr(out, k).cpu().numpy(), ref[k], what=k)
    zi, lqi = flow.logq(out.phi, return_z=True)
    assert_sites_close(zi.cpu().numpy(), out.z.cpu().numpy(), rtol=1e-4, what="z(inverse)")
    for B in (200, 450, 1400):
        big = flow.sample(B, seed=9, phi4=(m2, lam), return_z=True)
        for k in ("phi", "z", "logq", "S", "logw"):
            assert torch.equal(getattr(big, k)[:5], getattr(out, k)), (B, k)
        zb, lqb = flow.logq(big.phi, return_z=True)
        assert torch.equal(zb[:5], zi) and torch.equal(lqb[:5], lqi), B
    assert P.device_status() == 0
