"""GPU tests of the tensor-core kernel's forms (gf_flow_tc.cu): one or two
configurations per CTA, two or four epilogue groups, conv1's site and channel
splits, the halo pass of h1, and both forms of the LeakyReLU."""
import numpy as np
import pytest

import gf_inputs as gi
from gpu_util import TC_MODE, assert_logw_close, assert_sites_close, require_gpu

pytestmark = pytest.mark.gpu


# two configurations per CTA against one: the smallest lattices, the padded
# width, conv1 with and without the halo pass (2D from L = 32 on); then the
# shapes that never fit two (four groups; two at width 32)
@pytest.mark.parametrize("nd,L,c", [(2, 8, 8), (2, 8, 32), (2, 16, 24), (2, 48, 16), (2, 32, 16), (2, 32, 32), (3, 4, 16),
                                    (3, 8, 16), (2, 64, 16), (3, 12, 16), (3, 16, 8), (3, 8, 32)])
def test_configurations_do_not_depend_on_the_batch(nd, L, c):
    """Each configuration of a batch that fills every CTA several times is the
    one a launch of its own gives: the field to the bit, the lattice sums (FP64
    accurate, grouped by the CTA's threads) to 1e-11 of their terms' size."""
    torch, P = require_gpu()
    shape = gi.FlowShape(nd, L, 2, c, c)
    if not P.tensor_core_supported(shape):
        pytest.skip("not a shape of the tensor-core kernel")
    flow = P.Flow(shape, gi.init_weights(shape, seed=3), precision="bf16")
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    B = 4 * sms + 3
    big = flow.sample(B, seed=8, counter0=0, phi4=(-4.0, 6.0))
    for k in (0, sms - 1, 2 * sms, B - 2):
        one = flow.sample(2, seed=8, counter0=k, phi4=(-4.0, 6.0))
        assert torch.equal(one.phi, big.phi[k:k + 2])
        for name in ("logq", "S", "logw"):
            a, b = getattr(one, name), getattr(big, name)[k:k + 2]
            assert ((a - b).abs() <= 1e-11 * shape.V).all(), name
    assert P.device_status() == 0


# LeakyReLU slopes above one take the other form of the packed selection; zero
# and negative slopes the first
@pytest.mark.parametrize("slope", [-0.5, 0.0, 1.0, 1.5])
@pytest.mark.parametrize("nd,L,c", [(2, 32, 16), (3, 12, 16), (3, 8, 32)])
def test_slopes_match_the_emulated_oracle(orc, nd, L, c, slope):
    """Bounds: twice the drift that FP32-level differences before the roundings
    give on other inputs of the same flow, from the oracle alone."""
    torch, P = require_gpu()
    shape = gi.FlowShape(nd, L, 2, c, c, leaky_slope=slope)
    w = gi.init_weights(shape, seed=5)
    m2, lam = -4.0, 6.0
    emu = orc.flow_sample(shape, w, m2, lam, 64, seed=77, bf16_mask=TC_MODE)
    f32 = orc.flow_sample(shape, w, m2, lam, 64, seed=77, bf16_mask=TC_MODE | orc.F32_ACC | orc.Z_JITTER)
    scale = np.maximum(np.abs(emu["phi"]), np.sqrt((emu["phi"] ** 2).mean(1, keepdims=True)))
    site = 2 * (np.abs(f32["phi"] - emu["phi"]) / scale).max()
    scalar = 2 * max((np.abs(f32[k] - emu[k]) / np.maximum(np.abs(emu[k]), 1.0)).max() for k in ("logq", "S", "logw"))
    flow = P.Flow(shape, w, precision="bf16")
    out = flow.sample(4, seed=31, counter0=2, phi4=(m2, lam))
    ref = orc.flow_sample(shape, w, m2, lam, 4, seed=31, counter0=2, bf16_mask=TC_MODE)
    assert_sites_close(out.phi.cpu().numpy(), ref["phi"], rtol=site)
    for k in ("logq", "S", "logw"):
        assert_logw_close(getattr(out, k).cpu().numpy(), ref[k], rtol=scalar, what=k)
    assert P.device_status() == 0
