"""The fused FP32 kernel's tiles, CTA sizes and weight staging against the oracle.

A launch picks its conv2 tile and CTA size from the batch; the results must not
depend on that.  Shapes: lattices that are no multiple of a warp's 32 sites or
of the slices per phase, every width, the smallest lattice, more than 1,024
sites (the other summation order), several stages of weights per pass, and two
whose activations leave no room to stage weights in shared memory.
"""
import numpy as np
import pytest

import gf_inputs as gi
import oracle
from gpu_util import require_gpu

pytestmark = pytest.mark.gpu

SHAPES = [(2, 2, 8), (2, 6, 8), (2, 8, 24), (2, 10, 16), (2, 16, 32), (2, 36, 24), (2, 64, 32),
          (3, 4, 24), (3, 6, 8), (3, 6, 32), (3, 10, 16), (3, 12, 32), (3, 14, 24), (3, 18, 24), (3, 22, 16)]


@pytest.mark.parametrize("nd,L,width", SHAPES)
def test_every_batch_size_gives_the_oracles_results(nd, L, width):
    torch, P = require_gpu()
    shape = gi.FlowShape(nd, L, 3, width, width)
    w = gi.init_weights(shape, seed=4)
    flow = P.Flow(shape, w)
    phi4 = (-4.0, 6.0)
    # one CTA per SM and fewer, several CTAs per SM, more configurations than resident CTAs
    batches = [2, 150, 700, 2500] if L ** nd <= 1024 else [2, 150, 310]
    runs = [flow.sample(B, seed=11, counter0=5, phi4=phi4, return_z=True) for B in batches]
    for r in runs[1:]:
        for k in ("phi", "logq", "S", "logw", "z"):
            assert torch.equal(getattr(r, k)[:2], getattr(runs[0], k)), (k, r.phi.shape)
    big = runs[-1]
    one = flow.sample(1, seed=11, counter0=5 + batches[-1] - 1, phi4=phi4)
    assert torch.equal(one.phi[0], big.phi[-1]) and torch.equal(one.logw[0], big.logw[-1])
    # the FP32 path's stated tolerances: 1e-5 per site, 1e-4 per log weight
    ref = oracle.flow_sample(shape, w, *phi4, 2, seed=11, counter0=5)
    phi = runs[0].phi.cpu().numpy()
    rms = np.sqrt((ref["phi"] ** 2).mean(1, keepdims=True))
    assert (np.abs(phi - ref["phi"]) <= 1e-5 * np.maximum(np.abs(ref["phi"]), rms)).all()
    for k in ("logq", "S", "logw"):
        v = getattr(runs[0], k).cpu().numpy()
        assert (np.abs(v - ref[k]) <= 1e-4 * np.maximum(np.abs(ref[k]), 1)).all(), k
    # the inverse gives z back; it amplifies a site's rounding by at most e per
    # updating layer, on the scale of the largest |z|
    z, logq = flow.logq(big.phi, return_z=True)
    assert (z - big.z).abs().max().item() <= 1e-5 * np.e ** 3 * big.z.abs().max().item()
    assert ((logq - big.logq).abs() <= 1e-4 * big.logq.abs().clamp(min=1)).all()
    assert P.device_status() == 0
