"""Rounding error of the streaming action where the hopping sum's bias is coarse next to |S|."""
import numpy as np
import pytest

from gpu_util import require_gpu

pytestmark = pytest.mark.gpu


# m2 and lam at which a configuration's estimated error is about 8e-14 of |S|: within the
# limit at which it was summed again while a fold took 4 sites (1e-13), beyond the present one
@pytest.mark.parametrize("nd,L,m2,lam", [(2, 16, -3.0, 1.0), (2, 32, -3.0, 1.0), (2, 64, -3.5, 1.75),
                                         (3, 8, -4.5, 1.5), (3, 16, -4.0, 1.75)])
def test_action_error_within_the_estimate(nd, L, m2, lam):
    torch, P = require_gpu()
    n, rng = 400, np.random.default_rng(L)
    x = (rng.choice([-0.7, 0.7], (n, 1)) + 0.4 * rng.standard_normal((n, L ** nd))).astype(np.float32)
    S = P.phi4_action(nd, L, (m2, lam), torch.tensor(x, device="cuda")).cpu().numpy()
    y = x.astype(np.longdouble).reshape((n,) + (L,) * nd)
    lap = sum(2 * y - np.roll(y, 1, d) - np.roll(y, -1, d) for d in range(1, nd + 1))
    ref = (y * lap + np.longdouble(m2) * y * y + np.longdouble(lam) * y ** 4).reshape(n, -1).sum(1)
    # a configuration is summed again when the rms estimate of its error exceeds 6e-14 |S|
    assert np.linalg.norm((S - ref).astype(np.float64)) <= 6e-14 * np.linalg.norm(ref.astype(np.float64))
