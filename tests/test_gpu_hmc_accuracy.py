"""Rounding errors of the HMC trajectory: the field and dH against extended precision."""
import numpy as np
import pytest

import oracle
from gpu_util import require_gpu

pytestmark = pytest.mark.gpu

LD = np.longdouble


def _trajectory(nd, L, m2, lam, phi, steps, eps, seed, dtype):
    """Fields and dH of one trajectory per chain in extended precision; dtype FP64: the
    momenta and the field rounded once per step, everything else exact."""
    x, chains = phi.astype(LD).reshape((-1,) + (L,) * nd), len(phi)
    pi = np.stack([oracle.hmc_momenta(L ** nd, seed, c, 0) for c in range(chains)]).astype(LD).reshape(x.shape)
    axes, m2, lam, eps = range(1, nd + 1), LD(m2), LD(lam), LD(eps)
    once = lambda v: v.astype(dtype).astype(LD)
    lap = lambda x: sum(2 * x - np.roll(x, 1, d) - np.roll(x, -1, d) for d in axes)
    force = lambda x: 2 * lap(x) + 2 * m2 * x + 4 * lam * x ** 3
    H = lambda x, pi: (pi * pi / 2 + x * lap(x) + m2 * x * x + lam * x ** 4).reshape(chains, -1).sum(1)
    H0 = H(x, pi)
    pi = once(pi - eps / 2 * force(x))
    for i in range(1, steps + 1):
        x = once(x + eps * pi)
        pi = once(pi - (eps if i < steps else eps / 2) * force(x))
    return x.reshape(chains, -1), H(x, pi) - H0


def _run(nd, L, m2, lam, phi, steps, eps, seed):
    torch, P = require_gpu()
    t = torch.tensor(phi, device="cuda")
    dH, acc = P.hmc_trajectory(nd, L, (m2, lam), t, steps, eps, seed=seed, traj_index=0)
    return t.cpu().numpy(), dH.cpu().numpy(), acc.cpu().numpy().astype(bool)


@pytest.mark.parametrize("nd,L", [(3, 6), (2, 16)])
def test_field_error_is_that_of_one_rounding_a_step(nd, L):
    # A free massive field: every coefficient acts on every step, so a rounded one adds
    # up.  Bound: twice the error of rounding momentum and field once per step (the
    # form with the force written out has 1.05 of it, coefficients that carry the step 3.9).
    m2, lam, steps, eps, chains = 0.5, 0.0, 40, 0.06, 24
    rng = np.random.default_rng(5)
    phi = rng.choice([-0.7, 0.7], (chains, 1)) + 0.4 * rng.standard_normal((chains, L ** nd))
    got, _, acc = _run(nd, L, m2, lam, phi, steps, eps, 7)
    exact, _ = _trajectory(nd, L, m2, lam, phi, steps, eps, 7, LD)
    once, _ = _trajectory(nd, L, m2, lam, phi, steps, eps, 7, np.float64)
    assert acc.sum() >= chains // 2
    off = lambda v: float(np.linalg.norm((v.astype(LD) - exact)[acc]))
    assert off(got) <= 2.0 * off(once)


@pytest.mark.parametrize("nd,L", [(3, 8), (2, 16), (3, 5)])
def test_dH_of_a_smooth_large_field(nd, L):
    # H is a sum of positive terms of about 1; a sum that takes phi^2 (2500) apart from
    # its neighbours' products loses 2500 units in the last place of it instead.
    # Bound: 64 roundings of H (a thread's 2 x 10 additions a site, 5 + 8 over the block).
    chains, steps, eps = 24, 4, 0.02
    rng = np.random.default_rng(3)
    phi = 50.0 + 0.1 * rng.standard_normal((chains, L ** nd))
    _, dH, _ = _run(nd, L, 0.0, 0.0, phi, steps, eps, 11)
    _, ref = _trajectory(nd, L, 0.0, 0.0, phi, steps, eps, 11, LD)
    H = L ** nd * (0.5 + 2 * nd * 0.01)
    assert np.abs(dH - ref.astype(np.float64)).max() <= 64 * 2.0 ** -53 * H
