"""Edges of the chain kernels: the batched MH scan's chunk and batch boundaries
and the lags and cluster sizes of the series reductions, against the oracle."""
import numpy as np
import pytest

import oracle
from gpu_util import require_gpu

pytestmark = pytest.mark.gpu


def _series(kind, n, seed):
    g = np.random.default_rng(seed)
    lw = g.normal(0.0, {"mixed": 1.0, "sticky": 30.0, "free": 1e-3}.get(kind, 1.0), n)
    if kind == "special":                     # NaN, infinities, signed zeros
        lw[g.integers(0, n, n // 7 + 1)] = np.nan
        lw[g.integers(0, n, n // 11 + 1)] = -np.inf
        lw[g.integers(0, n, n // 5 + 1)] = -0.0
        lw[g.integers(0, n, n // 5 + 1)] = 0.0
    return lw


@pytest.mark.parametrize("kind", ["mixed", "sticky", "free", "special"])
@pytest.mark.parametrize("n", [1, 31, 32, 33, 128, 129, 992, 1024, 1025, 3077, 20000])
def test_mh_scan_matches_the_sequential_chain(n, kind):
    torch, P = require_gpu()
    lw = _series(kind, n, n)
    ref_state = oracle.new_mh_state(77, 3)
    ridx, racc = oracle.mh_chain(ref_state, lw)
    t = torch.tensor(lw, device="cuda")
    st = P.new_mh_state(77, 3)
    # one call, and the same chain cut into calls of uneven length
    idx, acc = P.mh_chain(st, t)
    assert (idx.cpu().numpy() == ridx).all() and (acc.cpu().numpy() == racc).all()
    cut = P.new_mh_state(77, 3)
    got = [P.mh_chain(cut, t[a:b].contiguous()) for a, b in ((0, n // 3), (n // 3, n // 2), (n // 2, n)) if b > a]
    assert (torch.cat([i for i, _ in got]).cpu().numpy() == ridx).all()
    assert (torch.cat([a for _, a in got]).cpu().numpy() == racc).all()
    assert torch.equal(st, cut)
    s = P.read_mh_state(st)
    assert s.step == n and s.idx_cur == ridx[-1] and s.n_acc == racc[1:].sum()
    assert np.float64(s.logw_cur).tobytes() == lw[ridx[-1]].tobytes()
    na = P.new_mh_state(77, 3)
    idx2, acc2 = P.mh_chain_noalloc(na, t)
    assert torch.equal(idx2, idx) and torch.equal(acc2, acc) and torch.equal(na, st)


# FP64 sums of n products in any order: about n^(1/2) 2^-53 relative to the sum of magnitudes
@pytest.mark.parametrize("n,t_max", [(1, 0), (2, 1), (40, 39), (1024, 151), (1025, 152), (2047, 7), (2048, 303),
                                     (5000, 1000), (16384, 1300)])
def test_autocorrelation_and_ess_edges(n, t_max):
    torch, P = require_gpu()
    g = np.random.default_rng(n)
    y = np.cumsum(g.normal(size=n)) * 0.1 + 5.0
    gamma, summ = P.autocorr(torch.tensor(y, device="cuda"), t_max)
    d = y - y.mean()
    ref = np.array([np.dot(d[:n - t], d[t:]) / (n - t) for t in range(t_max + 1)])
    scale = np.array([np.dot(np.abs(d[:n - t]), np.abs(d[t:])) / (n - t) for t in range(t_max + 1)])
    # (the mean's rounding, about 2^-52 |mean|, enters twice, times sum |d|)
    tol = 2.0 ** -45 * scale + 2.0 ** -48 * np.abs(y.mean()) * np.abs(d).sum() / n + 1e-300
    assert (np.abs(gamma.cpu().numpy() - ref) <= tol).all()
    tau, W = 0.5, t_max
    gg = gamma.cpu().numpy()
    if gg[0] > 0:
        for t in range(1, t_max + 1):
            tau += gg[t] / gg[0]
            if t >= 5.0 * tau:
                W = t
                break
        assert np.allclose(summ.cpu().numpy(), [tau, W, tau * np.sqrt((4 * W + 2) / n), y.mean()], rtol=1e-12)
    lw = g.normal(100.0, 2.0, n)
    w = np.exp(lw - lw.max())
    assert abs(P.ess(torch.tensor(lw, device="cuda")).item() - w.sum() ** 2 / (n * (w * w).sum())) <= 1e-13
