"""The work that users of this framework have it do, as cases that can be timed and compared.

A user samples lattice configurations from RealNVP flows (FP32, or with the convolutions on the
tensor cores), scores given configurations, trains flows with the reverse KL loss, runs the FP64
HMC comparison sampler and analyses the resulting chains.  `listed()` holds one case for each of
these at the sizes of the framework's own workloads (the paper's 2D L=8 example, the 2D L=32
training flow, the 3D L=16 flow, the serving mix, HMC on 512 chains); `draw()` gives others of the
same ranges.  `exact()` is the same mathematics in 64 bits with plain torch and numpy.
"""
import math
import types

import numpy as np
import torch

import paper_2208_08903_gb300 as P
from paper_2208_08903_gb300 import api, autograd


def listed():
    return [
        # the paper's printed example: a 2D L=8 flow, one batch of 64 proposals and its Metropolis test
        # (the smallest call: launches and latency count)
        dict(name="example_2d8_fp32", kind="sample", nd=2, L=8, layers=16, hidden="8,8", ksize=3,
             precision="fp32", batch=64, mh=True, m2=-4.0, lam=8.0),
        # serving mix, 2D L=32 width 32 at the largest request size, tensor-core precision
        dict(name="sample_2d32_w32_bf16", kind="sample", nd=2, L=32, layers=24, hidden="32,32", ksize=3,
             precision="bf16", batch=8192, mh=False, m2=-4.0, lam=6.0),
        # serving mix, a ragged request of a 3D L=12 width-16 flow, tensor-core precision
        dict(name="sample_3d12_w16_bf16", kind="sample", nd=3, L=12, layers=16, hidden="16,16", ksize=3,
             precision="bf16", batch=999, mh=False, m2=-4.0, lam=6.0),
        # the 3D L=16 flow at its batch of 4096 (the framework's headline workload)
        dict(name="sample_3d16_w32_bf16", kind="sample", nd=3, L=16, layers=16, hidden="32,32", ksize=3,
             precision="bf16", batch=4096, mh=False, m2=-6.0, lam=5.0),
        # serving mix, a model that stays in FP32 because its activations do not fit the tensor-core kernel
        dict(name="sample_3d12_w32_fp32", kind="sample", nd=3, L=12, layers=16, hidden="32,32", ksize=3,
             precision="fp32", batch=300, mh=False, m2=-4.0, lam=6.0),
        # the 3D L=16 flow in plain FP32 (the precision of the paper's software)
        dict(name="sample_3d16_w32_fp32", kind="sample", nd=3, L=16, layers=16, hidden="32,32", ksize=3,
             precision="fp32", batch=608, mh=False, m2=-6.0, lam=5.0),
        # another network of the paper's model section: three hidden convolutions, kernel size 5
        dict(name="sample_2d16_k5_fp32", kind="sample", nd=2, L=16, layers=12, hidden="16,16,8", ksize=5,
             precision="fp32", batch=500, mh=False, m2=-4.0, lam=8.0),
        # log q of given configurations (reweighting, the inverse direction) on a 2D L=64 flow
        dict(name="logq_2d64_w16_bf16", kind="logq", nd=2, L=64, layers=16, hidden="16,16", ksize=3,
             precision="bf16", batch=1500),
        # reverse-KL training step with Adam of the 2D L=32 flow at batch 1024 (forward and backward)
        dict(name="train_2d32_w32", kind="train", nd=2, L=32, layers=24, hidden="32,32", ksize=3,
             batch=1024, m2=-4.0, lam=8.0),
        # the paper's training batch of 64 on a small flow, loss built in torch (autograd front end)
        dict(name="autograd_2d16_w16", kind="autograd", nd=2, L=16, layers=12, hidden="16,16", ksize=3,
             batch=64, m2=-4.0, lam=8.0),
        # the HMC comparison: one trajectory of 512 chains on 3D L=16, FP64
        dict(name="hmc_3d16", kind="hmc", nd=3, L=16, chains=512, steps=20, eps=0.05, m2=-6.0, lam=5.0),
        # analysis of 16,384 proposals: Metropolis chain over their log weights, action, magnetisation,
        # two-point function, chain averages with autocorrelation time, effective sample size
        dict(name="analysis_3d16", kind="analysis", nd=3, L=16, batch=16384, t_max=1000, m2=-6.0, lam=5.0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(["sample", "logq", "train", "autograd", "hmc", "analysis"], [6, 2, 2, 1, 2, 2])[0]
    nd = rng.choice([2, 3])
    m2, lam = round(rng.uniform(-6.0, -2.0), 3), round(rng.uniform(1.0, 10.0), 3)
    L = rng.choice([8, 10, 12, 16, 16, 20, 24, 32, 32, 48, 64] if nd == 2 else [6, 8, 8, 10, 12, 12, 14, 16, 16])
    if kind == "hmc":
        return dict(kind=kind, nd=nd, L=L, chains=_log_int(rng, 16, 512), steps=rng.randint(10, 20),
                    eps=round(rng.uniform(0.01, 0.05), 4), m2=m2, lam=lam)
    if kind == "analysis":
        batch = _log_int(rng, 500, min(65536, 16384 * 4096 // L ** nd))
        return dict(kind=kind, nd=nd, L=L, batch=batch, t_max=min(1000, batch // 4), m2=m2, lam=lam)
    width = rng.choice([8, 16, 24, 32])
    case = dict(kind=kind, nd=nd, L=L, layers=rng.randint(12, 24), hidden=f"{width},{width}", ksize=3)
    if kind in ("train", "autograd"):
        top, low = 1.5e12, 64                          # training runs in FP32
    else:
        case["precision"] = rng.choice(["bf16", "bf16", "fp32"])
        if case["precision"] == "bf16" and not api.tensor_core_supported(_shape(case)):
            case["precision"] = "fp32"
        if case["precision"] == "fp32" and nd == 2 and L <= 16 and rng.random() < 0.3:
            case["hidden"], case["ksize"] = rng.choice([("16", 3), ("8,16", 5), ("16,16,8", 5), ("12,12,12", 3)])
        top, low = (4e12 if case["precision"] == "bf16" else 6e11 if case["ksize"] == 3 else 1.5e11), 64
    case["batch"] = 1
    per = work(dict(case, m2=m2, lam=lam))["flops"]
    case["batch"] = _log_int(rng, low, max(low, min(8192, int(top / per))))
    if kind == "logq":
        return case
    if kind == "sample":
        case["mh"] = rng.random() < 0.3 and case["precision"] == "fp32"
    return dict(case, m2=m2, lam=lam)


# ---------------------------------------------------------------------------
# What a user's program has in hand, and one pass through the public entry points
# ---------------------------------------------------------------------------
def _shape(case):
    h = tuple(int(v) for v in case["hidden"].split(","))
    return types.SimpleNamespace(nd=case["nd"], L=case["L"], n_layers=case["layers"], hidden=h, c1=h[0], c2=h[-1],
                                 ksize=case["ksize"], use_final_tanh=True, leaky_slope=0.01)


def _convs(case):
    ch = (1,) + _shape(case).hidden + (2,)
    return list(zip(ch[:-1], ch[1:]))


def _weights(case, seed):
    """Kaiming-uniform weights (the default of convolution layers), canonical order, FP64."""
    g = np.random.default_rng(seed)
    taps = case["ksize"] ** case["nd"]
    out = []
    for _ in range(case["layers"]):
        for ci, co in _convs(case):
            a = 1.0 / math.sqrt(ci * taps)
            out.append(g.uniform(-a, a, size=co * ci * taps))
            out.append(g.uniform(-a, a, size=co))
    return np.concatenate(out)


def _field(case, n, seed, dtype):
    """Configurations as they come from a thermalised chain: both signs, fluctuations about the minimum."""
    g = torch.Generator(device="cuda").manual_seed(seed + 77)
    V = case["L"] ** case["nd"]
    sign = torch.where(torch.rand(n, 1, device="cuda", dtype=dtype, generator=g) < 0.5, -0.7, 0.7).to(dtype)
    return sign + 0.4 * torch.randn(n, V, device="cuda", dtype=dtype, generator=g)


def _logw(n, seed):
    """Log weights of proposals from a trained flow (a spread of about one)."""
    g = torch.Generator(device="cuda").manual_seed(seed + 99)
    return 50.0 + torch.randn(n, device="cuda", dtype=torch.float64, generator=g)


def prepare(case, seed):
    s = types.SimpleNamespace(case=case, seed=seed, kind=case["kind"], phi4=(case.get("m2", 0.0), case.get("lam", 0.0)))
    if s.kind == "hmc":
        s.phi, s.traj = _field(case, case["chains"], seed, torch.float64), 0
        return s
    if s.kind == "analysis":
        s.phi, s.logw = _field(case, case["batch"], seed, torch.float32), _logw(case["batch"], seed)
        return s
    s.flow = P.Flow(_shape(case), _weights(case, seed), precision=case.get("precision", "fp32"))
    if s.kind == "logq":
        s.phi = _field(case, case["batch"], seed, torch.float32)
    elif s.kind == "train":
        s.m, s.v = (torch.zeros(s.flow.n_params, device="cuda") for _ in range(2))
        s.step = 0
        s.ws = torch.empty(s.flow.train_workspace_bytes(case["batch"]), device="cuda", dtype=torch.uint8)
    elif s.kind == "autograd":
        s.theta = s.flow.get_weights().requires_grad_(True)
    elif case["mh"]:
        s.state0 = api.new_mh_state(seed)
    return s


def run(s):
    c = s.case
    if s.kind == "sample":
        r = s.flow.sample(c["batch"], seed=s.seed, counter0=0, phi4=s.phi4)
        out = dict(phi=r.phi, logq=r.logq, S=r.S, logw=r.logw)
        if c["mh"]:
            out["state"] = s.state0.clone()
            out["chain_idx"], out["accepted"] = api.mh_chain(out["state"], r.logw)
        return out
    if s.kind == "logq":
        z, logq = s.flow.logq(s.phi, return_z=True)
        return dict(z=z, logq=logq)
    if s.kind == "train":
        s.step += 1
        loss, grad = s.flow.train_step(c["batch"], s.phi4, seed=s.seed, counter0=0, lr=1e-3, adam_m=s.m, adam_v=s.v,
                                       adam_t=s.step, workspace=s.ws)
        return dict(loss=loss, grad=grad, adam_m=s.m, adam_v=s.v)
    if s.kind == "autograd":
        s.theta.grad = None
        loss = autograd.reverse_kl_loss(s.flow, s.theta, c["batch"], s.phi4, seed=s.seed, counter0=0)
        loss.backward()
        return dict(loss=loss.detach(), grad=s.theta.grad)
    if s.kind == "hmc":
        dH, acc = api.hmc_trajectory(c["nd"], c["L"], s.phi4, s.phi, c["steps"], c["eps"], s.seed, s.traj)
        s.traj += 1
        return dict(phi=s.phi, dH=dH, accepted=acc)
    state = api.new_mh_state(s.seed)
    idx, acc = api.mh_chain(state, s.logw)
    S = api.phi4_action(c["nd"], c["L"], s.phi4, s.phi)
    M, C = api.observables(c["nd"], c["L"], s.phi)
    series = api.chain_gather(idx, M).abs().contiguous()
    gamma, summary = api.autocorr(series, c["t_max"])
    return dict(chain_idx=idx, accepted=acc, S=S, M=M, C=C, series=series, gamma=gamma, summary=summary,
                ess=api.ess(s.logw))


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    V = case["L"] ** case["nd"]
    if case["kind"] == "hmc":       # force 20, kick 2, drift 2 operations per site and step; field in and out
        return dict(bytes=case["chains"] * (16 * V + 9), flops=24.0 * case["chains"] * V * case["steps"])
    if case["kind"] == "analysis":  # fields once; log weights, chain, S, M, C, series, Gamma
        n = case["batch"]
        return dict(bytes=n * (4 * V + 8 + 9 + 8 + 8 + 8 * case["L"] + 8) + 8 * case["t_max"],
                    flops=float(n) * (V * 3 * (case["nd"] + 3) + 2 * (case["t_max"] + 1)))
    B, T, convs = case["batch"], case["ksize"] ** case["nd"], _convs(case)
    flops, params = 0.0, 0
    for j, (ci, co) in enumerate(convs):
        # the masked input has every other site zero; the head is needed at every other site
        live = T / 2 if j == 0 else T
        flops += 2.0 * V * live * ci * co * (0.5 if j == len(convs) - 1 else 1.0)
        params += ci * co * T + co
    flops *= B * case["layers"]
    params *= case["layers"]
    if case["kind"] in ("train", "autograd"):   # forward, input gradients, weight gradients
        moments = 4 * 2 * params if case["kind"] == "train" else 0
        return dict(bytes=4 * 2 * params + 2 * moments + 8, flops=3 * flops)
    io = 4 * V + 24 + (9 if case.get("mh") else 0) if case["kind"] == "sample" else 8 * V + 8
    return dict(bytes=B * io + 4 * params, flops=flops)


# ---------------------------------------------------------------------------
# The same in 64 bits
# ---------------------------------------------------------------------------
def _mulhilo(a, b):
    m = np.uint64(0xFFFFFFFF)
    s = np.uint64(32)
    al, ah, bl, bh = a & m, a >> s, b & m, b >> s
    t = al * bl
    u = ah * bl + (t >> s)
    v = al * bh + (u & m)
    return ah * bh + (u >> s) + (v >> s), a * b


def _philox(key0, key1, c0, c1, c2, c3):
    """Philox4x64-10 (Salmon et al. 2011) of broadcast uint64 counters: four uint64 arrays."""
    m0, m1 = np.uint64(0xD2E7470EE14C6C93), np.uint64(0xCA5A826395121157)
    w0, w1, full = 0x9E3779B97F4A7C15, 0xBB67AE8584CAA73B, (1 << 64) - 1
    c0, c1, c2, c3 = (np.array(v, dtype=np.uint64) for v in np.broadcast_arrays(c0, c1, c2, c3))
    for r in range(10):
        k0, k1 = np.uint64((key0 + r * w0) & full), np.uint64((key1 + r * w1) & full)
        hi0, lo0 = _mulhilo(c0, m0)
        hi1, lo1 = _mulhilo(c2, m1)
        c0, c1, c2, c3 = hi1 ^ c1 ^ k0, lo1, hi0 ^ c3 ^ k1, lo0
    return c0, c1, c2, c3


def _normals(words, bits):
    """Box-Muller from four words: (2k+1) 2^-(bits+1) with k the top `bits` bits."""
    u = [(2.0 * (w >> np.uint64(64 - bits)).astype(np.float64) + 1.0) * 2.0 ** -(bits + 1) for w in words]
    out = []
    for a, b in ((u[0], u[1]), (u[2], u[3])):
        r = np.sqrt(-2.0 * np.log(a))
        out += [r * np.cos(2 * np.pi * b), r * np.sin(2 * np.pi * b)]
    return np.stack(out, -1)


def _prior(case, seed):
    V, B = case["L"] ** case["nd"], case["batch"]
    b, j = np.arange(B, dtype=np.uint64)[:, None], np.arange((V + 3) // 4, dtype=np.uint64)[None]
    return _normals(_philox(seed, 0, b, j, np.uint64(0), np.uint64(1)), 23).reshape(B, -1)[:, :V]


def _uniforms(seed, n, *counter):
    w = _philox(seed, 0, *counter)[0]
    return (2.0 * (w >> np.uint64(12)).astype(np.float64) + 1.0) * 2.0 ** -53


def _lattice(case, x):
    return x.reshape((-1,) + (case["L"],) * case["nd"])


def _lap(case, x):
    return sum(2 * x - x.roll(1, d) - x.roll(-1, d) for d in range(1, case["nd"] + 1))


def _action(case, x):
    x = _lattice(case, x)
    return (x * _lap(case, x) + case["m2"] * x * x + case["lam"] * x ** 4).flatten(1).sum(1)


def _split(case, w):
    """Per layer [(W [T][ci][co], b [co]), ...] of flat canonical weights."""
    T, at, out = case["ksize"] ** case["nd"], 0, []
    for _ in range(case["layers"]):
        layer = []
        for ci, co in _convs(case):
            W = w[at:at + co * ci * T].reshape(co, ci, T).permute(2, 1, 0)
            at += co * ci * T
            layer.append((W, w[at:at + co]))
            at += co
        out.append(layer)
    return out


def _net(case, layer, x, keep):
    """(s, t) of one coupling layer's network for the lattice field x with the sites `keep` visible."""
    nd, k = case["nd"], case["ksize"]
    h = torch.where(keep, x, torch.zeros_like(x)).unsqueeze(-1)
    for j, (W, b) in enumerate(layer):
        y = b
        for t in range(k ** nd):
            off = [(t // k ** (nd - 1 - d)) % k - k // 2 for d in range(nd)]
            y = y + h.roll([-o for o in off], list(range(1, nd + 1))) @ W[t]
        h = torch.nn.functional.leaky_relu(y, 0.01) if j < len(layer) - 1 else y
    return torch.tanh(h[..., 0]), h[..., 1]


def _flow(case, w, x, inverse):
    """(field, sum of s) of the coupling stack on flat configurations x."""
    n = torch.meshgrid(*[torch.arange(case["L"], device=x.device)] * case["nd"], indexing="ij")
    parity = sum(n) % 2
    x, ld = _lattice(case, x), 0.0
    layers = list(enumerate(_split(case, w)))
    for l, layer in reversed(layers) if inverse else layers:
        keep = parity == l % 2
        s, t = _net(case, layer, x, keep)
        y = (x - t) * torch.exp(-s) if inverse else x * torch.exp(s) + t
        x, ld = torch.where(keep, x, y), ld + torch.where(keep, torch.zeros_like(s), s).flatten(1).sum(1)
    return x.flatten(1), ld


def _logr(z):
    return -0.5 * (z * z).sum(1) - 0.5 * z.shape[1] * math.log(2 * math.pi)


def _exact_flow(case, seed):
    train = case["kind"] in ("train", "autograd")
    V, B = case["L"] ** case["nd"], case["batch"]
    w = torch.from_numpy(_weights(case, seed)).cuda().float().double()
    w.requires_grad_(train)
    if case["kind"] == "logq":
        x0 = _field(case, B, seed, torch.float32).double()
    else:
        x0 = torch.from_numpy(_prior(case, seed)).cuda()
    wide = sum(ci for ci, _ in _convs(case)) * case["ksize"] ** case["nd"] * case["layers"] if train else 4 * 32
    chunk = max(1, int(8e9 / (8 * V * wide)))
    parts, loss = [], 0.0
    for a in range(0, B, chunk):
        z = x0[a:a + chunk]
        with torch.set_grad_enabled(train):
            x, ld = _flow(case, w, z, case["kind"] == "logq")
            logq = _logr(x if case["kind"] == "logq" else z) - ld
            if case["kind"] == "logq":
                parts.append((x, logq))
                continue
            S = _action(case, x)
            if train:
                part = (logq + S).sum() / B
                part.backward()
                loss += part.item()
            else:
                parts.append((x, logq, S, -S - logq))
    if train:
        g = w.grad
        out = dict(loss=torch.full((1,) if case["kind"] == "train" else (), loss, dtype=torch.float64), grad=g)
        return dict(out, adam_m=0.1 * g, adam_v=0.001 * g * g) if case["kind"] == "train" else out
    names = ("z", "logq") if case["kind"] == "logq" else ("phi", "logq", "S", "logw")
    out = dict(zip(names, (torch.cat(p) for p in zip(*parts))))
    return dict(out, state=None, chain_idx=None, accepted=None) if case.get("mh") else out


def _exact_hmc(case, seed):
    c, V, eps = case["chains"], case["L"] ** case["nd"], case["eps"]
    x = start = _field(case, c, seed, torch.float64)
    i, j = np.arange(c, dtype=np.uint64)[:, None], np.arange((V + 3) // 4, dtype=np.uint64)[None]
    pi = torch.from_numpy(_normals(_philox(seed, 0, i, np.uint64(0), j, np.uint64(3)), 52).reshape(c, -1)[:, :V]).cuda()

    def force(x):
        y = _lattice(case, x)
        return (2 * _lap(case, y) + 2 * case["m2"] * y + 4 * case["lam"] * y ** 3).flatten(1)

    H0 = 0.5 * (pi * pi).sum(1) + _action(case, x)
    pi = pi - 0.5 * eps * force(x)
    for k in range(1, case["steps"] + 1):
        x = x + eps * pi
        pi = pi - (eps if k < case["steps"] else 0.5 * eps) * force(x)
    dH = 0.5 * (pi * pi).sum(1) + _action(case, x) - H0
    u = _uniforms(seed, c, np.arange(c, dtype=np.uint64), np.uint64(0), np.uint64(0), np.uint64(4))
    acc = -dH > torch.from_numpy(np.log(u)).cuda()
    return dict(phi=torch.where(acc[:, None], x, start), dH=dH, accepted=None)


def _exact_analysis(case, seed):
    n, L, V = case["batch"], case["L"], case["L"] ** case["nd"]
    x, logw = _field(case, n, seed, torch.float32).double(), _logw(n, seed)
    u = _uniforms(seed, n, np.arange(n, dtype=np.uint64), np.uint64(0), np.uint64(0), np.uint64(2))
    key, lw = (logw.cpu().numpy() - np.log(u)).tolist(), logw.cpu().tolist()
    idx, cur = [], 0
    for k in range(n):
        if k == 0 or key[k] > lw[cur]:
            cur = k
        idx.append(cur)
    M = x.mean(1)
    slices = x.reshape(n, L, -1).sum(2)
    C = torch.stack([(slices * slices.roll(-t, 1)).sum(1) / V for t in range(L)], 1)
    series = M[torch.tensor(idx, device=x.device)].abs()
    y = series - series.mean()
    gamma = torch.stack([(y[:n - t] * y[t:]).sum() / (n - t) for t in range(case["t_max"] + 1)])
    g, tau, W = (gamma / gamma[0]).tolist(), 0.5, case["t_max"]
    for t in range(1, case["t_max"] + 1):
        tau += g[t]
        if t >= 5.0 * tau:
            W = t
            break
    summary = torch.tensor([tau, W, tau * math.sqrt((4 * W + 2) / n), series.mean().item()], dtype=torch.float64)
    e = torch.exp(logw - logw.max())
    return dict(chain_idx=None, accepted=None, S=_action(case, x), M=M, C=C, series=series, gamma=gamma,
                summary=summary, ess=(e.sum() ** 2 / (n * (e * e).sum())).reshape(1))


def exact(case, seed):
    if case["kind"] == "hmc":
        return _exact_hmc(case, seed)
    if case["kind"] == "analysis":
        return _exact_analysis(case, seed)
    if work(case)["flops"] > 6e12:      # about a teraflop a second in 64 bits
        return None
    return _exact_flow(case, seed)
