"""The work that users of this framework give it, as cases that can be timed.

Every case is one call of a training (or inference) loop through the public
entry points: ``Network.set_inputs`` + ``Network.simulate`` + the library's
readout and weight read-back into the caller's device buffers, the stand-alone
learning-signal product, or a predictor call on host arrays.  Networks, inputs
and parameters are drawn from the seed, with the sizes, rates, weights and
constants of the repository's own workloads.

``listed()`` names the cases, ``draw(rng)`` gives more of the same ranges,
``prepare`` builds what the user's program holds, ``run`` is one pass,
``work`` its unavoidable bytes and operations, and ``exact`` the same results
in 64 bits from plain torch for the cases where that is quick.
"""
from __future__ import annotations

import ctypes
import math
import types

import numpy as np
import torch

import paper_2511_21674_gb300 as ep

DEV = "cuda"
FP32, BF16, FP16 = 0, 1, 2


def listed():
    return [
        # the tutorial-sized task: one sample, 20 inputs, 100 LIF neurons,
        # all-to-all, one update per 1000-step call
        dict(name="pattern", family="pattern", n_in=20, n_rec=100, n_out=1, T=1000, launch_mode=1),
        # event-camera classification: a batch of 64 uneven samples in the
        # persistent form, one update per call
        dict(name="events_batch64", family="events", side=34, n_rec=200, n_out=10, batch=64, T=350,
             len_lo=250, U=0, launch_mode=2),
        # the same task with weight updates every 50 steps inside the call
        dict(name="events_windows", family="events", side=34, n_rec=200, n_out=10, batch=64, T=350,
             len_lo=250, U=50, launch_mode=1),
        # the same task with fewer, shorter samples and an odd network size,
        # default launches
        dict(name="events_small", family="events", side=19, n_rec=73, n_out=7, batch=9, T=233,
             len_lo=160, U=0, launch_mode=1),
        # evidence accumulation: long sequences, slow adaptation, Adam
        dict(name="cue_batch32", family="cue", pop=10, n_rec=100, batch=32, n_cues=7, t_delay=1000,
             launch_mode=1),
        # balanced network of 1e5 neurons, 1e8 synapses, FP32 traces
        dict(name="balanced_fp32", family="sparse", n_rec=100_000, k_in=1000, n_out=1, T=1000, U=100,
             trace=FP32),
        # a network of ordinary size with odd dimensions, FP16 traces
        dict(name="balanced_20k", family="sparse", n_rec=20_011, k_in=500, n_out=10, T=500, U=50,
             trace=FP16),
        # the largest: a million neurons, 1e9 synapses, BF16 traces
        dict(name="million_bf16", family="sparse", n_rec=1_000_000, k_in=1000, n_out=100, T=1000, U=100,
             trace=BF16),
        # the scaling experiment's network: in-degree 10,000, long windows
        dict(name="scaling", family="scaling", n_rec=128_000, k_rec=10_000, n_in=1000, k_in=100, n_out=10,
             T=1000, U=1000, trace=BF16),
        # learning signals formed outside a simulation
        dict(name="signals", family="signals", n_rec=1_000_000, n_out=100, U=100, batch=1),
        # the predictor's per-step inference and its training step
        dict(name="predictor_infer", family="predictor", rows=256, n_out=10, hidden=256, train=False),
        dict(name="predictor_train", family="predictor", rows=4096, n_out=10, hidden=256, train=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    family = rng.choice(["pattern", "events", "events", "cue", "sparse", "sparse", "scaling", "signals",
                         "predictor"])
    if family == "pattern":
        return dict(family=family, n_in=_log_int(rng, 5, 60), n_rec=_log_int(rng, 30, 400),
                    n_out=rng.randint(1, 5), T=_log_int(rng, 100, 1500), launch_mode=rng.choice([1, 2]))
    if family == "events":
        U = rng.choice([0, 0, 40, 50])
        T = _log_int(rng, 80, 350)
        if U:
            T = max(2, T // U) * U
        return dict(family=family, side=rng.randint(8, 34), n_rec=_log_int(rng, 40, 320),
                    n_out=rng.randint(2, 12), batch=_log_int(rng, 1, 64), T=T, len_lo=max(1, int(0.7 * T)),
                    U=U, launch_mode=1 if U else rng.choice([1, 2]))
    if family == "cue":
        return dict(family=family, pop=rng.randint(5, 12), n_rec=_log_int(rng, 50, 200),
                    batch=_log_int(rng, 2, 32), n_cues=rng.choice([3, 5, 7]), t_delay=rng.randint(100, 1000),
                    launch_mode=rng.choice([1, 2]))
    if family == "sparse":
        n = _log_int(rng, 4000, 300_000)
        U = rng.choice([20, 50, 100, 125])
        return dict(family=family, n_rec=n, k_in=min(_log_int(rng, 100, 1500), n // 4),
                    n_out=_log_int(rng, 1, 100), T=U * rng.randint(2, 8), U=U,
                    trace=rng.choice([FP32, BF16, FP16]))
    if family == "scaling":
        n = _log_int(rng, 4000, 64_000)
        U = rng.choice([100, 250, 500, 1000])
        return dict(family=family, n_rec=n, k_rec=min(_log_int(rng, 500, 5000), n // 4),
                    n_in=_log_int(rng, 50, 1000), k_in=_log_int(rng, 5, 50), n_out=rng.randint(2, 20), T=U,
                    U=U, trace=rng.choice([FP32, BF16]))
    if family == "signals":
        batch = rng.choice([1, 1, _log_int(rng, 2, 64)])
        return dict(family=family, n_rec=_log_int(rng, 100, 1_000_000 // batch), n_out=_log_int(rng, 1, 200),
                    U=_log_int(rng, 20, 350 if batch > 1 else 128), batch=batch)
    return dict(family=family, rows=_log_int(rng, 16, 4096), n_out=rng.randint(2, 16), hidden=256,
                train=rng.choice([True, False]))


# ------------------------------------------------------------ network parts


class Spec(types.SimpleNamespace):
    """The parameters `Network` takes, with the repository's common values."""

    def __init__(self, **kw):
        base = dict(batch=1, neuron_model=0, dt=1.0, tau_m=20.0, tau_a=200.0, beta_a=0.0, v_th=0.6, t_ref=2,
                    tau_out=20.0, kappa_e=None, gamma=0.5, beta_sg=1.0 / 0.6, loss=0, feedback=0,
                    update_interval=0, continuous=0, lr=1e-3, max_delay=1, drive_weight=0.0, drive_rate=0.0,
                    drive_seed=0, surrogate=0, reset_mode=0, v_reset=0.0, c_reg=0.0, f_target=0.0,
                    beta_reg=0.0, sign_mask=0, optimizer=0, adam_b1=0.9, adam_b2=0.999, adam_eps=1e-7,
                    if_period=0, if_seed=0, d_out=0, d_ls=0)
        base.update(kw)
        super().__init__(**base)

    def drive_thresholds(self):
        """floor(2^32 CDF(m)) of the Poisson drive."""
        if self.drive_weight == 0.0 or self.drive_rate <= 0.0:
            return np.zeros(0, np.uint32)
        thr, p, m = [], math.exp(-self.drive_rate), 0
        cdf = p
        while cdf < 1.0 - 1e-12 and m < 63:
            thr.append(min(int(math.floor(cdf * 4294967296.0)), 4294967295))
            m += 1
            p *= self.drive_rate / m
            cdf += p
        return np.asarray(thr, np.uint32)


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 1000003 + 17)
    return g


def _randn(g, *shape, std=1.0):
    return torch.randn(*shape, generator=g, device=DEV) * std


def _lists(raster):
    """Raster [B, T, n] (bool) -> per-step spike lists on the host."""
    B, T, n = raster.shape
    flat = raster.reshape(B * T, n)
    ptr = torch.zeros(B * T + 1, dtype=torch.int64, device=DEV)
    ptr[1:] = torch.cumsum(flat.sum(1), 0)
    return ptr.cpu().numpy(), flat.nonzero()[:, 1].to(torch.int32).cpu().numpy()


def _sinusoids(g, T, n_out):
    """Sum of four sinusoids per readout: periods U[100, 1000], amplitudes
    U[0.5, 2], random phases."""
    t = torch.arange(1, T + 1, device=DEV, dtype=torch.float64)[:, None, None]
    u = torch.rand(3, n_out, 4, generator=g, device=DEV, dtype=torch.float64)
    s = (0.5 + 1.5 * u[1]) * torch.sin(2 * math.pi * (t / (100.0 + 900.0 * u[0]) + u[2]))
    return (s.sum(2) / 4.0).float().cpu().numpy()[None]


def _dense_csr(mask, W):
    """Rows = sources, columns = targets, delay 1."""
    ptr = torch.zeros(mask.shape[0] + 1, dtype=torch.int64, device=DEV)
    ptr[1:] = torch.cumsum(mask.sum(1), 0)
    col = mask.nonzero()[:, 1].to(torch.int32)
    return ptr, col, W[mask].contiguous(), torch.ones(col.shape[0], dtype=torch.uint8, device=DEV)


def _indegree_csr(g, n_pre, n_post, k, max_delay, same):
    """Fixed in-degree k without multapses (one source per stratum) and, in a
    recurrent population, without autapses: CSR by source, targets ascending."""
    span = n_pre - 1 if same else n_pre
    s = span // k
    key = torch.empty(n_post * k, dtype=torch.int64, device=DEV)
    rows = max(1, 50_000_000 // k)
    m = torch.arange(k, device=DEV, dtype=torch.int64)[None, :] * s
    for j0 in range(0, n_post, rows):
        j1 = min(n_post, j0 + rows)
        j = torch.arange(j0, j1, device=DEV, dtype=torch.int64)[:, None]
        pre = m + torch.randint(0, s, (j1 - j0, k), generator=g, device=DEV)
        if same:
            pre += j + 1
            pre %= n_pre
        pre *= n_post
        pre += j
        pre *= 8
        if max_delay > 1:
            pre += torch.randint(0, max_delay, (j1 - j0, k), generator=g, device=DEV)
        key[j0 * k:j1 * k] = pre.reshape(-1)
        del pre
    key = torch.sort(key).values
    delay = ((key & 7) + 1).to(torch.uint8)
    key >>= 3
    pre = torch.div(key, n_post, rounding_mode="floor")
    col = (key - pre * n_post).to(torch.int32)
    del key
    ptr = torch.zeros(n_pre + 1, dtype=torch.int64, device=DEV)
    bounds = torch.arange(1, n_pre + 1, device=DEV, dtype=torch.int64)
    ptr[1:] = torch.searchsorted(pre, bounds)
    return ptr, col, delay, pre


def _pattern(case, seed):
    g = _gen(seed)
    n_in, n, K, T = case["n_in"], case["n_rec"], case["n_out"], case["T"]
    spec = Spec(n_in=n_in, n_rec=n, n_out=K, T=T, lr=1e-3 / T)
    W = torch.cat([_randn(g, n_in, n, std=n_in ** -0.5), _randn(g, n, n, std=n ** -0.5)])
    mask = torch.ones(n_in + n, n, dtype=torch.bool, device=DEV)
    mask[n_in:].fill_diagonal_(False)
    w_out = _randn(g, n, K, std=n ** -0.5)
    x = torch.rand(1, T, n_in, generator=g, device=DEV) < 0.05
    inputs = (*_lists(x), _sinusoids(g, T, K), np.ones((1, T), np.uint8), np.full(1, T, np.int32))
    return spec, W, mask, w_out, inputs


def _events(case, seed):
    g = _gen(seed)
    side, n, K, B, T = case["side"], case["n_rec"], case["n_out"], case["batch"], case["T"]
    n_in = 2 * side * side
    spec = Spec(n_in=n_in, n_rec=n, n_out=K, T=T, batch=B, neuron_model=1, beta_a=1.7, loss=1, lr=1e-4,
                update_interval=case["U"])
    W = torch.cat([_randn(g, n_in, n, std=3.0 * n_in ** -0.5), _randn(g, n, n, std=(0.1 * n) ** -0.5)])
    mask = torch.ones(n_in + n, n, dtype=torch.bool, device=DEV)
    # recurrent in-degree 10 %, no autapses (a fixed number of synapses)
    order = torch.rand(n, n, generator=g, device=DEV)
    order.fill_diagonal_(2.0)
    mask[n_in:] = False
    mask[n_in:].scatter_(0, order.argsort(0)[:max(1, (n - 1) // 10)], True)
    w_out = _randn(g, n, K, std=n ** -0.5)
    # class blobs whose centre moves along three saccade legs
    cls = torch.randint(0, K, (B,), generator=g, device=DEV)
    lengths = torch.randint(case["len_lo"], T + 1, (B,), generator=g, device=DEV)
    centre = side * (0.25 + 0.5 * torch.rand(K, 2, generator=g, device=DEV))
    sigma = 2.5 + 2.0 * torch.rand(K, generator=g, device=DEV)
    t = torch.arange(T, device=DEV)
    leg = torch.clamp(t // 100, max=2)
    corner = torch.tensor([[-2.0, -2.0], [0.0, 2.0], [2.0, -2.0], [-2.0, -2.0]], device=DEV)
    shift = corner[leg] + (corner[leg + 1] - corner[leg]) * ((t % 100) / 100.0)[:, None]
    c = centre[cls][:, None, :] + shift[None]                                   # [B, T, 2]
    grid = torch.arange(side, device=DEV, dtype=torch.float32)
    d2 = (grid[:, None] - c[..., 0, None, None]) ** 2 + (grid - c[..., 1, None, None]) ** 2
    sg = sigma[cls][:, None, None, None]
    on = torch.exp(-d2 / (2 * sg ** 2)).reshape(B, T, -1)
    off = torch.exp(-(d2.sqrt() - 2 * sg) ** 2 / (2 * sg ** 2)).reshape(B, T, -1)
    rate = torch.cat([on, off], 2)
    rate *= (4000.0 / 300.0) / rate.sum(2, keepdim=True)
    live = t[None, :] < lengths[:, None]
    x = (torch.rand(B, T, n_in, generator=g, device=DEV) < rate) & live[..., None]
    targets = torch.zeros(B, T, K, device=DEV)
    targets[torch.arange(B, device=DEV), :, cls] = 1.0
    window = live & (t[None, :] >= lengths[:, None] - 25)
    inputs = (*_lists(x), targets.cpu().numpy(), window.to(torch.uint8).cpu().numpy(),
              lengths.to(torch.int32).cpu().numpy())
    return spec, W, mask, w_out, inputs


def _cue(case, seed):
    g = _gen(seed)
    pop, n, B, n_cues = case["pop"], case["n_rec"], case["batch"], case["n_cues"]
    n_in, T = 4 * pop, n_cues * 150 + case["t_delay"] + 150
    spec = Spec(n_in=n_in, n_rec=n, n_out=2, T=T, batch=B, neuron_model=1, tau_a=2000.0, beta_a=1.7, loss=1,
                lr=1e-4, optimizer=1)
    W = torch.cat([_randn(g, n_in, n, std=n_in ** -0.5), _randn(g, n, n, std=n ** -0.5)])
    mask = torch.ones(n_in + n, n, dtype=torch.bool, device=DEV)
    mask[n_in:].fill_diagonal_(False)
    w_out = _randn(g, n, 2, std=n ** -0.5)
    side = torch.randint(0, 2, (B, n_cues), generator=g, device=DEV)
    label = (side.sum(1) * 2 > n_cues).long()
    rate = torch.zeros(B, T, 4, device=DEV)
    rate[..., 3] = 10.0
    for q in range(n_cues):
        rate[torch.arange(B, device=DEV), q * 150:q * 150 + 100, side[:, q]] = 40.0
    rate[:, T - 150:, 2] = 40.0
    x = torch.rand(B, T, n_in, generator=g, device=DEV) < rate.repeat_interleave(pop, 2) / 1000.0
    targets = torch.zeros(B, T, 2, device=DEV)
    targets[torch.arange(B, device=DEV), :, label] = 1.0
    window = np.zeros((B, T), np.uint8)
    window[:, T - 150:] = 1
    inputs = (*_lists(x), targets.cpu().numpy(), window, np.full(B, T, np.int32))
    return spec, W, mask, w_out, inputs


DENSE = dict(pattern=_pattern, events=_events, cue=_cue)


def _no_inputs(T):
    return np.zeros(T + 1, np.int64), np.zeros(0, np.int32)


def _sparse(case, seed):
    """Excitatory/inhibitory network with fixed in-degree, delays 1..5,
    Poisson drive and random feedback; the recurrent strength k J is kept."""
    g = _gen(seed)
    n, k, K, T = case["n_rec"], case["k_in"], case["n_out"], case["T"]
    million = K >= 100
    spec = Spec(n_in=0, n_rec=n, n_out=K, T=T, feedback=1, update_interval=case["U"], continuous=1, lr=1e-8,
                max_delay=5, drive_weight=0.03 if million else 0.04, drive_rate=0.85 if million else 1.2,
                drive_seed=seed * 7919 + 17)
    ptr, col, delay, pre = _indegree_csr(g, n, n, k, 5, True)
    J = 10.0 / k
    w = torch.where(pre < int(0.8 * n), J, -5.0 * J).float()
    del pre
    w_out = _randn(g, n, K, std=n ** -0.5)
    fb = _randn(g, n, K, std=K ** -0.5)
    inputs = (*_no_inputs(T), _sinusoids(g, T, K), np.ones((1, T), np.uint8), np.full(1, T, np.int32))
    return spec, (ptr, col, w, delay, w_out, None, fb), inputs


def _scaling(case, seed):
    """Ignore-and-fire neurons at 5 Hz, Poisson inputs at 5 Hz, sparse readout
    (in-degree n / 128) and feedback (out-degree 100 per readout)."""
    g = _gen(seed)
    n, n_in, K, T = case["n_rec"], case["n_in"], case["n_out"], case["T"]
    spec = Spec(n_in=n_in, n_rec=n, n_out=K, T=T, feedback=1, update_interval=case["U"], continuous=1,
                lr=1e-6, max_delay=5, if_period=200, if_seed=seed * 7919 + 29)
    p0, c0, d0, _ = _indegree_csr(g, n_in, n, min(case["k_in"], n_in), 1, False)
    p1, c1, d1, pre = _indegree_csr(g, n, n, case["k_rec"], 5, True)
    w = torch.cat([torch.full((c0.shape[0],), 0.001, device=DEV),
                   torch.where(pre < int(0.8 * n), 0.001, -0.005).float()])
    del pre
    ptr = torch.cat([p0, p1[1:] + p0[-1]])
    col, delay = torch.cat([c0, c1]), torch.cat([d0, d1])
    del c0, c1, d0, d1
    k_out = max(1, n // 128)
    mask = torch.rand(n, K, generator=g, device=DEV) < k_out / n
    w_out = _randn(g, n, K, std=k_out ** -0.5) * mask
    fb = _randn(g, n, K) * (torch.rand(n, K, generator=g, device=DEV) < min(1.0, 100.0 / n))
    x = torch.rand(1, T, n_in, generator=g, device=DEV) < 0.005
    inputs = (*_lists(x), _sinusoids(g, T, K), np.ones((1, T), np.uint8), np.full(1, T, np.int32))
    return spec, (ptr, col, w, delay, w_out, mask.to(torch.uint8), fb), inputs


SPARSE = dict(sparse=_sparse, scaling=_scaling)


# ------------------------------------------------------------ the interface


def _host_rows(case, seed):
    """Predictor rows: readout potentials and 64 group rates, error targets."""
    rng = np.random.default_rng(seed)
    R, K = case["rows"], case["n_out"]
    x = np.concatenate([rng.standard_normal((R, K)) * 2.0, rng.exponential(15.0, (R, 64))], 1)
    return x.astype(np.float32), (rng.standard_normal((R, K)) * 0.3).astype(np.float32)


def _predictor_params(case, seed):
    rng = np.random.default_rng(seed + 99)
    n_in, H, K = case["n_out"] + 64, case["hidden"], case["n_out"]
    p = dict(W1=rng.standard_normal((n_in, H)) / math.sqrt(n_in), b1=0.01 * rng.standard_normal(H),
             W2=rng.standard_normal((H, H)) / math.sqrt(H), b2=0.01 * rng.standard_normal(H),
             W3=rng.standard_normal((H, K)) / math.sqrt(H), b3=0.01 * rng.standard_normal(K))
    scale = np.concatenate([np.full(K, 0.5), np.full(64, 1.0 / 15.0)]).astype(np.float32)
    return {k: v.astype(np.float32) for k, v in p.items()}, scale


LR_PREDICTOR = 1e-3


def prepare(case, seed):
    s = types.SimpleNamespace(case=case)
    if case["family"] == "signals":
        g = _gen(seed)
        s.fb = _randn(g, case["n_rec"], case["n_out"], std=case["n_out"] ** -0.5)
        s.E = _randn(g, case["batch"], case["U"], case["n_out"])
        return s
    if case["family"] == "predictor":
        s.x, s.e = _host_rows(case, seed)
        p, scale = _predictor_params(case, seed)
        s.pred = ep.Predictor(case["n_out"] + 64, case["n_out"], hidden=case["hidden"], max_rows=case["rows"],
                              params=ep.Predictor.pack(p))
        s.pred.set_input_scale(scale)
        return s
    if case["family"] in DENSE:
        spec, W, mask, w_out, s.inputs = DENSE[case["family"]](case, seed)
        s.net = ep.Network(spec, *_dense_csr(mask, W), w_out, launch_mode=case["launch_mode"])
        s.grads = True
    else:
        spec, net, s.inputs = SPARSE[case["family"]](case, seed)
        torch.cuda.empty_cache()
        s.net = ep.Network(spec, *net, trace_dtype=case["trace"], record_grad=0)
        del net
        s.grads = False
    torch.cuda.empty_cache()
    f = dict(dtype=torch.float32, device=DEV)
    n = s.net
    s.out = dict(y=torch.empty(spec.batch, spec.T, spec.n_out, **f), loss=torch.empty(spec.batch, **f),
                 w_in=torch.empty(n.nnz_in, **f), w_rec=torch.empty(n.nnz - n.nnz_in, **f),
                 w_out=torch.empty(spec.n_rec, spec.n_out, **f))
    if s.grads:
        s.out.update({"g" + k[1:]: torch.empty_like(v) for k, v in s.out.items() if k.startswith("w_")})
    torch.cuda.synchronize()
    return s


def _ok(net, status):
    if status != 0:
        raise ep.EpropError(status, net.lib.eprop_last_error(net.h).decode())


def _ptr(t):
    return None if t is None or t.numel() == 0 else ctypes.c_void_p(t.data_ptr())


def run(state):
    case = state.case
    if case["family"] == "signals":
        return ep.learning_signals(state.fb, state.E)
    if case["family"] == "predictor":
        if not case["train"]:
            return state.pred.forward(state.x)
        loss = state.pred.train_step(state.x, state.e, LR_PREDICTOR)
        return dict(loss=loss, params=state.pred.read("params"))
    net, out = state.net, state.out
    net.set_inputs(*state.inputs)
    net.simulate()
    _ok(net, net.lib.eprop_readout(net.h, _ptr(out["y"]), _ptr(out["loss"]), None, 1))
    for proj, key in ((ep.PROJ_IN, "_in"), (ep.PROJ_REC, "_rec"), (ep.PROJ_OUT, "_out")):
        w = out["w" + key]
        if w.numel():
            _ok(net, net.lib.eprop_read_weights_grads(net.h, proj, _ptr(w), _ptr(out.get("g" + key)), 1))
    return out


def work(case):
    f = case["family"]
    if f == "signals":
        n, U, K, B = case["n_rec"], case["U"], case["n_out"], case["batch"]
        return dict(bytes=4 * (n * K + B * U * K + B * U * n), flops=2 * B * U * n * K)
    if f == "predictor":
        R, K, H = case["rows"], case["n_out"], case["hidden"]
        p = (K + 64) * H + H * H + H * K
        if case["train"]:
            return dict(bytes=4 * (R * (2 * K + 64) + 8 * p), flops=6 * R * p)
        return dict(bytes=4 * (R * (2 * K + 64) + p), flops=2 * R * p)
    # a simulation: synapse records (target and delay 4, weight 4 read and 4
    # written, 4 read back and 4 returned, the carried trace read and
    # written), inputs and outputs; operations per neuron step and per
    # synapse event
    if f in DENSE:
        n, K, B = case["n_rec"], case.get("n_out", 2), case.get("batch", 1)
        if f == "pattern":
            n_in, T, ev = case["n_in"], case["T"], 0.05 * case["n_in"]
            nnz = n_in * n + n * (n - 1)
        elif f == "events":
            n_in, T, ev = 2 * case["side"] ** 2, case["T"], 13.3
            nnz = n_in * n + 0.1 * n * (n - 1)
        else:
            n_in, T, ev = 4 * case["pop"], case["n_cues"] * 150 + case["t_delay"] + 150, 0.015 * 4 * case["pop"]
            nnz = n_in * n + n * (n - 1)
        trace = 0
        events = B * T * (ev * n + 0.01 * nnz)
    else:
        n, K, B, T = case["n_rec"], case["n_out"], 1, case["T"]
        nnz = n * case["k_in"] if f == "sparse" else n * (case["k_rec"] + min(case["k_in"], case["n_in"]))
        trace = 4 if case["trace"] == FP32 else 2
        events = 0.005 * T * nnz
    return dict(bytes=nnz * (20 + 2 * trace) + 8 * n * K + 8 * B * T * K, flops=4 * events + 20 * B * T * n)


# --------------------------------------------------- the same in 64 bits


def exact(case, seed):
    if case["family"] == "signals":
        s = prepare(case, seed)
        return torch.einsum("buk,jk->buj", s.E.double(), s.fb.double())
    if case["family"] == "predictor":
        return _exact_predictor(case, seed)
    if case["family"] in DENSE:
        return _exact_dense(*DENSE[case["family"]](case, seed))
    return None          # networks of up to 1e9 synapses: no quick 64-bit form


def _exact_predictor(case, seed):
    p, scale = _predictor_params(case, seed)
    x, e = _host_rows(case, seed)
    names = ("W1", "b1", "W2", "b2", "W3", "b3")
    P = [torch.tensor(p[k], dtype=torch.float64, device=DEV, requires_grad=True) for k in names]
    X = torch.tensor(x, dtype=torch.float64, device=DEV) * torch.tensor(scale, dtype=torch.float64, device=DEV)
    gelu = torch.nn.functional.gelu
    Y = gelu(gelu(X @ P[0] + P[1]) @ P[2] + P[3]) @ P[4] + P[5]
    if not case["train"]:
        return Y.detach()
    loss = 0.5 * ((Y - torch.tensor(e, dtype=torch.float64, device=DEV)) ** 2).sum() / case["rows"]
    loss.backward()
    # the first Adam step: m / (1 - b1) = g, v / (1 - b2) = g^2
    flat = torch.cat([(q - LR_PREDICTOR * q.grad / (q.grad.abs() + 1e-8)).detach().reshape(-1) for q in P])
    return dict(loss=float(loss.detach()), params=flat)


def _exact_dense(spec, W, mask, w_out, inputs):
    """Time-driven e-prop of one call on dense matrices (delay 1)."""
    f64 = dict(dtype=torch.float64, device=DEV)
    x_ptr, x_ids, targets, window, lengths = inputs
    B, T, n, n_in, K = spec.batch, spec.T, spec.n_rec, spec.n_in, spec.n_out
    U = spec.update_interval or T
    c32 = lambda v: float(np.float32(v))  # noqa: E731  (constants are FP32 fields)
    alpha, rho, kappa = (math.exp(-1.0 / t) for t in (spec.tau_m, spec.tau_a, spec.tau_out))
    v_th, gamma, bsg, lr = c32(spec.v_th), c32(spec.gamma), c32(spec.beta_sg), c32(spec.lr)
    alif = spec.neuron_model == 1
    beta = c32(spec.beta_a) if alif else 0.0
    x = torch.zeros(B * T, n_in, **f64)
    rows = torch.repeat_interleave(torch.arange(B * T), torch.as_tensor(np.diff(x_ptr)))
    x[rows.to(DEV), torch.as_tensor(x_ids, device=DEV).long()] = 1.0
    x = x.reshape(B, T, n_in)
    W, M = torch.where(mask, W, 0.0).double(), mask.double()
    Wo = w_out.double()
    tgt, win = torch.as_tensor(targets, **f64), torch.as_tensor(window, **f64)
    length = torch.as_tensor(lengths, device=DEV)
    z = torch.zeros(B, n, **f64)
    v, a, zf, ref = z.clone(), z.clone(), z.clone(), z.clone()
    psi_prev = z.clone()
    zbar = torch.zeros(B, n_in + n, **f64)
    ebar = torch.zeros(B, n_in + n, n, **f64)
    eps = torch.zeros_like(ebar) if alif else None
    y, loss, ys = torch.zeros(B, K, **f64), torch.zeros(B, **f64), []
    G, Go = torch.zeros_like(W), torch.zeros_like(Wo)
    gsum, gosum = torch.zeros_like(W), torch.zeros_like(Wo)
    m = [torch.zeros_like(W), torch.zeros_like(Wo)]
    s2 = [torch.zeros_like(W), torch.zeros_like(Wo)]
    src = torch.zeros(B, n_in + n, **f64)
    for t in range(T):
        live = (t < length).double()[:, None]
        if alif:
            a = rho * a + z
        vth = v_th + beta * a
        v = alpha * v + src @ W - z * vth
        free = (ref <= 0).double() * live
        psi = gamma * torch.clamp(1.0 - bsg * (v - vth).abs(), min=0.0) * free
        z = (v - vth > 0).double() * free
        ref = torch.where(z > 0, float(spec.t_ref), ref - (ref > 0).double())
        if alif:
            eps = psi_prev[:, None, :] * zbar[:, :, None] + (rho - beta * psi_prev)[:, None, :] * eps
        zbar = alpha * zbar + src
        ebar = kappa * ebar + psi[:, None, :] * (zbar[:, :, None] - (beta * eps if alif else 0.0))
        psi_prev = psi
        zf = kappa * zf + z
        y = kappa * y + z @ Wo
        ys.append(y * live)
        wt = (win[:, t] * live[:, 0])[:, None]
        if spec.loss == 0:
            E = wt * (y - tgt[:, t])
            loss += 0.5 * (wt * (y - tgt[:, t]) ** 2).sum(1)
        else:
            E = wt * (torch.softmax(y, 1) - tgt[:, t])
            loss += -(wt * tgt[:, t] * torch.log_softmax(y, 1)).sum(1)
        L = E @ Wo.T
        G += torch.einsum("bj,bij->ij", L, ebar)
        Go += zf.T @ E
        src = torch.cat([x[:, t], z], 1)
        if (t + 1) % U == 0:
            G, Go = G * M / B, Go / B
            gsum += G
            gosum += Go
            if spec.optimizer == 1:
                k = (t + 1) // U
                b1, b2, eh = c32(spec.adam_b1), c32(spec.adam_b2), c32(spec.adam_eps)
                eta = lr * math.sqrt(1 - b2 ** k) / (1 - b1 ** k)
                for q, (w_, g_) in enumerate(((W, G), (Wo, Go))):
                    m[q] = b1 * m[q] + (1 - b1) * g_
                    s2[q] = b2 * s2[q] + (1 - b2) * g_ * g_
                    w_ -= eta * m[q] / (s2[q].sqrt() + eh)
            else:
                W -= lr * G
                Wo -= lr * Go
            G, Go = torch.zeros_like(W), torch.zeros_like(Wo)
    i, r = mask[:n_in], mask[n_in:]
    return dict(y=torch.stack(ys, 1), loss=loss, w_in=W[:n_in][i], w_rec=W[n_in:][r], w_out=Wo,
                g_in=gsum[:n_in][i], g_rec=gsum[n_in:][r], g_out=gosum)
