"""The work whose speed is measured: calls that a user of the library makes, through its public entry points.

A "monitor" case is one bfm.monitor() call on a device-resident scene (synthetic: season + noise + steps + cloud runs),
"batch" one replay of a bfm.Batch of uneven tiles, "trace" one bfm.trace() of chosen pixels, "lambda" one
bfm.bfm_lambda() simulation.  Copies between host and device are not among them: their time is the host link's.
"""
import math

import numpy as np
import torch

import paper_1807_01751_gb300 as bfm

F = 23.0  # 16-day revisit: 23 dates make a year
CHUNK = 1 << 17  # pixels per step of the 64-bit evaluation

# lambda(alpha = 0.05, h = 0.25, N/n) as the simulation gives it
LAMBDA = {1.2: 1.3398, 1.4: 1.5277, 1.6: 1.6239, 1.8: 1.6876, 2.0: 1.7325, 2.2: 1.7722, 2.4: 1.8015, 2.6: 1.8266,
          2.8: 1.8487, 3.0: 1.8624}


def _monitor(name, dtype, m, N, n_hist, k, miss, mask=False, extremes=False, complete=False):
    return dict(name=name, kind="monitor", dtype=dtype, m=m, N=N, n_hist=n_hist, k=k, miss=miss, h=0.25, mask=mask,
                extremes=extremes, complete=complete)


def listed():
    return [
        # one small tile on its own (interactive use): launch and latency
        _monitor("small tile", "f32", 4096, 228, 100, 3, 0.3),
        # a clipped region of interest: an odd width, so rows are not 16-byte aligned
        _monitor("odd width", "f32", 100003, 228, 100, 3, 0.3),
        # a tile of a tiling service: int16 storage, fewer harmonics, few clouds
        _monitor("tile int16", "i16", 249776, 256, 163, 2, 0.29),
        # a tile with cloud bits from a separate mask layer, and the map of the largest |MOSUM|
        _monitor("masked tile with map", "f32", 1048576, 414, 228, 3, 0.4, mask=True, extremes=True),
        # one harmonic on a history of 254 dates
        _monitor("one harmonic int16", "i16", 500000, 522, 254, 1, 0.41),
        # a history of 347 dates (15 years of 16-day revisits)
        _monitor("long history int16", "i16", 1951528, 586, 347, 2, 0.47),
        # a full Landsat-size scene, the benchmark's workload, in both storage types
        _monitor("scene float", "f32", 8388608, 414, 228, 3, 0.6),
        _monitor("scene int16", "i16", 8388608, 414, 228, 3, 0.6),
        # the same scene gap-filled beforehand: complete series
        _monitor("scene complete", "f32", 8388608, 414, 228, 3, 0.0, complete=True),
        # many uneven tiles in one launch
        dict(name="batch of tiles", kind="batch", tiles=12, scale=0.5, tiles_seed=4),
        # the residuals and MOSUM process of pixels of interest
        dict(name="trace of pixels", kind="trace", dtype="f32", m=262144, N=414, n_hist=228, k=3, miss=0.6, h=0.25,
             count=4096),
        # the critical value of a monitoring set-up, once per configuration
        dict(name="critical value", kind="lambda", h=0.25, horizon=414 / 228, grid=1000, paths=100000),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    u = rng.random()
    if u < 0.08:
        return dict(kind="batch", tiles=rng.randint(4, 12), scale=rng.uniform(0.05, 0.5), tiles_seed=rng.randrange(1000))
    if u < 0.16:
        return dict(kind="lambda", h=rng.choice([0.25, 0.5, 1.0]), horizon=rng.uniform(1.2, 3.0),
                    grid=_log_int(rng, 200, 1000), paths=_log_int(rng, 1000, 100000))
    N = rng.randint(120, 600)
    k = rng.randint(1, 3)
    n_hist = int(N * rng.uniform(0.4, 0.7))
    miss = min(rng.uniform(0.2, 0.7), 1.0 - 4.0 * (2 + 2 * k) / n_hist)
    dtype = rng.choice(["f32", "i16"])
    m = _log_int(rng, 500, 2000000)
    if rng.random() < 0.7:
        m = -(-m // 8) * 8
    if u < 0.26:
        return dict(kind="trace", dtype=dtype, m=max(m, 4096), N=N, n_hist=n_hist, k=k, miss=miss, h=0.25,
                    count=_log_int(rng, 64, 4096))
    complete = u > 0.85
    c = _monitor("", dtype, m, N, n_hist, k, 0.0 if complete else miss, mask=not complete and rng.random() < 0.25,
                 extremes=rng.random() < 0.25, complete=complete)
    del c["name"]
    return c


def _tiles(case):
    """The tiles of a batch: pixels log-U[1e4, 2e6] (scaled), N ~ U{120..600}, k ~ U{1..3}, histories of 40-70 %,
    20-70 % missing, int16."""
    r = np.random.default_rng(case["tiles_seed"])
    out = []
    for _ in range(case["tiles"]):
        m = int(math.exp(r.uniform(math.log(1e4), math.log(2e6))) * case["scale"])
        N, k = int(r.integers(120, 601)), int(r.integers(1, 4))
        n_hist, miss = int(r.uniform(0.4, 0.7) * N), float(r.uniform(0.2, 0.7))
        miss = min(miss, 1.0 - 4.0 * (2 + 2 * k) / n_hist)
        out.append(dict(dtype="i16", m=-(-m // 8) * 8, N=N, n_hist=n_hist, k=k, miss=miss, h=0.25, mask=False,
                        extremes=False, complete=False))
    return out


def _lam(c):
    T = min(max(c["N"] / c["n_hist"], 1.2), 3.0)
    return float(np.interp(T, list(LAMBDA), list(LAMBDA.values())))


def _dates(N):
    """16-day revisits with a jitter of up to 3 days, in units of 16 days."""
    return (16.0 * np.arange(1, N + 1) + np.random.default_rng(N).integers(-3, 4, N)) / 16.0


def _design(N, k):
    t = _dates(N)
    cols = [np.ones(N), t]
    for j in range(1, k + 1):
        cols += [np.sin(2 * np.pi * j * t / F), np.cos(2 * np.pi * j * t / F)]
    return np.stack(cols, 1)


def _scene(c, seed):
    """Y [N][m] (NaN / -32768 where clouded), and the words of an explicit mask (or None)."""
    m, N, n_hist, miss = c["m"], c["N"], c["n_hist"], c["miss"]
    g = torch.Generator(device="cuda")
    g.manual_seed(seed * 7919 + N)
    rand = lambda *s: torch.rand(*s, generator=g, device="cuda")  # noqa: E731
    X = torch.tensor(_design(N, 3)[:, 2:], dtype=torch.float32, device="cuda")
    coef = rand(6, m).mul_(0.3)
    step = rand(m).mul_(0.4).add_(-0.5)
    at = (n_hist + rand(m) * (N - n_hist)).to(torch.int32)
    at[rand(m) >= 0.1] = N  # one pixel in ten breaks
    p_clear, p_cloud = 0.25, 0.25 * miss / (1.0 - miss)  # cloud runs of four dates
    cloud = rand(m) < miss
    f32 = c["dtype"] == "f32"
    Y = torch.empty((N, m), dtype=torch.float32 if f32 else torch.int16, device="cuda")
    noise, u = torch.empty(m, device="cuda"), torch.empty(m, device="cuda")
    bits = None
    if c.get("mask"):
        words = torch.randint(-2 ** 31, 2 ** 31, (2, N, (m + 31) // 32), generator=g, device="cuda", dtype=torch.int64)
        bits = (words[0] | words[1]).to(torch.int32)  # three in four dates usable
    for t in range(N):
        y = X[t] @ coef
        noise.normal_(generator=g)
        y.add_(noise, alpha=0.04).add_(0.5)
        y += step * (at <= t)
        if not f32:
            y.mul_(1e4).round_().clamp_(-32767, 32767)
        if miss > 0:
            if t:
                u.uniform_(generator=g)
                cloud = torch.where(cloud, u >= p_clear, u < p_cloud)
            y.masked_fill_(cloud, math.nan if f32 else -32768.0)
        Y[t] = y
    return Y, bits


def _args(c):
    return dict(n_hist=c["n_hist"], h_frac=c["h"], lam=_lam(c))


def prepare(case, seed):
    kind = case["kind"]
    if kind == "lambda":
        return dict(case, seed=seed)
    if kind == "batch":
        batch, keep = bfm.Batch(), []
        for i, c in enumerate(_tiles(case)):
            design, (Y, _) = bfm.Design(_dates(c["N"]), c["k"], F), _scene(c, seed + 1000 * i)
            keep.append((design, batch.add(design, Y, **_args(c))))
        return dict(kind=kind, batch=batch, keep=keep, outs=[o for _, o in keep])
    design = bfm.Design(_dates(case["N"]), case["k"], F)
    Y, bits = _scene(case, seed)
    if kind == "trace":
        status = bfm.monitor(design, Y, **_args(case))["status"]
        g = torch.Generator(device="cuda")
        g.manual_seed(seed)
        pixels = torch.randperm(case["m"], generator=g, device="cuda")[:case["count"]].contiguous()
        return dict(kind=kind, design=design, Y=Y, args=dict(n_hist=case["n_hist"], h_frac=case["h"], status=status,
                                                             pixels=pixels))
    out = bfm.empty_outputs(design.K, case["m"])
    if case["extremes"]:
        out["max_mosum"] = torch.empty(case["m"], dtype=torch.float32, device="cuda")
    args = dict(_args(case), mask_bits=bits, out=out, max_mosum=case["extremes"])
    if case["complete"]:
        args["algo"] = bfm.BFM_ALGO_COMPLETE
    return dict(kind=kind, design=design, Y=Y, args=args)


def run(state):
    kind = state["kind"]
    if kind == "lambda":
        lam, stats = bfm.bfm_lambda(0.05, state["h"], state["horizon"], state["grid"], state["paths"], state["seed"],
                                    return_stats=True)
        return dict(lam=lam, stats=stats)
    if kind == "batch":
        state["batch"].run()
        return state["outs"]
    if kind == "trace":
        return bfm.trace(state["design"], state["Y"], **state["args"])
    return bfm.monitor(state["design"], state["Y"], **state["args"])


def work(case):
    if case["kind"] == "lambda":
        steps = round(case["horizon"] * case["grid"]) * case["paths"]
        return dict(bytes=8 * case["paths"], flops=60 * steps)  # a normal (log, cos, sqrt) and a handful of operations
    if case["kind"] == "batch":
        parts = [work(dict(c, kind="monitor")) for c in _tiles(case)]
        return {key: sum(p[key] for p in parts) for key in ("bytes", "flops")}
    N, n, K, elt = case["N"], case["n_hist"], 2 + 2 * case["k"], 4 if case["dtype"] == "f32" else 2
    if case["kind"] == "trace":
        px, out = case["count"], 8 * N
    else:
        px, out = case["m"], 13 + 4 * K + (4 if case["extremes"] else 0) + (N / 8 if case["mask"] else 0)
    # history: normal equations and one residual; solve; monitoring: residual, window, test
    flops = n * (K * (K + 1) + 4 * K) + K ** 3 / 3 + 4 * K * K + (N - n) * (2 * K + 6)
    return dict(bytes=int(px * (N * elt + out)), flops=int(px * flops * (1 - case["miss"])))


def _exact_columns(c, Y, bits, lam):
    """The definition in 64 bits for the columns Y [N][c]: outputs, residuals and MOSUM process by date."""
    N, n_hist, k = c["N"], c["n_hist"], c["k"]
    K, px, dev = 2 + 2 * k, Y.shape[1], Y.device
    nan = math.nan
    valid = ~torch.isnan(Y) if Y.dtype == torch.float32 else Y != -32768
    if bits is not None:
        valid &= bits
    y = torch.where(valid, Y.double(), 0.0)
    X = _design(N, k)
    lo, hi = X[0, 1], X[-1, 1]
    mid, half = (lo + hi) / 2, (hi - lo) / 2
    X[:, 1] = (X[:, 1] - mid) / half
    X = torch.tensor(X, device=dev)
    vh, yh = valid[:n_hist].double(), y[:n_hist]
    G = ((X[:n_hist, :, None] * X[:n_hist, None, :]).reshape(n_hist, K * K).T @ vh).reshape(K, K, px)
    b = X[:n_hist].T @ yh
    n = valid[:n_hist].sum(0)
    L = torch.zeros_like(G)
    regular = torch.ones(px, dtype=torch.bool, device=dev)
    for j in range(K):
        d = G[j, j] - (L[j, :j] ** 2).sum(0)
        regular &= (d >= 1e-5 * G[j, j]) & (G[j, j] > 0)
        L[j, j] = d.clamp_min(1e-300).sqrt()
        for i in range(j + 1, K):
            L[i, j] = (G[i, j] - (L[i, :j] * L[j, :j]).sum(0)) / L[j, j]
    beta = torch.zeros_like(b)
    for i in range(K):
        beta[i] = (b[i] - (L[i, :i] * beta[:i]).sum(0)) / L[i, i]
    for i in reversed(range(K)):
        beta[i] = (beta[i] - (L[i + 1:, i] * beta[i + 1:]).sum(0)) / L[i, i]
    resid = torch.where(valid, y - X @ beta, 0.0)
    sigma = ((resid[:n_hist] ** 2).sum(0) / (n - K)).sqrt()
    fit = (n > K) & regular
    degenerate = ~(sigma > 1e-6 * yh.abs().amax(0))
    h = torch.floor(c["h"] * n.double()).long().clamp_min(1).minimum(n.clamp_min(1))
    pos = valid.cumsum(0)
    S = resid.cumsum(0)
    at = torch.zeros((N + 1, px), dtype=torch.float64, device=dev)  # S by position; missing dates repeat theirs
    at.scatter_(0, pos, S)
    W = S - at.gather(0, (pos - h).clamp_min(0))
    mon = valid & (torch.arange(N, device=dev)[:, None] >= n_hist) & fit
    mo = torch.where(mon, W / (sigma * n.double().sqrt()), nan)
    mo = torch.where(mon & degenerate, 0.0, mo)
    ratio = pos / n.clamp_min(1)
    bound2 = lam * lam * torch.where(ratio > math.e, ratio.log(), 1.0)
    cross = mon & (mo * mo > bound2)
    count = mon.sum(0)
    brk = torch.where(cross.any(0), cross.to(torch.uint8).argmax(0), -1)
    mean = torch.where(mon, mo, 0.0).sum(0) / count
    top = torch.where(mon, mo, 0.0)
    top = top.gather(0, top.abs().argmax(0)[None])[0]
    status = torch.zeros(px, dtype=torch.uint8, device=dev)
    status[count == 0] = 4
    status[degenerate] = 3
    mean = torch.where(degenerate, 0.0, mean)
    top = torch.where((count == 0) & ~degenerate, nan, top)
    status[~regular] = 2
    status[n <= K] = 1
    beta[0] -= beta[1] * mid / half
    beta[1] /= half
    un = lambda v: torch.where(fit, v, nan)  # noqa: E731
    out = dict(break_idx=torch.where(fit, brk, -1).int(), mean_mosum=un(mean), sigma=un(sigma), beta=un(beta),
               status=status)
    if c.get("extremes"):
        out["max_mosum"] = un(top)
    return out, torch.where(valid & fit, resid, nan), mo


def _exact_scene(c, Y, words):
    lam, parts = _lam(c), []
    for a in range(0, c["m"], CHUNK):
        cols = Y[:, a:a + CHUNK]
        bits = None
        if words is not None:
            w = words[:, a // 32:(a + cols.shape[1] + 31) // 32]
            shifts = torch.arange(32, device=w.device, dtype=torch.int32)
            bits = ((w[:, :, None] >> shifts) & 1).bool().reshape(c["N"], -1)[:, :cols.shape[1]]
        parts.append(_exact_columns(c, cols, bits, lam)[0])
    return {key: torch.cat([p[key] for p in parts], -1) for key in parts[0]}


def _exact_lambda(case, seed):
    """Every path's statistic in 64 bits, from the generator that the entry point documents."""
    h, G, paths = case["h"], case["grid"], case["paths"]
    steps, lag = round(case["horizon"] * G), round(h * G)
    wrap = lambda v: (v + 2 ** 63) % 2 ** 64 - 2 ** 63  # noqa: E731
    gold, m1, m2 = (wrap(v) for v in (0x9E3779B97F4A7C15, 0xBF58476D1CE4E5B9, 0x94D049BB133111EB))
    r = torch.arange(paths, device="cuda")
    state = wrap(seed * 0xA0761D6478BD642F + 1) + r * wrap(0xE7037ED1A0B428DB) + gold  # one draw discarded
    shift = lambda z, s: (z >> s) & ((1 << (64 - s)) - 1)  # noqa: E731

    def uniform():
        nonlocal state
        state = state + gold
        z = (state ^ shift(state, 30)) * m1
        z = (z ^ shift(z, 27)) * m2
        return shift(z ^ shift(z, 31), 11).double()

    W = torch.zeros((steps + 1, paths), dtype=torch.float64, device="cuda")
    for i in range(1, steps + 1):
        u1, u2 = (uniform() + 1.0) * 2.0 ** -53, uniform() * 2.0 ** -53
        torch.add(W[i - 1], (-2.0 * u1.log()).sqrt() * (2 * math.pi * u2).cos(), alpha=1.0 / math.sqrt(G), out=W[i])
    best = torch.zeros(paths, dtype=torch.float64, device="cuda")
    for i in range(G, steps + 1):
        scale = math.sqrt(math.log(i / G)) if i / G > math.e else 1.0
        best = torch.maximum(best, (W[i] - W[i - lag] - h * W[G]).abs() / scale)
    q = min(max(math.ceil(0.95 * paths) - 1, 0), paths - 1)
    return dict(lam=float(best.sort().values[q]), stats=best.cpu().numpy())


def exact(case, seed):
    kind = case["kind"]
    if kind == "lambda":
        return _exact_lambda(case, seed)
    if kind == "batch":
        return [_exact_scene(c, *_scene(c, seed + 1000 * i)) for i, c in enumerate(_tiles(case))]
    if kind == "trace":
        state = prepare(case, seed)
        cols = state["Y"][:, state["args"]["pixels"]]
        _, resid, mo = _exact_columns(case, cols, None, _lam(case))
        return dict(mo=mo.T.contiguous(), resid=resid.T.contiguous())
    return _exact_scene(case, *_scene(case, seed))
