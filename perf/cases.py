"""The workloads that this library is timed on, through its public entry points.

Each case is work that a user of the cached denoiser has it do: a control
loop's single query, a batch of queries of one policy, the candidates of a
schedule search, the activation trace and dissimilarity map that seed the
search, and the schedules drawn from the map.  Model shapes are the library's
own configurations (paper_2607_20293_gb300.synth.CONFIGS).

A program loads one policy and then serves queries with it, so the handle
(packed weights, caches, workspace) is kept from one state to the next;
observations, noise and candidate schedules are new in every state.
"""
import math

import numpy as np
import torch

from paper_2607_20293_gb300 import binding, synth

# ---------------------------------------------------------------- the cases

# kind        what it stands for
#   fp32      a small fp32 policy with a short DDIM loop
#   control   one robot's control loop: a few queries, no allocation once it runs
#   batch     a batch of queries of one policy under one schedule
#   trace     the all-refresh activations that the dissimilarity map is made from
#   search    one generation of the schedule search: few candidates, few observations
#   population  a large candidate evaluation
#   guided    dissimilarity map of a trace and the schedules drawn from it
#   map       the map alone, in its costlier metrics


def listed():
    return [
        # the smallest: fp32, 2 layers, 10 DDIM steps, 3 queries
        dict(name="fp32_b3", kind="fp32", batch=3, steps=10, frac=0.5),
        # Push-T-shaped policy, one query per control step, refresh fraction 1/8
        dict(name="control_b1", kind="control", batch=1, frac=0.125),
        # manipulation policy, 64 environments, every unit with a refresh rate of its own (0.05 .. 0.6)
        dict(name="manip_b64", kind="batch", model="manip", batch=64, hetero=4),
        # the same policy for 300 environments: 4,800 action-token rows, no multiple of a tile
        dict(name="manip_b300", kind="batch", model="manip", batch=300, frac=0.125),
        # scale-up policy (12 layers, 512 wide): a small odd batch, the benchmark's batch, full refresh
        dict(name="scale_b50", kind="batch", model="scale1024", batch=50, frac=0.25),
        dict(name="scale_b1024", kind="batch", model="scale1024", batch=1024, frac=0.125),
        dict(name="scale_b256_full", kind="batch", model="scale1024", batch=256, frac=1.0),
        # trace of 6 all-refresh queries
        dict(name="trace_b6", kind="trace", batch=6),
        # a generation of 21 new candidates of 240 cells on 4 observations
        dict(name="search_21x4", kind="search", candidates=21, obs=4, cells=240),
        # 64 candidates of 5 .. 60 % density on 16 observations
        dict(name="population_64x16", kind="population", candidates=64, obs=16),
        # cosine map of a 16-query trace and 64 schedules of 240 cells drawn from it
        dict(name="guided_n16", kind="guided", metric="cosine", steps=100, units=24, obs=16, entries=4096,
             schedules=64, cells=240),
        # Wasserstein-1 map (a sort of every activation) of a 4-query trace
        dict(name="map_w1_n4", kind="map", metric="w1", steps=100, units=24, obs=4, entries=4096),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _log(rng, lo, hi):
    return round(math.exp(rng.uniform(math.log(lo), math.log(hi))), 4)


def draw(rng):
    kind = rng.choice(["fp32", "control", "batch", "batch", "batch", "trace", "search", "population", "guided", "map"])
    if kind == "fp32":
        return dict(kind=kind, batch=_log_int(rng, 1, 40), steps=rng.choice([5, 10, 20, 25]), frac=_log(rng, 0.1, 1.0))
    if kind == "control":
        return dict(kind=kind, batch=_log_int(rng, 1, 24), frac=_log(rng, 0.05, 1.0))
    if kind == "batch":
        model = rng.choice(["pusht", "manip", "manip", "scale1024", "scale1024"])
        if model == "scale1024":
            batch = _log_int(rng, 32, 1024)
            frac = _log(rng, 0.05, min(1.0, 200.0 / batch))       # no more than the listed full refresh at 256
        else:
            batch = _log_int(rng, 2, 1024)
            if rng.random() < 0.5:
                return dict(kind=kind, model=model, batch=batch, hetero=rng.randint(5, 9999))
            frac = _log(rng, 0.05, min(1.0, 400.0 / batch))
        return dict(kind=kind, model=model, batch=batch, frac=frac)
    if kind == "trace":
        return dict(kind=kind, batch=_log_int(rng, 1, 16))
    if kind == "search":
        obs = rng.randint(1, 6)
        return dict(kind=kind, candidates=rng.randint(3, 120 // obs - 1), obs=obs, cells=rng.randint(96, 480))
    if kind == "population":
        return dict(kind=kind, candidates=rng.randint(12, 64), obs=rng.randint(11, 16))
    if kind == "guided":
        return dict(kind=kind, metric=rng.choice(["cosine", "mse", "l1"]), steps=rng.choice([10, 20, 25, 50, 100]),
                    units=3 * rng.randint(2, 12), obs=_log_int(rng, 1, 16), entries=4 * rng.randint(100, 1024),
                    schedules=_log_int(rng, 1, 64), cells=rng.randint(30, 60))
    # steps a multiple of 4: with an odd number of maps the sorted activations
    # would otherwise start off a 16-byte boundary of the scratch buffer
    return dict(kind=kind, metric=rng.choice(["w1", "w1", "l1", "mse"]), steps=rng.choice([20, 40, 60, 100]),
                units=3 * rng.randint(2, 10), obs=rng.randint(1, 4), entries=rng.choice([256, 512, 1024, 2048, 4096]))


# ---------------------------------------------------------------- policies

MAX_BATCH = {"tiny": 64, "pusht": 1040, "manip": 1024, "scale1024": 1024}
_policies = {}


def _config(case):
    kind = case["kind"]
    if kind == "fp32":
        return "tiny", synth.config("tiny", n_steps=case["steps"])
    name = case["model"] if kind == "batch" else "pusht"
    return name, synth.config(name)


def _policy(case):
    """The handle of the case's policy, made once per process."""
    name, cfg = _config(case)
    key = (name, cfg["n_steps"])
    if key not in _policies:
        weights = synth.make_weights(cfg, 0)
        _policies[key] = (cfg, weights, binding.Evo(cfg, weights, MAX_BATCH[name]))
    return _policies[key]


def _schedule(case, cfg):
    """The schedule that the policy is deployed with."""
    units, T = 3 * cfg["n_layer"], cfg["n_steps"]
    if case["kind"] == "trace":
        return np.ones((units, T), np.uint8)
    if "hetero" in case:                                    # every unit has a rate of its own
        return synth.heterogeneous_schedule(units, T, case["hetero"])
    if case["frac"] == 1.0:
        return np.ones((units, T), np.uint8)
    return synth.bernoulli_schedule(units, T, case["frac"])


def _candidates(case, cfg, seed):
    """Candidate schedules: cells drawn without replacement, likelier where a
    smooth map of the lattice is large.  A search generation holds a fixed
    number of cells of the unit lattice; the large evaluation layer lattices of
    5 .. 60 % density."""
    rng = np.random.default_rng(seed)
    T, P = cfg["n_steps"], case["candidates"]
    search = case["kind"] == "search"
    rows = 3 * cfg["n_layer"] if search else cfg["n_layer"]
    level = np.log(0.05 + synth.dissimilarity_map(rows, T, 5)).ravel() * 2.0
    S = np.zeros((P, rows * T), np.uint8)
    for p in range(P):
        k = case["cells"] if search else max(1, int(rng.uniform(0.05, 0.60) * rows * T))
        S[p, np.argsort(-(level + rng.gumbel(size=rows * T)))[:k]] = 1
    return S.reshape(P, rows, T)


def _randn(gen, *shape):
    return torch.randn(shape, generator=gen, device="cuda", dtype=torch.float32)


def _activations(case, gen):
    """[T][U][N][entries]: activations that drift along the denoising steps."""
    T, U, N, n = case["steps"], case["units"], case["obs"], case["entries"]
    base, drift = _randn(gen, U, N, n), _randn(gen, U, N, n)
    level = torch.rand((U, 1, 1), generator=gen, device="cuda") + 0.2
    x = torch.empty((T, U, N, n), device="cuda")
    for t in range(T):
        x[t] = level * (base + (t / T) * drift + 0.1 * _randn(gen, U, N, n))
    return x


# ---------------------------------------------------------------- what is timed

def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    kind = case["kind"]
    if kind in ("guided", "map"):
        s = dict(case=case, trace=_activations(case, gen))
        if kind == "guided":
            s["rnd"] = torch.randint(-(1 << 63), (1 << 63) - 1, (case["schedules"], case["cells"]), generator=gen,
                                     device="cuda", dtype=torch.int64)
        return s
    cfg, _, policy = _policy(case)
    population = kind in ("search", "population")
    n = case["obs"] if population else case["batch"]
    s = dict(case=case, policy=policy, obs=_randn(gen, n, cfg["n_obs"], cfg["obs_dim"]),
             noise=_randn(gen, synth.n_noise(cfg), n, cfg["horizon"], cfg["action_dim"]))
    if population:
        s["S"] = _candidates(case, cfg, int(seed))
    else:
        s["S"] = _schedule(case, cfg)
    if kind == "control":
        s["out"] = torch.empty((n, cfg["horizon"], cfg["action_dim"]), device="cuda")
    if kind == "trace":
        s["trace"] = torch.empty((cfg["n_steps"], 3 * cfg["n_layer"], n, cfg["horizon"], cfg["n_emb"]), device="cuda")
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "map":
        return binding.redundancy_map(s["trace"], case["metric"])
    if kind == "guided":
        d = binding.redundancy_map(s["trace"], case["metric"])
        return d, binding.guided_schedules(d, case["cells"], s["rnd"])
    if kind in ("search", "population"):
        return s["policy"].population(s["obs"], s["noise"], s["S"])
    if kind == "control":
        return s["policy"].denoise_noalloc(s["obs"], s["noise"], s["S"], s["out"])
    if kind == "trace":
        return s["policy"].denoise(s["obs"], s["noise"], s["S"], trace=s["trace"]), s["trace"]
    return s["policy"].denoise(s["obs"], s["noise"], s["S"])


# ---------------------------------------------------------------- what it cannot do without

def _cell_flops(cfg):
    """Of one refreshed cell and sample, by unit kind (causal scores counted once)."""
    E, H, C = cfg["n_emb"], cfg["horizon"], 1 + cfg["n_obs"]
    return [8 * H * E * E + 2 * H * (H + 1) * E, 4 * H * E * E + 4 * H * C * E, 16 * H * E * E]


def _fixed_flops(cfg):
    """Of one sample: observation tokens' keys and values once, input and output projection every step."""
    E, n = cfg["n_emb"], cfg["n_obs"]
    return (2 * n * cfg["obs_dim"] * E + 16 * n * E * E + cfg["n_layer"] * 4 * n * E * E
            + cfg["n_steps"] * 4 * cfg["horizon"] * cfg["action_dim"] * E)


def _cells(S, cfg):
    """Refreshed cells of lattices [..][rows][T] by unit kind."""
    per = S.reshape(-1, S.shape[-2], S.shape[-1]).sum((0, 2), dtype=np.int64)
    if S.shape[-2] == cfg["n_layer"]:
        return [int(per.sum())] * 3
    return [int(per[u::3].sum()) for u in range(3)]


def _model_bytes(cfg):
    size = 4 if cfg["dtype"] == "fp32" else 2
    return size * sum(int(np.prod(shape)) for _, shape in synth.weight_shapes(cfg))


def work(case):
    kind = case["kind"]
    if kind in ("guided", "map"):
        T, U, N, n = case["steps"], case["units"], case["obs"], case["entries"]
        pairs = U * N * T * (T + 1) // 2 if case["metric"] == "cosine" else U * N * T * (T - 1) // 2
        flops = pairs * n * (2 if case["metric"] != "mse" else 3)
        size = 4 * T * U * N * n + 4 * U * T
        if kind == "guided":
            size += case["schedules"] * (8 * case["cells"] + U * T)
        return dict(bytes=size, flops=flops)
    _, cfg = _config(case)
    chunk = 4 * cfg["horizon"] * cfg["action_dim"]
    population = kind in ("search", "population")
    if population:
        S = _candidates(case, cfg, 0)
        n, runs = case["obs"], case["obs"] * (case["candidates"] + 1)
        cells = [c + cfg["n_layer"] * cfg["n_steps"] for c in _cells(S, cfg)]     # + the all-refresh reference
        flops = n * sum(c * f for c, f in zip(cells, _cell_flops(cfg)))
        out = (case["candidates"] * n) * chunk + 4 * case["candidates"]
    else:
        S = _schedule(case, cfg)
        n = runs = case["batch"]
        flops = n * sum(c * f for c, f in zip(_cells(S, cfg), _cell_flops(cfg)))
        out = n * chunk
    size = _model_bytes(cfg) + 4 * n * cfg["n_obs"] * cfg["obs_dim"] + synth.n_noise(cfg) * n * chunk + S.size + out
    if kind == "trace":
        size += 4 * cfg["n_steps"] * 3 * cfg["n_layer"] * n * cfg["horizon"] * cfg["n_emb"]
    return dict(bytes=size, flops=flops + runs * _fixed_flops(cfg))


# About four times what the paths show against 64 bits.  fp32 loop and maps:
# 32-bit sums (the cosine map ends in 1 - cos, which cancels).  bf16 loops: the
# GEMM operands, attention probabilities and caches are rounded to 8 bits in
# every unit, and each rounding travels through the rest of the loop; the
# final actions are off by 0.0008 .. 0.0024, a unit's own output (trace) by 0.006.
def tolerance(case):
    kind = case["kind"]
    if kind == "guided":
        # whole values: a draw whose target falls between two roundings of a weight
        return dict(rel=1e-5, max=1e-4, differ=0.01)
    if kind == "map":
        return dict(rel=1e-5, max=1e-4)
    if kind == "fp32":
        return dict(rel=2e-6, max=1e-4)
    return dict(rel=2.3e-2 if kind == "trace" else 1e-2)


# ---------------------------------------------------------------- in 64 bits

def _exact_map(trace, metric):
    T, U, N, n = trace.shape
    d = torch.zeros((U, T), dtype=torch.float64, device=trace.device)
    for u in range(U):
        for r in range(N):
            x = trace[:, u, r].double()
            if metric == "cosine":
                g = x @ x.T
                norm = g.diagonal().sqrt()
                nn = norm[:, None] * norm[None, :]
                term = torch.where(nn == 0, torch.ones_like(g), 1 - g / nn)
            else:
                if metric == "w1":
                    x = x.sort(dim=1).values
                term = torch.empty((T, T), dtype=torch.float64, device=x.device)
                for t in range(T):
                    e = x[t] - x
                    term[t] = (e * e).mean(1) if metric == "mse" else e.abs().mean(1)
            term.fill_diagonal_(0)
            d[u] += term.sum(1) / (T - 1)
    return d / N


def _sampler(cfg):
    f = lambda s: math.cos((s + 0.008) / 1.008 * math.pi / 2) ** 2  # noqa: E731
    n, stride = cfg["train_steps"], cfg["train_steps"] // cfg["n_steps"]
    ab = np.cumprod([1 - min(1 - f((i + 1) / n) / f(i / n), 0.999) for i in range(n)])
    return ab, stride


def _layer_norm(x, g, b):
    m = x.mean(-1, keepdim=True)
    v = ((x - m) ** 2).mean(-1, keepdim=True)
    return (x - m) / torch.sqrt(v + 1e-5) * g + b


def _attend(q, k, v, heads, causal):
    N, H, E = q.shape
    C = k.shape[1]
    q, k, v = (z.reshape(N, -1, heads, E // heads).transpose(1, 2) for z in (q, k, v))
    s = q @ k.transpose(2, 3) / math.sqrt(E // heads)
    if causal:
        s = s.masked_fill(torch.ones((H, C), dtype=torch.bool, device=q.device).triu(1), -math.inf)
    return (s.softmax(-1) @ v).transpose(1, 2).reshape(N, H, E)


def _exact_denoise(cfg, weights, obs, noise, S, trace=None):
    """Plain 64-bit loop; S [n][3L][T]: a lattice per sample (or one for all, n = 1).  A
    unit not refreshed yet adds nothing; a skipped one adds its last output."""
    dev = obs.device
    w = {k: torch.from_numpy(v).to(dev, torch.float64) for k, v in weights.items()}
    obs, noise = obs.double(), noise.double()
    N, H, E, L, T = obs.shape[0], cfg["horizon"], cfg["n_emb"], cfg["n_layer"], cfg["n_steps"]
    heads = cfg["n_head"]
    ab, stride = _sampler(cfg)

    def memory(x):
        h = x @ w["cm_w1"] + w["cm_b1"]
        h = h * torch.tanh(torch.nn.functional.softplus(h, threshold=1e9))
        return h @ w["cm_w2"] + w["cm_b2"]

    om = memory(obs @ w["obs_w"] + w["obs_b"] + w["cond_pos"][1:])
    half = E // 2
    freq = torch.exp(-math.log(10000.0) * torch.arange(half, device=dev, dtype=torch.float64) / (half - 1))
    x = noise[0].clone()
    cache = [None] * (3 * L)
    for t in range(T):
        k = (T - 1 - t) * stride
        tm = memory(torch.cat([torch.sin(k * freq), torch.cos(k * freq)]) + w["cond_pos"][0])
        mem = torch.cat([tm.expand(N, 1, E), om], 1)
        a = x @ w["in_w"] + w["in_b"] + w["pos"]
        for b in range(3 * L):
            p, u = "l%d." % (b // 3), b % 3
            rows = S[:, b, t]
            if rows.any():
                y = _layer_norm(a, w[p + "ln%d_g" % (u + 1)], w[p + "ln%d_b" % (u + 1)])
                if u == 0:
                    q, kk, v = (y @ w[p + "sa_wqkv"] + w[p + "sa_bqkv"]).split(E, -1)
                    r = _attend(q, kk, v, heads, True) @ w[p + "sa_wo"] + w[p + "sa_bo"]
                elif u == 1:
                    kk, v = (mem @ w[p + "ca_wkv"] + w[p + "ca_bkv"]).split(E, -1)
                    r = _attend(y @ w[p + "ca_wq"] + w[p + "ca_bq"], kk, v, heads, False) @ w[p + "ca_wo"] + w[p + "ca_bo"]
                else:
                    h = y @ w[p + "ff_w1"] + w[p + "ff_b1"]
                    r = 0.5 * h * (1 + torch.erf(h / math.sqrt(2.0))) @ w[p + "ff_w2"] + w[p + "ff_b2"]
                if rows.all() or cache[b] is None:
                    cache[b] = r if rows.all() else r * torch.from_numpy(rows).to(dev).double()[:, None, None]
                else:
                    keep = torch.from_numpy(rows.astype(bool)).to(dev)[:, None, None]
                    cache[b] = torch.where(keep, r, cache[b])
            if cache[b] is not None:
                a = a + cache[b]
            if trace is not None:
                trace[t, b] = cache[b] if cache[b] is not None else 0.0
        eps = _layer_norm(a, w["lnf_g"], w["lnf_b"]) @ w["head_w"] + w["head_b"]
        prev = k - stride
        at, ap = ab[k], ab[prev] if prev >= 0 else 1.0
        x0 = ((x - math.sqrt(1 - at) * eps) / math.sqrt(at)).clamp(-1, 1)
        if cfg["sampler"] == "ddpm":
            alpha = at / ap
            x = math.sqrt(ap) * (1 - alpha) / (1 - at) * x0 + math.sqrt(alpha) * (1 - ap) / (1 - at) * x
            if k > 0:
                x = x + math.sqrt(max((1 - ap) / (1 - at) * (1 - alpha), 1e-20)) * noise[1 + t]
        else:
            x = math.sqrt(ap) * x0 + math.sqrt(1 - ap) * (x - math.sqrt(at) * x0) / math.sqrt(1 - at)
    return x


def exact(case, seed):
    s = prepare(case, seed)
    kind = case["kind"]
    if kind in ("guided", "map"):
        d = _exact_map(s["trace"], case["metric"])
        return (d, None) if kind == "guided" else d
    cfg, weights, _ = _policy(case)
    units, T = 3 * cfg["n_layer"], cfg["n_steps"]
    S = s["S"]
    population = kind in ("search", "population")
    n = case["obs"] * (case["candidates"] + 1) if population else case["batch"]
    share = 1.0 if population else S.mean()                 # lattices that differ: every unit is computed for all
    if n * T * units * share * max(_cell_flops(cfg)) > 8e12:   # FP64 on this card: about 1 TFLOP/s
        return None
    if S.shape[-2] != units:
        S = np.repeat(S, 3, axis=-2)
    if population:
        P, N = case["candidates"], case["obs"]
        S = np.repeat(np.concatenate([S, np.ones((1, units, T), np.uint8)]), N, axis=0)
        x = _exact_denoise(cfg, weights, s["obs"].repeat(P + 1, 1, 1), s["noise"].repeat(1, P + 1, 1, 1), S)
        x = x.reshape(P + 1, N, -1)
        dev = (x[:P] - x[P]).norm(dim=2).mean(1)
        return x[:P].reshape(P, N, cfg["horizon"], cfg["action_dim"]), dev
    S = S[None]
    if kind == "trace":
        tr = torch.empty(s["trace"].shape, dtype=torch.float64, device="cuda")
        return _exact_denoise(cfg, weights, s["obs"], s["noise"], S, tr), tr
    return _exact_denoise(cfg, weights, s["obs"], s["noise"], S)
