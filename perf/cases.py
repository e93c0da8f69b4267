"""The workloads that this library's speed is judged by, each through its public entry points.

A case is one call, or one short sequence of calls, that a trainer makes every
step, on inputs drawn on the GPU from a seed.  The families:

``pool``       admission of a pool of completed trajectories: pace.score_pool, then
               pace.select (occupancy budget and rejection).  From a thousand to a
               million trajectories, groups of 1 to 16, every score mode.
``step``       a whole trainer step (step.PaceStep): scoring, selection, fused
               log-probs and loss of the accepted rows.
``logprob``    pace.token_logprob on one batch, with the fused loss or without:
               masked prompts, tool segments or every row in the loss.
``prefix``     pace.prefix_score: interrupted prefixes re-scored after a weight sync.
``train``      forward and backward of one batch: pace.token_logprob with the loss
               and the log-sum-exps, pace.surrogate_backward and
               pace.token_logprob_backward; or the two backward calls alone.
``surrogate``  the clipped objective on log-probabilities that are already there
               (a later epoch over the same batch): pace.surrogate_loss and
               pace.surrogate_backward.
``controls``   the other admission rules and the diagnostics: pace.stale_k,
               pace.staleness_histogram of its result, pace.quantile_admit.

Buffers and workspaces that a trainer allocates once (step.PaceStep does) are
made in prepare().  Lengths are quantiles of the stated distribution in an order
drawn from the seed, so a case has the same number of tokens for every seed.
"""
import math

import torch

from paper_2609_36830_gb300 import pace, step

DEV = "cuda"
I32, I64, U8 = torch.int32, torch.int64, torch.uint8
F32, F64, BF16 = torch.float32, torch.float64, torch.bfloat16
EXACT_FLOPS = 8e12  # 64-bit products that take about ten seconds


# ------------------------------------------------------------------ the cases

def listed():
    return [
        # The smallest whole step: 64 short trajectories and a toy head.  Launches,
        # latency and the host's share are all there is.
        {"name": "step_tiny", "family": "step", "n": 64, "G": 8, "lens": "uniform", "lo": 16,
         "hi": 256, "turns": False, "prompt": 0, "H": 256, "V": 2048, "occupancy": 4 / 3,
         "eps_high": 0.2},
        # A multi-turn tool-use step: tool output masked out in the middle of every
        # sequence, two of eight groups rejected, the 7B-shaped head.
        {"name": "step_multiturn", "family": "step", "n": 64, "G": 8, "lens": "turns", "lo": 2,
         "hi": 8, "turns": True, "prompt": 0, "H": 3584, "V": 152064, "occupancy": 4 / 3,
         "eps_high": 0.28},
        # Admission of the pool of one ordinary step.
        {"name": "pool_1k", "family": "pool", "n": 1024, "G": 8, "median": 2048, "mode": 0,
         "gamma": 4, "window": 512, "occupancy": 2.0},
        # A larger pool in groups of twelve, the Generation-Staleness variant, an odd window.
        {"name": "pool_20k", "family": "pool", "n": 20004, "G": 12, "median": 2048, "mode": 2,
         "gamma": 2, "window": 777, "occupancy": 1.5},
        # The largest pool: a million trajectories, 3.4 G version tags.
        {"name": "pool_1m", "family": "pool", "n": 1048576, "G": 8, "median": 2048, "mode": 0,
         "gamma": 4, "window": 512, "occupancy": 2.0},
        # One micro-batch of eight sequences: log-probs and loss, prompts masked out.
        {"name": "logprob_micro", "family": "logprob", "n": 8, "G": 8, "median": 256,
         "prompt": 64, "mask": "prompt", "H": 2048, "V": 151936, "loss": True, "agg": 0,
         "temperature": 1.0},
        # Every row in the loss, a small model's head, an odd number of rows and of
        # vocabulary entries, no loss (a reference policy's log-probs).
        {"name": "logprob_dense", "family": "logprob", "n": 61, "G": 1, "median": 256,
         "prompt": 0, "mask": "none", "H": 1024, "V": 50001, "loss": False, "agg": 0,
         "temperature": 0.7},
        # Prefixes interrupted by a weight sync, re-scored under the new weights.
        {"name": "prefix_sync", "family": "prefix", "n": 24, "median": 640, "prompt": 128,
         "H": 2048, "V": 151936, "cap": 512},
        # Forward and backward of one micro-batch (gradients of hidden states and head).
        {"name": "train_micro", "family": "train", "n": 8, "G": 8, "median": 256, "prompt": 64,
         "H": 2048, "V": 151936, "forward": True, "temperature": 1.0},
        # Backward of a larger batch on the 7B-shaped head.
        {"name": "backward_batch", "family": "train", "n": 16, "G": 8, "median": 1024,
         "prompt": 256, "H": 3584, "V": 152064, "forward": False, "temperature": 1.0},
        # The objective and its derivative over a whole batch's stored log-probs.
        {"name": "surrogate_batch", "family": "surrogate", "n": 1024, "G": 8, "median": 4096,
         "prompt": 64, "agg": 0},
        # The prior-work admission rule on a 128k pool, the histogram of its lags, and
        # the sliding-window rule over the pool's groups.
        {"name": "controls_128k", "family": "controls", "n": 131072, "G": 8, "median": 2048,
         "bins": 64, "capacity": 512},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    f = rng.choice(("pool", "pool", "step", "logprob", "logprob", "prefix", "train", "train",
                    "surrogate", "controls"))
    heads = ((256, 2048), (1024, 50001), (2048, 151936), (3584, 152064))
    if f == "pool":
        G = rng.choice((1, 4, 8, 12, 16))
        return {"family": f, "n": max(1, _log_int(rng, 64, 1000000) // G) * G, "G": G,
                "median": _log_int(rng, 256, 2048), "mode": rng.choice((0, 0, 1, 2)),
                "gamma": rng.choice((1, 2, 4)), "window": _log_int(rng, 16, 4096),
                "occupancy": rng.uniform(0.9, 2.5)}
    if f == "step":
        H, V = rng.choice(heads)
        turns = rng.random() < 0.5
        G = rng.choice((4, 8))
        n = G * rng.randint(2, 56 // G)
        c = {"family": f, "n": n, "G": G, "turns": turns, "prompt": 0 if turns else rng.randint(0, 256),
             "H": H, "V": V, "occupancy": rng.uniform(1.0, 2.0), "eps_high": 0.28}
        return dict(c, lens="turns", lo=2, hi=8) if turns else dict(c, lens="uniform", lo=16,
                                                                    hi=_log_int(rng, 128, 4096))
    if f == "logprob":
        mask = rng.choice(("none", "prompt", "turns"))
        G = rng.choice((1, 4, 8))
        H, V = rng.choice(heads) if rng.random() < 0.6 else (64 * rng.randint(4, 64),
                                                             _log_int(rng, 2000, 160000))
        n = G * rng.randint(1, 32 // G)
        median = _log_int(rng, 16, 1200)
        return {"family": f, "n": n, "G": G, "median": median,
                "prompt": rng.randint(1, 300) if mask == "prompt" else 0, "mask": mask, "H": H,
                "V": V, "loss": rng.random() < 0.6, "agg": rng.choice((0, 0, 1)),
                "temperature": rng.choice((1.0, 1.0, 0.7))}
    if f == "prefix":
        H, V = rng.choice(heads)
        return {"family": f, "n": rng.randint(2, 48), "median": _log_int(rng, 48, 1400),
                "prompt": rng.randint(0, 256), "H": H, "V": V, "cap": rng.choice((512, 1024, 2048))}
    if f == "train":
        H, V = rng.choice(heads) if rng.random() < 0.6 else (64 * rng.randint(4, 64),
                                                             _log_int(rng, 2000, 160000))
        return {"family": f, "n": 8 * rng.randint(1, 2), "G": rng.choice((4, 8)),
                "median": _log_int(rng, 32, 900), "prompt": rng.randint(0, 256), "H": H, "V": V,
                "forward": rng.random() < 0.5, "temperature": rng.choice((1.0, 1.0, 0.7))}
    if f == "surrogate":
        G = rng.choice((4, 8, 16))
        return {"family": f, "n": G * max(1, _log_int(rng, 8, 1024) // G), "G": G,
                "median": _log_int(rng, 64, 4096), "prompt": rng.randint(0, 256),
                "agg": rng.choice((0, 1))}
    G = rng.choice((1, 8, 12))
    return {"family": f, "n": G * max(1, _log_int(rng, 512, 130000) // G), "G": G,
            "median": _log_int(rng, 256, 2048), "bins": _log_int(rng, 10, 1000),
            "capacity": rng.choice((64, 512, 4096))}


# ------------------------------------------------------------------ the inputs

def _gens(seed):
    g, h = torch.Generator(device=DEV), torch.Generator()
    g.manual_seed(int(seed))
    h.manual_seed(int(seed))
    return g, h


def _quantiles(n, lens, lo, hi, median=None, sigma=None):
    """n lengths at the quantiles (i + 1/2) / n of the distribution, ascending."""
    u = (torch.arange(n, dtype=F64) + 0.5) / n
    if lens == "uniform":
        return (lo + torch.floor(u * (hi - lo + 1))).to(I64)
    x = median * torch.exp(sigma * torch.special.ndtri(u))
    return torch.clamp(torch.round(x), lo, hi).to(I64)


def _pool_lens(case):
    return _quantiles(case["n"], "lognormal", 16, 32768, case["median"], 1.0)


def _batch_lens(case):
    if case["family"] == "step":
        return _quantiles(case["n"], "uniform", case["lo"], case["hi"])
    return _quantiles(case["n"], "lognormal", 16, 16384, case["median"], 0.75)


def _shuffled(x, h):
    return x[torch.randperm(x.numel(), generator=h)]


def _offsets(lens):
    return torch.cat([torch.zeros(1, dtype=I64), torch.cumsum(lens, 0)])


def _randint(g, lo, hi):
    """Per entry uniform in [lo, hi] (tensors)."""
    r = torch.rand(lo.shape, generator=g, device=DEV, dtype=F64)
    return lo + (r * (hi - lo + 1)).to(I64).minimum(hi - lo)


def _segments_of(lens, n_int, m, g):
    """Segment lengths [n, m + 1]: n_int <= m cuts at uniform places of each sequence."""
    pos = 1 + (torch.rand((lens.numel(), m), generator=g, device=DEV, dtype=F64)
               * (lens[:, None] - 1)).to(I64)
    pos = torch.where(torch.arange(m, device=DEV)[None, :] < n_int[:, None], pos, lens[:, None])
    pos = torch.sort(pos, dim=1).values
    zero = torch.zeros((lens.numel(), 1), dtype=I64, device=DEV)
    return torch.diff(torch.cat([zero, pos, lens[:, None]], dim=1), dim=1)


def _expand(values, seg, total):
    """Every segment's value, repeated over its length: int32 [total], a part at a time."""
    out = torch.empty(total, dtype=I32, device=DEV)
    at = 0
    for i in range(0, seg.shape[0], 65536):
        s = seg[i:i + 65536].reshape(-1)
        k = int(s.sum())
        out[at:at + k] = torch.repeat_interleave(values[i:i + 65536].reshape(-1).to(I32), s,
                                                 output_size=k)
        at += k
    return out


def _pool(case, g, h, lens, j=1000, max_int=8, max_lag=32):
    """Version tags and per-trajectory inputs: interruptions bump the tag by one."""
    n = lens.numel()
    lens = lens.to(DEV)
    n_int = torch.randint(0, max_int + 1, (n,), generator=g, device=DEV)
    start = j - _randint(g, n_int, torch.full_like(n_int, max_lag))
    c = _randint(g, start + n_int, torch.full_like(start, j))
    values = start[:, None] + torch.arange(max_int + 1, device=DEV)[None, :]
    seg = _segments_of(lens, n_int, max_int, g)
    drift = torch.randn(n, generator=g, device=DEV) * (0.05 * n_int)
    s_pre = torch.where(n_int > 0, drift.abs(), torch.full_like(drift, float("nan")))
    w = case.get("window", 512)
    window = (torch.randn(w, generator=g, device=DEV)
              * (0.05 * torch.randint(1, max_int + 1, (w,), generator=g, device=DEV))).abs()
    return {"tags": _expand(values, seg, int(lens.sum())), "offsets": _offsets(lens.cpu()).to(DEV),
            "c": c.to(I32), "s_pre": s_pre.to(F32), "window": window.to(F32), "j": j}


def _turn_segments(n, lo, hi):
    """Lengths of n multi-turn sequences' tool and model segments, both [n, hi] (0: unused)."""
    h = torch.Generator()
    h.manual_seed(n)
    turns = _shuffled(_quantiles(n, "uniform", lo, hi), h)
    model = _shuffled(_quantiles(n * hi, "uniform", 64, 1024), h).reshape(n, hi)
    tool = _shuffled(_quantiles(n * hi, "uniform", 32, 512), h).reshape(n, hi)
    at = torch.arange(hi)[None, :]
    used = at < turns[:, None]
    return turns, torch.where(used & (at > 0), tool, 0 * tool), torch.where(used, model, 0 * model)


def _turns(n, g, h, lo=2, hi=8, max_lag=10, j=200):
    """Multi-turn sequences: model segments with tool segments between them."""
    perm = torch.randperm(n, generator=h)
    turns, tool, model = (x[perm].to(DEV) for x in _turn_segments(n, lo, hi))
    seg = torch.stack([tool, model], dim=2).reshape(n, 2 * hi)
    lag = torch.randint(0, max_lag + 1, (n, hi), generator=g, device=DEV)
    lag = torch.sort(lag, dim=1, descending=True).values
    val = torch.stack([torch.full_like(lag, -1), j - lag], dim=2).reshape(n, 2 * hi)
    lens = seg.sum(1)
    last = torch.gather(lag, 1, (turns - 1)[:, None])[:, 0]
    c = _randint(g, j - last, torch.full_like(last, j))
    n_int = turns - 1
    s_pre = (torch.randn(n, generator=g, device=DEV) * (0.05 * n_int)).abs()
    window = (torch.randn(512, generator=g, device=DEV) * 0.2).abs()
    return {"tags": _expand(val, seg, int(lens.sum())), "offsets": _offsets(lens.cpu()).to(DEV),
            "c": c.to(I32), "s_pre": s_pre.to(F32), "window": window.to(F32), "j": j}


def _with_prompts(tags, offsets, prompt):
    """Row offsets and each row's tag (-1 on prompt and tool rows)."""
    n = offsets.numel() - 1
    if not prompt:
        return offsets, tags
    lens = torch.diff(offsets)
    seg = torch.stack([torch.full_like(lens, prompt), lens], dim=1).reshape(-1)
    kind = torch.tensor([0, 1], dtype=U8, device=DEV).repeat(n)
    is_resp = torch.repeat_interleave(kind, seg, output_size=int(seg.sum())).bool()
    version = torch.full((is_resp.numel(),), -1, dtype=I32, device=DEV)
    version[is_resp] = tags
    return offsets + prompt * torch.arange(n + 1, device=DEV), version


def _rows(case, g, h, p, reward_p=0.5):
    """The token batch of a pool: hidden states, head, targets, behaviour log-probs, rewards."""
    H, V = case["H"], case["V"]
    row_offsets, version = _with_prompts(p["tags"], p["offsets"], case.get("prompt", 0))
    n_rows, n = version.numel(), row_offsets.numel() - 1
    mask = (version >= 0).to(U8)
    lag = torch.where(version >= 0, p["j"] - version, 0 * version)
    behav = (-math.log(V) - 0.5) + torch.randn(n_rows, generator=g, device=DEV) * (0.05 * lag)
    hidden = torch.randn((n_rows, H), generator=g, device=DEV, dtype=BF16)
    w = torch.randn((V, H), generator=g, device=DEV, dtype=BF16).mul_(1.0 / math.sqrt(H))
    return {"row_offsets": row_offsets, "mask": mask, "hidden": hidden, "w": w,
            "targets": torch.randint(0, V, (n_rows,), generator=g, device=DEV, dtype=I32),
            "behav": behav.to(F32),
            "reward": (torch.rand(n, generator=g, device=DEV) < reward_p).to(F32)}


def _batch(case, g, h):
    """One batch of sequences: tags with a lag of up to eight versions, rows as masked."""
    if case.get("mask") == "turns":
        p = _turns(case["n"], g, h, 2, 4)
    else:
        p = _pool(case, g, h, _shuffled(_batch_lens(case), h), j=200, max_int=3, max_lag=8)
    return p, _rows(case, g, h, p)


def _n_target(case):
    return int(case["n"] / case["occupancy"])


def prepare(case, seed):
    g, h = _gens(seed)
    f = case["family"]
    s = {"case": case, "status": pace.new_status(DEV)}
    L = pace.lib()
    if f in ("pool", "controls"):
        p = _pool(case, g, h, _shuffled(_pool_lens(case), h))
        n, G = case["n"], case["G"]
        u = n // G
        s.update(p)
    if f == "pool":
        s["params"] = pace.score_params(mode=case["mode"], gamma=case["gamma"], group_size=G)
        s["budget"] = pace.budget_params(_n_target(case))
        s["out"] = {k: torch.empty(n, dtype=F64, device=DEV)
                    for k in ("kgen", "kwait", "weight", "score")}
        s["out"]["unit_score"] = torch.empty(u, dtype=F64, device=DEV)
        s["sel"] = {"accepted": torch.empty(n, dtype=I32, device=DEV),
                    "rejected": torch.empty(n, dtype=I32, device=DEV),
                    "flags": torch.empty(n, dtype=U8, device=DEV)}
        s["ws"] = pace.workspace(L.pace_score_pool_workspace_size(n, case["window"]), DEV)
        s["ws_sel"] = pace.workspace(L.pace_select_workspace_size(u), DEV)
    elif f == "controls":
        s["kbar"] = torch.empty(n, dtype=F64, device=DEV)
        s["admitted"] = torch.empty(n, dtype=U8, device=DEV)
        s["hist"] = torch.empty(2 * case["bins"], dtype=I32, device=DEV)
        s["ws"] = pace.workspace(L.pace_stale_k_workspace_size(n), DEV)
        s["unit_score"] = torch.rand(u, generator=g, device=DEV, dtype=F64) * 20
        s["ring"] = pace.ScoreWindow(case["capacity"], DEV)
        s["ring"].values.copy_(torch.rand(case["capacity"], generator=g, device=DEV, dtype=F64) * 20)
        s["ring"].state.copy_(torch.tensor([case["capacity"], case["capacity"] // 3]))
        s["decision"] = torch.empty(u, dtype=U8, device=DEV)
        s["kappa"] = torch.empty(1, dtype=F64, device=DEV)
    elif f == "step":
        p = (_turns(case["n"], g, h, case["lo"], case["hi"]) if case["turns"] else
             _pool(case, g, h, _shuffled(_batch_lens(case), h), j=200, max_int=3, max_lag=8))
        r = _rows(case, g, h, p)
        s.update(p, **r)
        x = step.StepInputs(
            tags=p["tags"], offsets=p["offsets"], c_version=p["c"], s_pre=p["s_pre"],
            window=p["window"], row_offsets=r["row_offsets"], mask=r["mask"],
            targets=r["targets"], behav_lp=r["behav"], reward=r["reward"], hidden=r["hidden"],
            w_vocab=r["w"], trainer_version=p["j"], n_target=_n_target(case),
            group_size=case["G"])
        s["step"] = step.PaceStep(x, loss_params=pace.loss_params(eps_high=case["eps_high"]))
    elif f == "surrogate":
        p = _pool(case, g, h, _shuffled(_batch_lens(case), h), j=200, max_int=3, max_lag=8)
        row_offsets, version = _with_prompts(p["tags"], p["offsets"], case["prompt"])
        n_rows, n, G = version.numel(), case["n"], case["G"]
        lp = -4.0 * torch.rand(n_rows, generator=g, device=DEV)
        lag = torch.where(version >= 0, p["j"] - version, 0 * version)
        d = torch.randn(n_rows, generator=g, device=DEV) * (0.05 * lag)
        # a ratio within rounding of a clip edge has two right derivatives: none is that close
        rho = torch.exp(d)
        near = ((rho - 0.8).abs() < 1e-4) | ((rho - 1.28).abs() < 1e-4) | ((rho - 10).abs() < 1e-3)
        s["lp"] = lp
        s["behav"] = lp - torch.where(near, 0 * d, d)
        s["mask"] = (version >= 0).to(U8)
        s["row_offsets"] = row_offsets
        s["accepted"] = (torch.rand(n // G, generator=g, device=DEV) < 0.75).to(U8) \
            .repeat_interleave(G)
        s["reward"] = (torch.rand(n, generator=g, device=DEV) < 0.5).to(F32)
        s["dlp"] = torch.empty(n_rows, dtype=F32, device=DEV)
        s["batch"] = pace.make_batch(row_offsets, n_rows, seq_accepted=s["accepted"],
                                     mask=s["mask"])
        s["ratio"] = torch.empty(n_rows, dtype=F32, device=DEV)
        s["ws"] = pace.workspace(L.pace_surrogate_loss_workspace_size(n_rows, n), DEV)
        s["ws_b"] = pace.workspace(L.pace_surrogate_backward_workspace_size(n_rows, n), DEV)
        _loss_args(s, case, n, ratio=s["ratio"])
    elif f == "logprob":
        p, r = _batch(case, g, h)
        s.update(p, **r)
        _head_buffers(s, case, mask=None if case["mask"] == "none" else r["mask"])
    elif f == "prefix":
        p, r = _batch(case, g, h)
        s.update(p, **r)
        s["batch"] = pace.make_batch(r["row_offsets"], r["mask"].numel(), mask=r["mask"])
        s["s_out"] = torch.empty(case["n"], dtype=F32, device=DEV)
        s["lp"] = torch.empty(r["mask"].numel(), dtype=F32, device=DEV)
        s["ws"] = pace.workspace(L.pace_prefix_score_workspace_size(
            r["mask"].numel(), case["n"], case["H"], case["V"]), DEV)
    else:
        p, r = _batch(case, g, h)
        s.update(p, **r)
        _head_buffers(s, case, mask=r["mask"])
        n_rows, n = r["mask"].numel(), case["n"]
        s["dlp"] = torch.empty(n_rows, dtype=F32, device=DEV)
        s["gh"] = torch.empty((n_rows, case["H"]), dtype=F32, device=DEV)
        s["gw"] = torch.empty((case["V"], case["H"]), dtype=F32, device=DEV)
        s["ws_d"] = pace.workspace(L.pace_surrogate_backward_workspace_size(n_rows, n), DEV)
        s["ws_b"] = pace.workspace(L.pace_token_logprob_backward_workspace_size(
            n_rows, n, case["H"], case["V"]), DEV)
        if not case["forward"]:
            _forward(s)
    return s


def _loss_args(s, case, n, ratio=None):
    s["loss"] = torch.zeros(1, dtype=F64, device=DEV)
    s["adv"] = torch.empty(n, dtype=F32, device=DEV)
    s["loss_args"] = pace.make_loss_args(s["behav"], s["reward"], case["G"],
                                         pace.loss_params(agg=case.get("agg", 0)), s["loss"],
                                         adv_out=s["adv"], ratio_out=ratio)


def _head_buffers(s, case, mask):
    n_rows = s["mask"].numel()
    s["lp"] = torch.empty(n_rows, dtype=F32, device=DEV)
    s["lse"] = torch.empty(n_rows, dtype=F32, device=DEV)
    s["batch"] = pace.make_batch(s["row_offsets"], n_rows, mask=mask)
    s["ws"] = pace.workspace(pace.token_logprob_workspace_size(n_rows, case["n"], case["H"],
                                                               case["V"]), DEV)
    _loss_args(s, case, case["n"])


def _forward(s):
    c = s["case"]
    pace.token_logprob(s["batch"], s["hidden"], s["w"], s["targets"], c["temperature"],
                       loss=s["loss_args"] if c.get("loss", True) else None, logprob=s["lp"],
                       lse=s["lse"], ws=s["ws"], status=s["status"])


# ------------------------------------------------------------------ one pass

def run(s):
    c = s["case"]
    f = c["family"]
    if f == "pool":
        pace.score_pool(s["tags"], s["offsets"], s["c"], s["s_pre"], s["j"], s["window"],
                        s["params"], out=s["out"], ws=s["ws"], status=s["status"])
        r_hat, k, acc, rej, flags = pace.select(s["out"]["unit_score"], c["G"], s["budget"],
                                                out=s["sel"], ws=s["ws_sel"], status=s["status"])
        return dict(s["out"], r_hat=r_hat, k=k, accepted=acc, rejected=rej, flags=flags,
                    status=s["status"])
    if f == "controls":
        kbar, adm = pace.stale_k(s["tags"], s["offsets"], s["j"], 16.0, kbar=s["kbar"],
                                 admitted=s["admitted"], ws=s["ws"], status=s["status"])
        hist = pace.staleness_histogram(kbar, adm, 0.0, 32.0, c["bins"], hist=s["hist"],
                                        status=s["status"])
        dec, kappa = pace.quantile_admit(s["unit_score"], 1.0 / 3.0, _batch_units(c), s["ring"],
                                         decision=s["decision"], kappa=s["kappa"],
                                         status=s["status"])
        return {"kbar": kbar, "admitted": adm, "hist": hist, "decision": dec, "kappa": kappa,
                "ring": s["ring"].values, "ring_state": s["ring"].state, "status": s["status"]}
    if f == "step":
        st = s["step"]
        k, r_hat = st.run()
        return dict(st.score_out, k=k, r_hat=r_hat, flags=st.sel_out["flags"],
                    accepted=st.sel_out["accepted"][:(st.U - k) * st.G],
                    rejected=st.sel_out["rejected"][:k * st.G], logprob=st.logprob, loss=st.loss,
                    adv=st.adv, status=st.status)
    if f == "surrogate":
        pace.surrogate_loss(s["batch"], s["lp"], s["loss_args"], ws=s["ws"], status=s["status"])
        pace.surrogate_backward(s["batch"], s["lp"], s["loss_args"], dlp=s["dlp"], ws=s["ws_b"],
                                status=s["status"])
        return {"loss": s["loss"], "adv": s["adv"], "ratio": s["ratio"], "dlp": s["dlp"],
                "status": s["status"]}
    if f == "logprob":
        _forward(s)
        out = {"lp": s["lp"], "lse": s["lse"], "status": s["status"]}
        return dict(out, loss=s["loss"], adv=s["adv"]) if c["loss"] else out
    if f == "prefix":
        pace.prefix_score(s["batch"], s["hidden"], s["w"], s["targets"], s["behav"],
                          cap_tokens=c["cap"], s_pre=s["s_out"], logprob=s["lp"], ws=s["ws"],
                          status=s["status"])
        return {"s_pre": s["s_out"], "lp": s["lp"], "status": s["status"]}
    out = {}
    if c["forward"]:
        _forward(s)
        out = {"lp": s["lp"], "lse": s["lse"], "loss": s["loss"]}
    pace.surrogate_backward(s["batch"], s["lp"], s["loss_args"], dlp=s["dlp"], ws=s["ws_d"],
                            status=s["status"])
    pace.token_logprob_backward(s["batch"], s["hidden"], s["w"], s["targets"], s["lse"], s["dlp"],
                                c["temperature"], grad_hidden=s["gh"], grad_w=s["gw"],
                                ws=s["ws_b"], status=s["status"])
    return dict(out, dlp=s["dlp"], gh=s["gh"], gw=s["gw"], status=s["status"])


def _batch_units(c):
    return c["n"] // c["G"] // 2


# ------------------------------------------------------------------ work and tolerance

def _row_counts(case):
    """(rows, rows in the loss) of a batch case; with rejected groups, the mean over seeds."""
    n, prompt = case["n"], case.get("prompt", 0)
    if case.get("turns") or case.get("mask") == "turns":
        lo, hi = (case["lo"], case["hi"]) if case.get("turns") else (2, 4)
        _, tool, model = _turn_segments(n, lo, hi)
        rows, in_loss = float(tool.sum() + model.sum()), float(model.sum())
    else:
        in_loss = float(_batch_lens(case).sum())
        rows = in_loss + n * prompt
        if case["family"] == "prefix":
            in_loss = float(_batch_lens(case).clamp(max=case["cap"]).sum())
    if case["family"] == "step":
        in_loss *= 1.0 - _k_units(case) / (n // case["G"])
    if case["family"] == "surrogate":
        in_loss *= 0.75
    return rows, in_loss


def _k_units(case):
    n, u = case["n"], case["n"] // case["G"]
    r = min(max((n - _n_target(case)) / n, 0.0), 1.0)
    return min(int(math.floor(min(r, 0.9) * u + 1e-9)), u)


def work(case):
    f, n = case["family"], case["n"]
    pool = 4 * case.get("window", 512) + n * (8 + 4 + 4 + 32 + 8 / case.get("G", 1) + 5)
    if f == "pool":
        return {"bytes": 4 * float(_pool_lens(case).sum()) + pool, "flops": 0.0}
    if f == "controls":
        # tags, offsets, kbar and its flags out; then the unit scores and decisions
        return {"bytes": 4 * float(_pool_lens(case).sum()) + n * (8 + 8 + 1)
                + 9 * n / case["G"] + 8 * case["bins"] + 16 * case["capacity"], "flops": 0.0}
    rows, in_loss = _row_counts(case)
    if f == "surrogate":
        # the loss: log-probs, behaviour log-probs and mask in, ratios out; then the
        # derivative: the same in, dlp out (two calls, each of them complete)
        return {"bytes": 2 * (rows * (1 + 4) + in_loss * 8) + n * 13, "flops": 0.0}
    H, V = case["H"], case["V"]
    head = 2.0 * H * V * in_loss
    b = in_loss * (2 * H + 4) + 2.0 * H * V + rows * (1 + 4 + 4)
    if f == "step":
        return {"bytes": b + 4 * rows + pool, "flops": head}
    if f == "train":
        passes = 3 + (1 if case["forward"] else 0)
        return {"bytes": b + rows * (4.0 * H + 12) + 4.0 * H * V, "flops": passes * head}
    return {"bytes": b, "flops": head}


def tolerance(case):
    f = case["family"]
    if f in ("pool", "controls"):
        return "exact"  # scores, lags and decisions are defined to the bit
    if f == "train":
        return {"rel": 1e-2, "max": 0.5}  # the logits' gradient is held in bf16 (1.7e-3 measured)
    if f == "surrogate":
        return {"rel": 1e-6, "max": 1e-4}  # 32-bit terms, 64-bit sums (1.3e-7 measured)
    # 32-bit sums over the hidden size and the vocabulary (2.5e-7 measured on the
    # log-probs, 1.7e-6 on a prefix's mean difference of two of them); a batch's loss
    # is the small remainder of advantages that cancel, ten times further off
    return {"rel": 3e-5, "max": 1e-3}


# ------------------------------------------------------------------ 64 bits

def _f64(x):
    """A one-element tensor: torch divides by it, where by a number it multiplies by the inverse."""
    return torch.tensor([float(x)], dtype=F64, device=DEV)


def _exact_pool(p, case, mode, gamma, G, n_target):
    o = p["offsets"]
    n = o.numel() - 1
    S, T = _segment_sums(p["tags"], o)
    c, j = p["c"].to(I64), p["j"]
    kgen = torch.where(T > 0, (c * T - S).to(F64) / T.clamp(min=1).to(F64), torch.zeros_like(T, dtype=F64))
    kwait = (j - c).to(F64)
    w = p["window"].numel()
    weight = torch.ones(n, dtype=F64, device=DEV)
    if w >= 32:
        ws = torch.sort(p["window"]).values
        q = torch.searchsorted(ws, p["s_pre"].nan_to_num(0.0), right=True).to(F64) / _f64(w)
        a, b = q.clone(), 1.0 - q
        b0 = b.clone()
        for _ in range(gamma - 1):
            a, b = a * q, b * b0
        weight = torch.where(torch.isnan(p["s_pre"]), weight, a / (a + b))
    score = (kwait + weight * kgen, kwait + kgen, weight * kgen)[mode]
    acc = torch.zeros(n // G, dtype=F64, device=DEV)
    for i in range(G):
        acc = acc + score.reshape(-1, G)[:, i]
    unit = acc / _f64(G)
    u = n // G
    r = min(max((n - n_target) / n, 0.0), 1.0)
    k = min(int(math.floor(min(r, 0.9) * u + 1e-9)), u)
    order = torch.sort(unit, descending=True, stable=True).indices
    flag = torch.ones(u, dtype=U8, device=DEV)
    flag[order[:k]] = 0
    flags = flag.repeat_interleave(G)
    ids = torch.arange(n, device=DEV, dtype=I32)
    return {"kgen": kgen, "kwait": kwait, "weight": weight, "score": score, "unit_score": unit,
            "k": k, "r_hat": r, "flags": flags, "accepted": ids[flags == 1],
            "rejected": ids[flags == 0]}


def _segment_sums(tags, o):
    """Exact sums and counts of the policy tags of every trajectory."""
    n = o.numel() - 1
    S, T = torch.empty(n, dtype=I64, device=DEV), torch.empty(n, dtype=I64, device=DEV)
    for i in range(0, n, 65536):
        e = min(n, i + 65536)
        a = int(o[i])
        t = tags[a:int(o[e])].to(I64)
        for out, x in ((S, t.clamp(min=0)), (T, (t >= 0).to(I64))):
            cs = torch.cat([torch.zeros(1, dtype=I64, device=DEV), torch.cumsum(x, 0)])
            out[i:e] = cs[o[i + 1:e + 1] - a] - cs[o[i:e] - a]
    return S, T


def _exact_logprob(hidden, w, targets, temperature, in_loss):
    """(lp, lse) in 64 bits of the rows in the loss, 0 elsewhere."""
    n = hidden.shape[0]
    lp, lse = torch.zeros(n, dtype=F64, device=DEV), torch.zeros(n, dtype=F64, device=DEV)
    rows = torch.nonzero(in_loss)[:, 0]
    wd = w.to(F64).T
    for i in range(0, rows.numel(), 2048):
        r = rows[i:i + 2048]
        z = (hidden[r].to(F64) @ wd) / temperature
        lse[r] = torch.logsumexp(z, 1)
        lp[r] = torch.gather(z, 1, targets[r].to(I64)[:, None])[:, 0] - lse[r]
    return lp, lse


def _exact_adv(reward, G, accepted):
    r = reward.to(F64).reshape(-1, G)
    a = accepted.to(F64).reshape(-1, G)
    cnt = a.sum(1, keepdim=True)
    mean = (r * a).sum(1, keepdim=True) / cnt.clamp(min=1)
    ss = (((r - mean) * a) ** 2).sum(1, keepdim=True)
    sd = torch.where(cnt > 1, torch.sqrt(ss / (cnt - 1).clamp(min=1)), torch.zeros_like(ss))
    eps = float(torch.tensor(1e-6, dtype=F32))
    return (((r - mean) / (sd + eps)) * a).reshape(-1)


def _exact_surrogate(lp, behav, row_offsets, in_loss, adv, agg, eps_high=0.28):
    """(loss, ratio, dlp) in 64 bits."""
    n = row_offsets.numel() - 1
    seq = torch.repeat_interleave(torch.arange(n, device=DEV), torch.diff(row_offsets),
                                  output_size=lp.numel())
    a = adv[seq]
    d = (lp.to(F64) - behav.to(F64)).clamp(-20, 20)
    rho = torch.exp(d)
    p1, p2 = -a * rho, -a * rho.clamp(1 - 0.2, 1 + eps_high)
    low = torch.maximum(p1, p2)
    dual = (a < 0) & (-10.0 * a < low)
    term = torch.where(dual, -10.0 * a, low)
    m = in_loss.to(F64)
    ratio = torch.where(in_loss, rho, torch.zeros_like(rho))
    g = torch.where((p1 >= p2) & ~dual & in_loss, -a * rho, torch.zeros_like(rho))
    cnt = torch.zeros(n, dtype=F64, device=DEV).index_add_(0, seq, m)
    tot = torch.zeros(n, dtype=F64, device=DEV).index_add_(0, seq, torch.where(in_loss, term, 0 * term))
    if agg == 0:
        total = cnt.sum().clamp(min=1)
        return (tot.sum() / total).reshape(1), ratio, g / total
    used = (cnt > 0).sum().clamp(min=1).to(F64)
    loss = (tot / cnt.clamp(min=1)).sum() / used
    return loss.reshape(1), ratio, g / (used * cnt.clamp(min=1)[seq])


def _exact_grads(s, dlp, lse, temperature):
    h, w, y = s["hidden"], s["w"], s["targets"].to(I64)
    gh = torch.zeros(h.shape, dtype=F64, device=DEV)
    gw = torch.zeros(w.shape, dtype=F64, device=DEV)
    wd = w.to(F64)
    rows = torch.nonzero(s["mask"])[:, 0]
    for i in range(0, rows.numel(), 2048):
        r = rows[i:i + 2048]
        hd = h[r].to(F64)
        G = -torch.exp((hd @ wd.T) / temperature - lse[r][:, None])
        G[torch.arange(r.numel(), device=DEV), y[r]] += 1.0
        G *= (dlp[r] / temperature)[:, None]
        gh[r] = G @ wd
        gw += G.T @ hd
    return gh, gw


def exact(case, seed):
    f = case["family"]
    if f in ("logprob", "prefix", "train") and work(case)["flops"] > EXACT_FLOPS:
        return None
    s = prepare(case, seed)
    status = torch.zeros(1, dtype=I32, device=DEV)
    if f == "pool":
        return dict(_exact_pool(s, case, case["mode"], case["gamma"], case["G"], _n_target(case)),
                    status=status)
    if f == "controls":
        return dict(_exact_controls(s, case), status=status)
    if f == "step":
        out = _exact_pool(s, case, 0, 4, case["G"], _n_target(case))
        adv = _exact_adv(s["reward"], case["G"], out["flags"])
        lp = loss = None
        if work(case)["flops"] <= EXACT_FLOPS:
            in_loss = (s["mask"] == 1) & (torch.repeat_interleave(
                out["flags"], torch.diff(s["row_offsets"])) == 1)
            lp, _ = _exact_logprob(s["hidden"], s["w"], s["targets"], 1.0, in_loss)
            loss, _, _ = _exact_surrogate(lp, s["behav"], s["row_offsets"], in_loss, adv, 0,
                                          case["eps_high"])
        return dict(out, logprob=lp, loss=loss, adv=adv, status=status)
    if f == "surrogate":
        in_loss = (s["mask"] == 1) & (torch.repeat_interleave(
            s["accepted"], torch.diff(s["row_offsets"])) == 1)
        adv = _exact_adv(s["reward"], case["G"], s["accepted"])
        loss, ratio, dlp = _exact_surrogate(s["lp"], s["behav"], s["row_offsets"], in_loss, adv,
                                            case["agg"])
        return {"loss": loss, "adv": adv, "ratio": ratio, "dlp": dlp, "status": status}
    ones = torch.ones(case["n"], dtype=U8, device=DEV)
    in_loss = s["mask"] == 1
    if f == "logprob":
        if case["mask"] == "none":
            in_loss = torch.ones_like(in_loss)
        lp, lse = _exact_logprob(s["hidden"], s["w"], s["targets"], case["temperature"], in_loss)
        out = {"lp": lp, "lse": lse, "status": status}
        if case["loss"]:
            adv = _exact_adv(s["reward"], case["G"], ones)
            loss, _, _ = _exact_surrogate(lp, s["behav"], s["row_offsets"], in_loss, adv,
                                          case["agg"])
            out.update(loss=loss, adv=adv)
        return out
    if f == "prefix":
        o = s["row_offsets"]
        seq = torch.repeat_interleave(torch.arange(case["n"], device=DEV), torch.diff(o))
        before = torch.cumsum(in_loss.to(I64), 0) - in_loss.to(I64)
        use = in_loss & (before - before[o[:-1].clamp(max=before.numel() - 1)][seq] < case["cap"])
        lp, _ = _exact_logprob(s["hidden"], s["w"], s["targets"], 1.0, use)
        d = torch.where(use, (lp - s["behav"].to(F64)).abs(), torch.zeros_like(lp))
        zero = torch.zeros(case["n"], dtype=F64, device=DEV)
        elig = zero.clone().index_add_(0, seq, in_loss.to(F64))
        mean = zero.clone().index_add_(0, seq, d) / elig.clamp(1, case["cap"])
        return {"s_pre": torch.where(elig >= 32, mean, torch.full_like(mean, float("nan"))),
                "lp": lp, "status": status}
    adv = _exact_adv(s["reward"], case["G"], ones)
    if case["forward"]:
        lp, lse = _exact_logprob(s["hidden"], s["w"], s["targets"], case["temperature"], in_loss)
    else:  # the forward's results are this case's inputs
        lp, lse = s["lp"].to(F64), s["lse"].to(F64)
    loss, _, dlp = _exact_surrogate(lp, s["behav"], s["row_offsets"], in_loss, adv, 0)
    gh, gw = _exact_grads(s, dlp, lse, case["temperature"])
    out = {"dlp": dlp, "gh": gh, "gw": gw, "status": status}
    return dict(out, lp=lp, lse=lse, loss=loss) if case["forward"] else out


def _exact_controls(s, case):
    S, T = _segment_sums(s["tags"], s["offsets"])
    kbar = torch.where(T > 0, (s["j"] * T - S).to(F64) / T.clamp(min=1).to(F64),
                       torch.zeros_like(T, dtype=F64))
    adm = (kbar <= 16.0).to(U8)
    nb = case["bins"]
    b = torch.floor(kbar / 32.0 * nb).clamp(0, nb - 1).to(I64)
    hist = torch.bincount(b + nb * adm.to(I64), minlength=2 * nb).to(I32).view(2, nb)
    cap = case["capacity"]
    vals, (cnt, head) = s["ring"].values.clone(), s["ring"].state.tolist()
    k = max(math.ceil((1.0 - 1.0 / 3.0) * cnt - 1e-9), 1)
    kappa = torch.sort(vals).values[k - 1].reshape(1)
    x = s["unit_score"]
    keep = (x <= kappa).to(I64)
    drawn = torch.cumsum(keep, 0) - keep < _batch_units(case) if _batch_units(case) > 0 \
        else torch.ones_like(keep, dtype=torch.bool)
    dec = torch.where(drawn, keep, 2 + 0 * keep).to(U8)
    nd = int(drawn.sum())
    i = torch.arange(max(0, nd - cap), nd, device=DEV)
    vals[(head + i) % cap] = x[i]
    state = torch.tensor([min(cap, cnt + nd), (head + nd) % cap], device=DEV)
    return {"kbar": kbar, "admitted": adm, "hist": hist, "decision": dec, "kappa": kappa,
            "ring": vals, "ring_state": state}
