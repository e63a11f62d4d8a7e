"""What the library's users have it do, as timed cases through its public calls.

Each listed case is one call pattern of the sampling path (acting, stepping,
rolling out, storing samples, preparing data, scoring trajectories) at a size
of this repository's workloads; draw() spreads the same patterns over the
ranges they are used in.  A case is a dict of plain values; prepare() makes
what a program holds before the call (markets, envs, ensembles, device
buffers), run() is one pass of the call pattern, work() the bytes and
operations it cannot do without, exact() its results in 64 bits.
"""
import numpy as np
import torch

import paper_2501_10709_gb300 as fr
from paper_2501_10709_gb300 import synth

PREC = {"fp32": fr.PREC_FP32, "bf16": fr.PREC_BF16, "fp16": fr.PREC_FP16, "bf16x3": fr.PREC_BF16X3,
        "fp8": fr.PREC_FP8}
STOCK_DIMS, CRYPTO_DIMS = (301, 256, 256, 30), (10, 128, 128, 3)
AGENTS_STOCK, AGENTS_CRYPTO = 3, 5
CASH = 100_000_000


def listed():
    return [
        # a live trading loop: one combined action for eight accounts per call
        {"name": "act_8", "kind": "act", "n": 8, "prec": "bf16"},
        # the unfused actor at the paper's env count
        {"name": "act_2048", "kind": "act", "n": 2048, "prec": "bf16"},
        # scoring a stored batch of observations with every agent
        {"name": "forward_77824", "kind": "forward", "n": 77824, "prec": "bf16"},
        # the same networks in the plain fp32 path (reference runs, calibration)
        {"name": "forward_fp32_8192", "kind": "forward", "n": 8192, "prec": "fp32"},
        # a learner's Double DQN targets for a batch of replay samples
        {"name": "q_targets_65536", "kind": "q_targets", "n": 65536, "prec": "fp16", "double": True, "dueling": False},
        # one VecEnv step with observations out, more envs than the L2 holds
        {"name": "step_stock_262144", "kind": "step_stock", "n": 262144, "assets": 30, "float_actions": True,
         "largest_first": False},
        # the same for the one-asset crypto envs
        {"name": "step_crypto_131072", "kind": "step_crypto", "n": 131072},
        # the paper's 2,048 envs, a whole rollout with the actors in the loop,
        # the actors new in every rollout (indicator table rebuilt)
        {"name": "rollout_stock_2048x256", "kind": "rollout_stock", "n": 2048, "steps": 256, "uneven": False,
         "prec": "bf16"},
        # second-level crypto envs under a five-agent vote
        {"name": "rollout_crypto_8192x1024", "kind": "rollout_crypto", "n": 8192, "steps": 1024, "prec": "fp16"},
        # a training iteration's samples: a recorded rollout pushed into the
        # replay buffer, and a minibatch drawn from it
        {"name": "collect_2048x64", "kind": "collect", "n": 2048, "steps": 64, "batch": 4096},
        # the indicator table of a market of 1,000 days and 30 assets
        {"name": "indicators_1000x30", "kind": "indicators", "days": 1000, "assets": 30},
        # the performance metrics of a stored batch of trajectories
        {"name": "traj_metrics_2048x256", "kind": "traj_metrics", "n": 2048, "steps": 256, "dones": False},
    ]


def _log(rng, lo, hi):
    return int(round(float(np.exp(rng.uniform(np.log(lo), np.log(hi))))))


def draw(rng):
    kind = rng.choice(["act", "forward", "q_targets", "step_stock", "step_crypto", "rollout_stock",
                       "rollout_crypto", "collect", "indicators", "traj_metrics"])
    c = {"kind": kind}
    if kind == "act":
        c.update(n=_log(rng, 1, 4096), prec=rng.choice(["bf16", "bf16", "fp16", "fp8"]))
    elif kind == "forward":
        c["prec"] = rng.choice(["bf16", "fp16", "fp8", "fp32"])
        c["n"] = _log(rng, 256, 8192) if c["prec"] == "fp32" else _log(rng, 2048, 77824)
    elif kind == "q_targets":
        c.update(n=_log(rng, 256, 65536), prec=rng.choice(["fp16", "bf16x3", "fp32"]), double=rng.random() < 0.7,
                 dueling=rng.random() < 0.4)
    elif kind == "step_stock":
        c.update(n=_log(rng, 1, 262144), assets=rng.choice([30, 30, 30, rng.randint(1, 32)]),
                 float_actions=rng.random() < 0.7, largest_first=rng.random() < 0.2)
    elif kind == "step_crypto":
        c.update(n=_log(rng, 1, 131072))
    elif kind == "rollout_stock":
        c.update(n=_log(rng, 8, 4096), steps=_log(rng, 16, 256), uneven=rng.random() < 0.4,
                 prec=rng.choice(["bf16", "bf16", "fp16", "fp8"]))
    elif kind == "rollout_crypto":
        c.update(n=_log(rng, 64, 8192), steps=_log(rng, 64, 512), prec=rng.choice(["fp16", "fp16", "bf16"]))
    elif kind == "collect":
        c.update(n=_log(rng, 64, 2048), steps=_log(rng, 8, 64), batch=_log(rng, 256, 16384))
    elif kind == "indicators":
        c.update(days=_log(rng, 100, 2520), assets=_log(rng, 5, 100))
    else:
        c.update(n=_log(rng, 64, 8192), steps=_log(rng, 16, 1024), dones=rng.random() < 0.5)
    return c


# ------------------------------------------------------------------- inputs

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed & 0x7FFFFFFF)
    return g


def _stock_obs(n, seed):
    """Observations as the stock envs show them: cash, prices, holdings (many
    of them zero) and small indicator ratios."""
    g = _gen(seed)
    r = lambda *s: torch.rand(*s, device="cuda", generator=g)  # noqa: E731
    cash, price = r(n, 1), 0.2 + 3.8 * r(n, 30)
    hold = torch.floor(300 * torch.clamp(r(n, 30) - 0.4, min=0.0)) * 0.01
    ind = 0.1 * torch.randn(n, 240, device="cuda", generator=g)
    return torch.cat([cash, price, hold, ind], 1).contiguous()


def _crypto_obs(n, seed):
    g = _gen(seed)
    cash = torch.rand(n, 1, device="cuda", generator=g)
    pos = torch.randint(0, 11, (n, 1), device="cuda", generator=g) / 10.0
    fac = torch.clamp(torch.randn(n, 8, device="cuda", generator=g), -5.0, 5.0)
    return torch.cat([cash, pos, fac], 1).contiguous()


def _stock_ensemble(ctx, prec, seed):
    e = fr.ensemble_create(ctx, STOCK_DIMS, synth.actor_params(STOCK_DIMS, AGENTS_STOCK, seed), precision=PREC[prec])
    if prec == "fp8":
        fr.ensemble_calibrate_sync(e, _stock_obs(4096, seed + 7))
    return e


def _q_dims(case):
    return CRYPTO_DIMS[:-1] + (4,) if case["dueling"] else CRYPTO_DIMS


def _q_params(case, seed, which):
    return synth.actor_params(_q_dims(case), AGENTS_CRYPTO, seed + which, out_scale=4.0)


def _q_heads(case):
    return [fr.HEAD_DUELING if case["dueling"] and j % 2 else fr.HEAD_Q for j in range(AGENTS_CRYPTO)]


def _q_batch(case, seed):
    g = _gen(seed + 1)
    rew = 0.05 * torch.randn(case["n"], device="cuda", generator=g)
    done = (torch.rand(case["n"], device="cuda", generator=g) < 0.01).to(torch.uint8)
    return _crypto_obs(case["n"], seed), rew, done


STEP_DAYS, STEP_WARM = 500, 4


def _step_stock_inputs(case, seed):
    n, k = case["n"], case["assets"]
    rng = np.random.default_rng(seed)
    mk = synth.stock_market(STEP_DAYS, k, seed)
    start = rng.integers(60, STEP_DAYS - 250, n).astype(np.int32)
    bps = rng.integers(-100, 101, (n, k), dtype=np.int16)
    g = _gen(seed)
    acts = []
    for _ in range(STEP_WARM + 1):
        u = torch.rand(n, k, device="cuda", generator=g) * 2.4 - 1.2
        if not case["float_actions"]:
            u = torch.trunc(torch.clamp(u, -1.0, 1.0) * 100).to(torch.int32)
        acts.append(u.contiguous())
    return mk, start, bps, acts


def _step_crypto_inputs(case, seed):
    n = case["n"]
    mk = synth.crypto_market(50_000, seed)
    start = np.random.default_rng(seed).integers(3600, 50_000 - 3600, n).astype(np.int32)
    g = _gen(seed)
    acts = [torch.randint(0, 3, (n,), device="cuda", generator=g).to(torch.uint8) for _ in range(STEP_WARM + 1)]
    return mk, start, acts


def _ohlc(case, seed):
    m = synth.stock_market(case["days"], case["assets"], seed)
    return [np.ascontiguousarray(x) for x in (m.close, m.high, m.low)]


def _traj(case, seed):
    """Rewards of value paths with 1% steps, and the done flags of windows."""
    g = _gen(seed)
    T, n = case["steps"], case["n"]
    walk = torch.cumsum(0.01 * torch.randn(T, n, device="cuda", generator=g, dtype=torch.float64), 0)
    v = torch.round(CASH * torch.exp(walk)).to(torch.int64)
    rew = torch.diff(v, dim=0, prepend=torch.full((1, n), CASH, device="cuda", dtype=torch.int64)).contiguous()
    done = None
    if case["dones"]:
        last = torch.randint(0, 2 * T, (n,), device="cuda", generator=g)
        done = (torch.arange(T, device="cuda")[:, None] >= last[None, :]).to(torch.uint8).contiguous()
    return rew, done


# ------------------------------------------------------------------ prepare

def _state_buffers(env, hold=True):
    dev = "cuda"
    return {"cash": torch.empty(env.N, dtype=torch.int64, device=dev),
            "hold": torch.empty(env.N * env.K, dtype=torch.int32, device=dev),
            "steps": torch.empty(env.N, dtype=torch.int32, device=dev),
            "done": torch.empty(env.N, dtype=torch.uint8, device=dev)}


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case, "kind": kind}
    if kind == "indicators":
        s["ohlc"] = [torch.from_numpy(x).cuda() for x in _ohlc(case, seed)]
        s["out"] = torch.empty(case["days"], 8, case["assets"], device="cuda")
        return s
    if kind == "traj_metrics":
        s["rew"], s["done"] = _traj(case, seed)
        s["out"] = torch.empty(case["n"], 11, dtype=torch.float64, device="cuda")
        return s
    ctx = s["ctx"] = fr.fr_ctx_create(0)
    if kind in ("act", "forward"):
        s["ens"] = _stock_ensemble(ctx, case["prec"], seed)
        s["obs"] = _stock_obs(case["n"], seed)
        s["out"] = torch.empty(*((case["n"], 30) if kind == "act" else (AGENTS_STOCK, case["n"], 30)), device="cuda")
    elif kind == "q_targets":
        new = lambda w: fr.ensemble_create(ctx, _q_dims(case), _q_params(case, seed, w),  # noqa: E731
                                           precision=PREC[case["prec"]], combine=fr.COMBINE_VOTE, out_act=0,
                                           heads=_q_heads(case))
        s["online"], s["target"] = new(0), new(1)
        s["batch"] = _q_batch(case, seed)
        s["out"] = torch.empty(AGENTS_CRYPTO, case["n"], device="cuda")
    elif kind in ("step_stock", "step_crypto"):
        if kind == "step_stock":
            mk, start, bps, acts = _step_stock_inputs(case, seed)
            s["mk"] = fr.fr_market_create(ctx, mk)
            s["env"] = fr.env_create(ctx, s["mk"], start=start, window=250, bps=bps, auto_reset=True,
                                     buy_order=fr.BUY_LARGEST_FIRST if case["largest_first"] else fr.BUY_ASCENDING)
            s["act_kind"] = fr.ACT_F32_UNIT if case["float_actions"] else fr.ACT_I32_SHARES
        else:
            mk, start, acts = _step_crypto_inputs(case, seed)
            s["mk"] = fr.fr_market_create(ctx, mk)
            s["env"] = fr.env_create(ctx, s["mk"], start=start, window=3600, auto_reset=True)
            s["act_kind"] = fr.ACT_U8_DISCRETE
        env = s["env"]
        for a in acts[:-1]:
            fr.env_step(env, a, s["act_kind"])
        torch.cuda.synchronize()
        s["act"] = acts[-1]
        s["out"] = {"rew": torch.empty(env.N, dtype=torch.int64, device="cuda"),
                    "rew_f32": torch.empty(env.N, device="cuda"),
                    "done": torch.empty(env.N, dtype=torch.uint8, device="cuda"),
                    "obs": torch.empty(env.N, env.D, device="cuda")}
    elif kind in ("rollout_stock", "collect"):
        n, T = case["n"], case["steps"]
        days = 1000
        mk = synth.stock_market(days, 30, seed)
        if case.get("uneven"):
            e = synth.stock_envs_uneven(n, 30, days, w_lo=5, w_hi=T + 1, seed=seed)
        else:
            e = synth.stock_envs_cohorts(n, 30, days, T + 1, 128, seed)
        s["mk"] = fr.fr_market_create(ctx, mk)
        env = s["env"] = fr.env_create(ctx, s["mk"], start=e.start, window=e.W, n_assets=e.Ke, bps=e.bps)
        s["ens"] = _stock_ensemble(ctx, case.get("prec", "bf16"), seed)
        fr.env_set_table_cache(env, False)
        s["metrics"] = torch.empty(n, 3, dtype=torch.float64, device="cuda")
        if kind == "rollout_stock":
            s["state"] = _state_buffers(env)
        else:
            dev, B = "cuda", case["batch"]
            s["rb"] = fr.replay_create(ctx, env, 262144)
            s["seed"] = seed
            s["traj"] = {"obs": torch.empty(T, n, env.D, device=dev), "act": torch.empty(T, n, 30, device=dev),
                         "rew": torch.empty(T, n, dtype=torch.int64, device=dev),
                         "rew_f32": torch.empty(T, n, device=dev),
                         "done": torch.empty(T, n, dtype=torch.uint8, device=dev)}
            s["last"] = torch.empty(n, env.D, device=dev)
            s["sample"] = {"obs": torch.empty(B, env.D, device=dev), "next_obs": torch.empty(B, env.D, device=dev),
                           "act": torch.empty(B, 30, device=dev), "rew": torch.empty(B, device=dev),
                           "done": torch.empty(B, dtype=torch.uint8, device=dev),
                           "index": torch.empty(B, dtype=torch.int64, device=dev)}
    elif kind == "rollout_crypto":
        n, T, S = case["n"], case["steps"], 100_000
        mk = synth.crypto_market(S, seed)
        e = synth.crypto_envs(n, S, T + 1, seed)
        s["mk"] = fr.fr_market_create(ctx, mk)
        env = s["env"] = fr.env_create(ctx, s["mk"], start=e.start, window=e.W, pmax=e.pmax)
        s["ens"] = fr.ensemble_create(ctx, CRYPTO_DIMS, synth.actor_params(CRYPTO_DIMS, AGENTS_CRYPTO, seed,
                                                                          out_scale=4.0),
                                      precision=PREC[case["prec"]], combine=fr.COMBINE_VOTE, out_act=0)
        s["metrics"] = torch.empty(n, 3, dtype=torch.float64, device="cuda")
        s["state"] = _state_buffers(env)
    else:
        raise ValueError(kind)
    return s


# ---------------------------------------------------------------------- run

def run(s):
    kind = s["kind"]
    if kind == "act":
        fr.ensemble_act(s["ens"], s["obs"], s["out"])
    elif kind == "forward":
        fr.ensemble_forward(s["ens"], s["obs"], s["out"])
    elif kind == "q_targets":
        obs, rew, done = s["batch"]
        fr.ensemble_q_targets(s["online"], s["target"], obs, rew, done, gamma=0.99, double_q=s["case"]["double"],
                              y=s["out"])
    elif kind in ("step_stock", "step_crypto"):
        fr.env_step(s["env"], s["act"], s["act_kind"], **s["out"])
    elif kind == "indicators":
        fr.market_indicators(*s["ohlc"], out=s["out"])
    elif kind == "traj_metrics":
        fr.trajectory_metrics(s["rew"], s["done"], v0=CASH, out=s["out"])
    elif kind in ("rollout_stock", "rollout_crypto"):
        fr.env_reset(s["env"])
        fr.rollout(s["env"], s["ens"], s["case"]["steps"], metrics=s["metrics"])
        fr.env_get_state(s["env"], **s["state"])
        return {"metrics": s["metrics"], **s["state"]}
    else:
        env, T, tr = s["env"], s["case"]["steps"], s["traj"]
        fr.env_reset(env)
        fr.rollout(env, s["ens"], T, traj=tr, metrics=s["metrics"])
        fr.env_observe(env, s["last"])
        fr.replay_push(s["rb"], env, tr, T, s["last"])
        fr.replay_sample(s["rb"], s["case"]["batch"], s["seed"], out=s["sample"])
        return {"traj": tr, "last": s["last"], "metrics": s["metrics"], "sample": s["sample"]}
    return s["out"]


# --------------------------------------------------------------------- work

def _mlp(dims, agents):
    return (2 * agents * sum(a * b for a, b in zip(dims, dims[1:])),
            4 * agents * sum(a * b + b for a, b in zip(dims, dims[1:])))


def work(case):
    kind = case["kind"]
    if kind in ("act", "forward"):
        fl, wb = _mlp(STOCK_DIMS, AGENTS_STOCK)
        out = 120 * (AGENTS_STOCK if kind == "forward" else 1)
        return {"bytes": case["n"] * (1204 + out) + wb, "flops": case["n"] * fl}
    if kind == "q_targets":
        fl, wb = _mlp(_q_dims(case), AGENTS_CRYPTO)
        nets = 2 if case["double"] else 1
        return {"bytes": case["n"] * (40 + 5 + 4 * AGENTS_CRYPTO) + nets * wb, "flops": case["n"] * fl * nets}
    if kind == "step_stock":
        # per env: action row, constants (asset count, start, window, bps) and
        # state (cash, holdings, step, done, accumulators) read, state, reward
        # (twice), done flag and observation written; the market once
        k = case["assets"]
        per = 4 * k + (12 + 2 * k) + 2 * (8 + 4 * k + 4 + 1 + 40) + 13 + 4 * (1 + 10 * k)
        return {"bytes": case["n"] * per + STEP_DAYS * k * 40, "flops": case["n"] * k * 20}
    if kind == "step_crypto":
        per = 1 + 12 + 2 * (8 + 4 + 4 + 1 + 40) + 13 + 40 + 49
        return {"bytes": case["n"] * per, "flops": case["n"] * 40}
    if kind in ("rollout_stock", "collect"):
        fl, wb = _mlp(STOCK_DIMS, AGENTS_STOCK)
        n, T = case["n"], case["steps"]
        steps = n * (T + 4) / 2 if case.get("uneven") else n * T
        by = n * 2 * 300 + wb + 1000 * 30 * 40
        if kind == "collect":
            # trajectory rows written, read back, stored as transitions
            # (observations twice), and the minibatch read and written
            row = 1204 + 120 + 8 + 4 + 1
            by += n * T * (2 * row + 2 * 1204 + 125) + 2 * case["batch"] * (2 * 1204 + 133)
        return {"bytes": by, "flops": steps * fl}
    if kind == "rollout_crypto":
        fl, wb = _mlp(CRYPTO_DIMS, AGENTS_CRYPTO)
        return {"bytes": case["n"] * 200 + wb + 100_000 * 41, "flops": case["n"] * case["steps"] * fl}
    if kind == "indicators":
        return {"bytes": case["days"] * case["assets"] * 56, "flops": case["days"] * case["assets"] * 500}
    b = case["n"] * case["steps"] * (9 if case["dones"] else 8) + case["n"] * 88
    return {"bytes": b, "flops": case["n"] * case["steps"] * 20}


# -------------------------------------------------------------------- exact

def _mlp64(dims, flat, x, tanh):
    layers = synth.unpack_params(dims, flat)
    for i, (W, b) in enumerate(layers):
        W = torch.from_numpy(np.ascontiguousarray(W)).cuda().double().reshape(dims[i + 1], dims[i])
        x = x @ W.T + torch.from_numpy(np.ascontiguousarray(b)).cuda().double()
        x = torch.relu(x) if i + 1 < len(layers) else (torch.tanh(x) if tanh else x)
    return x


def _heads64(case, j, y):
    if not case["dueling"]:
        return y
    if j % 2 == 0:
        return y[:, :3]
    return y[:, :1] + y[:, 1:] - y[:, 1:].mean(1, keepdim=True)


def _price(close, bps):
    return np.maximum(1, (close * (10_000 + bps) + 5_000) // 10_000)


def _step_stock64(case, seed):
    """One step after the warm-up steps, in whole numbers, asset by asset."""
    mk, start, bps, acts = _step_stock_inputs(case, seed)
    n, k = case["n"], case["assets"]
    b = bps.astype(np.int64)
    cash, hold = np.full(n, CASH, np.int64), np.zeros((n, k), np.int64)
    fee = lambda g: (g * 10 + 9_999) // 10_000  # noqa: E731
    rew = None
    for t, a in enumerate(acts):
        a = a.cpu().numpy()
        if case["float_actions"]:
            q = np.trunc(np.clip(a.astype(np.float64), -1.0, 1.0) * 100).astype(np.int64)
        else:
            q = a.astype(np.int64)
        p, p1 = _price(mk.close[start + t], b), _price(mk.close[start + t + 1], b)
        v0 = cash + (p * hold).sum(1)
        sell = np.minimum(np.maximum(-q, 0), hold)
        g = sell * p
        cash, hold = cash + (g - fee(g)).sum(1), hold - sell
        order = (np.argsort(-np.maximum(q, 0), axis=1, kind="stable") if case["largest_first"]
                 else np.broadcast_to(np.arange(k), (n, k)))
        rows = np.arange(n)
        for i in range(k):
            j = order[:, i]
            pj = p[rows, j]
            buy = np.minimum(np.maximum(q[rows, j], 0), cash * 10_000 // (pj * 10_010))
            cost = buy * pj + fee(buy * pj)
            over = cost > cash
            buy = np.where(over, buy - 1, buy)
            more = buy + 1
            fits = (more <= q[rows, j]) & (more * pj + fee(more * pj) <= cash)
            buy = np.where(fits, more, buy)
            cash = cash - (buy * pj + fee(buy * pj))
            hold[rows, j] += buy
        rew = cash + (p1 * hold).sum(1) - v0
    return rew, cash, hold, p1


def exact(case, seed):
    kind = case["kind"]
    if kind in ("act", "forward"):
        P = synth.actor_params(STOCK_DIMS, AGENTS_STOCK, seed)
        x = _stock_obs(case["n"], seed).double()
        y = torch.stack([_mlp64(STOCK_DIMS, P[j], x, True) for j in range(AGENTS_STOCK)])
        return y if kind == "forward" else y.mean(0)
    if kind == "q_targets":
        obs, rew, done = _q_batch(case, seed)
        on, tg = _q_params(case, seed, 0), _q_params(case, seed, 1)
        out = []
        for j in range(AGENTS_CRYPTO):
            qt = _heads64(case, j, _mlp64(_q_dims(case), tg[j], obs.double(), False))
            qo = _heads64(case, j, _mlp64(_q_dims(case), on[j], obs.double(), False)) if case["double"] else qt
            best = torch.gather(qt, 1, qo.argmax(1, keepdim=True))[:, 0]
            out.append(rew.double() + torch.where(done != 0, 0.0, 0.99) * best)
        return torch.stack(out)
    if kind == "step_stock":
        rew, cash, hold, p = _step_stock64(case, seed)
        # the indicators of the observation are checked by their own case
        return {"rew": None, "rew_f32": rew * 1e-6, "done": None, "obs": None}
    if kind == "step_crypto":
        mk, start, acts = _step_crypto_inputs(case, seed)
        cash, pos = np.full(case["n"], CASH, np.int64), np.zeros(case["n"], np.int64)
        rew = None
        for t, a in enumerate(acts):
            a, d = a.cpu().numpy(), start + t
            m, sp = mk.mid[d], mk.spread[d].astype(np.int64)
            v0, bid = cash + pos * m, m - sp // 2
            ask = bid + sp
            buy = (a == 2) & (pos < 10) & (cash >= ask)
            sell = (a == 0) & (pos > 0)
            cash = cash - np.where(buy, ask, 0) + np.where(sell, bid, 0)
            pos = pos + buy - sell
            rew = cash + pos * mk.mid[d + 1] - v0
        d = start + len(acts)
        obs = np.concatenate([cash[:, None] * 1e-8, pos[:, None] / 10.0, mk.fac[d].astype(np.float64)], 1)
        return {"rew": None, "rew_f32": rew * 1e-6, "done": None, "obs": obs}
    if kind == "indicators":
        return _indicators64(*[x.astype(np.float64) for x in _ohlc(case, seed)])
    if kind == "traj_metrics":
        rew, done = _traj(case, seed)
        return _traj64(rew.cpu().numpy(), None if done is None else done.cpu().numpy())
    # whole rollouts: the actors' rounding decides the trades, and what follows
    # from them has no value of its own in 64 bits
    return None


def _indicators64(c, h, lo):
    T, K = c.shape
    out = np.zeros((T, 8, K))
    tp = (h + lo + c) / 3.0
    a12, a26 = 2.0 / 13.0, 2.0 / 27.0
    e12, e26 = c[0].copy(), c[0].copy()
    z = np.zeros(K)
    G, L, TR, DP, DM = z, z, z, z, z
    for t in range(T):
        cp = c[t - 1] if t else c[0]
        d = c[t] - cp
        tr = np.maximum(np.maximum(h[t] - lo[t], np.abs(h[t] - cp)), np.abs(lo[t] - cp))
        up = h[t] - h[t - 1] if t else z
        dn = lo[t - 1] - lo[t] if t else z
        new = [np.maximum(d, 0), np.maximum(-d, 0), tr, np.where((up > dn) & (up > 0), up, 0.0),
               np.where((dn > up) & (dn > 0), dn, 0.0)]
        if t:
            e12, e26 = a12 * c[t] + (1 - a12) * e12, a26 * c[t] + (1 - a26) * e26
            G, L, TR, DP, DM = (w + (x - w) / 30.0 for w, x in zip((G, L, TR, DP, DM), new))
        else:
            G, L, TR, DP, DM = new
        out[t, 0] = (e12 - e26) / c[t]
        w20, w30, w60 = c[max(0, t - 19):t + 1], c[max(0, t - 29):t + 1], c[max(0, t - 59):t + 1]
        s, sd = w20.mean(0), w20.std(0)
        out[t, 1], out[t, 2] = (s + 2 * sd) / c[t] - 1, (s - 2 * sd) / c[t] - 1
        with np.errstate(divide="ignore", invalid="ignore"):
            rsi = np.where(L > 0, 100 - 100 / (1 + G / L), np.where(G > 0, 100.0, 50.0))
            wt = tp[max(0, t - 29):t + 1]
            mad = np.abs(wt - wt.mean(0)).mean(0)
            cci = np.where(mad > 0, (tp[t] - wt.mean(0)) / (0.015 * mad), 0.0)
            den = np.where(TR > 0, TR, 1.0)
            p, m = 100 * DP / den, 100 * DM / den
            dx = np.where(p + m > 0, 100 * np.abs(p - m) / (p + m), 0.0)
        out[t, 3], out[t, 4], out[t, 5] = rsi / 100, cci / 100, dx / 100
        out[t, 6], out[t, 7] = w30.mean(0) / c[t] - 1, w60.mean(0) / c[t] - 1
    return out


def _traj64(rew, done, ann=252.0, gamma=0.99):
    T, n = rew.shape
    live = np.ones((T, n), bool)
    if done is not None:
        live[1:] = np.cumsum(done[:-1] != 0, 0) == 0
    cnt = live.sum(0)
    v = CASH + np.cumsum(np.where(live, rew, 0), 0)
    prev = np.vstack([np.full((1, n), CASH), v[:-1]])
    rho = np.where(live, v / prev - 1.0, 0.0)
    mean = rho.sum(0) / cnt
    var = np.where(live, (rho - mean) ** 2, 0.0).sum(0) / np.maximum(cnt - 1, 1)
    sd = np.sqrt(np.where(cnt > 1, var, 0.0))
    peak = np.maximum.accumulate(np.maximum(v, CASH), 0)
    mdd = np.minimum((v / peak - 1.0).min(0), 0.0)
    cr = v[-1] / CASH - 1.0
    annual = (v[-1] / CASH) ** (ann / cnt) - 1.0
    down = np.sqrt((np.minimum(rho, 0.0) ** 2).sum(0) / cnt)
    neg, pos = np.maximum(-rho, 0.0).sum(0), np.maximum(rho, 0.0).sum(0)
    disc = (np.where(live, rew, 0) * (gamma ** np.arange(1, T + 1))[:, None]).sum(0)
    ratio = lambda a, b: np.where(b != 0, a / np.where(b != 0, b, 1.0), 0.0)  # noqa: E731
    return np.stack([cr, ratio(mean, sd) * np.sqrt(ann), mdd, annual, sd * np.sqrt(ann), ratio(cr, -mdd),
                     ratio(mean, down) * np.sqrt(ann), ratio(annual, -mdd), ratio(pos, neg), disc, cnt], 1)
