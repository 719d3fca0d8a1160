"""The workloads whose speed this library is measured on: forget requests and decode steps on a paged
KV cache, through the calls of ``PagedKVCache``.

Three families:
  replay   crop every agent to its tau, append its sanitized suffix, attend the suffix queries (one
           call per layer).  With a suffix of one token this is a re-decoded position.
  rounds   crop, then one ``replay_rounds`` call: turn-structured suffixes whose known turns are
           re-prefilled and whose dependent turns are re-decoded one position per round.
  branch   fork a base session several times, replay a different suffix on every branch, release the
           branches.
A pass leaves the cache as it found it (crop + append of the same length restores the page tables), so
passes repeat.  Outputs are the attention outputs and the K / V pools the pass wrote into.

Sizes are those of the repository's benchmark, its tests, and the sessions the method is reported on
(1.2k-1.3k tokens of a 32-layer GQA 32/8 model, about 133 of them recomputed).
"""
from __future__ import annotations

import random

import numpy as np
import torch

from paper_2609_04875_gb300.binding import (POLICY_SELECTIVE, TURN_INPUT, TURN_MODEL_DEP, TURN_MODEL_INDEP,
                                            PagedKVCache, replay_schedule)


def _replay(name, agents, layers, hq, hkv, d, ps, t, keep=(0.0, 0.0), suffix=(0, 0), prepared=False, shape_seed=1):
    """A replay case: sessions of t[0]..t[1] tokens; each keeps a share keep[0]..keep[1] of its tokens, or,
    with suffix[1] > 0, all but suffix[0]..suffix[1] of them.  prepared: the calls are marshalled once
    (prepare_*), as a program does that repeats them layer after layer and step after step."""
    return {"name": name, "family": "replay", "agents": agents, "layers": layers, "hq": hq, "hkv": hkv, "d": d,
            "ps": ps, "t_lo": t[0], "t_hi": t[1], "keep_lo": keep[0], "keep_hi": keep[1], "s_lo": suffix[0],
            "s_hi": suffix[1], "prepared": prepared, "shape_seed": shape_seed}


def _rounds(name, agents, hq, hkv, d, ps, p, turns, inp, out, indep, shape_seed=1):
    """A rounds case: clean prefixes of p[0]..p[1] tokens, then `turns` pairs of an input turn (inp) and a
    model turn (out); `indep` of the model turns (never the last) do not depend on the target."""
    return {"name": name, "family": "rounds", "agents": agents, "layers": 1, "hq": hq, "hkv": hkv, "d": d, "ps": ps,
            "p_lo": p[0], "p_hi": p[1], "turns": turns, "in_lo": inp[0], "in_hi": inp[1], "out_lo": out[0],
            "out_hi": out[1], "indep": indep, "shape_seed": shape_seed}


def _branch(name, branches, layers, hq, hkv, d, ps, t, suffix, shape_seed=1):
    """A branch case: a base session of t tokens, forked `branches` times; every branch keeps its own
    share of the base and replays suffix[0]..suffix[1] tokens."""
    return {"name": name, "family": "branch", "agents": branches, "layers": layers, "hq": hq, "hkv": hkv, "d": d,
            "ps": ps, "t_lo": t, "t_hi": t, "s_lo": suffix[0], "s_hi": suffix[1], "shape_seed": shape_seed}


def listed():
    return [
        # one forget request of a small single-layer model: launches and latency
        _replay("tiny", 1, 1, 8, 8, 64, 16, (640, 640), suffix=(128, 128)),
        # one forget request of a reported episode: every layer of a 32-layer model, short launches
        _replay("episode", 1, 32, 32, 8, 128, 16, (1330, 1330), suffix=(133, 133), prepared=True),
        # many agents' requests batched into one ragged launch, ordinary session lengths
        _replay("agent_batch", 16, 1, 32, 8, 128, 16, (2048, 8192), keep=(0.2, 0.9), shape_seed=3),
        # the same for a model with 64-wide heads and larger pages
        _replay("batch_d64", 6, 2, 32, 8, 64, 32, (1000, 6000), keep=(0.2, 0.9), shape_seed=4),
        # late targets of long sessions: few new tokens over long prefixes, bound by reading K and V
        _replay("short_suffix", 8, 1, 32, 8, 128, 16, (32784, 32784), suffix=(16, 16)),
        # early targets of long sessions, wide GQA groups: compute-bound prefill
        _replay("long_suffix", 4, 1, 64, 8, 128, 64, (20480, 20480), suffix=(16384, 16384)),
        # one long session, several layers: an early and a late target
        _replay("session_early", 1, 2, 32, 8, 128, 16, (16384, 16384), keep=(0.3, 0.3), prepared=True),
        _replay("session_late", 1, 8, 32, 8, 128, 16, (16384, 16384), keep=(0.9, 0.9), prepared=True),
        # one position re-decoded for every agent of a batch
        _replay("decode_batch", 16, 1, 32, 8, 128, 16, (2048, 8192), suffix=(1, 1), shape_seed=3),
        # one position re-decoded on one long session through every layer of a 32-layer model
        _replay("decode_deep", 1, 32, 64, 8, 128, 64, (12003, 12003), suffix=(1, 1), prepared=True),
        # turn-structured suffixes: a few prefill rounds and many decode rounds
        _rounds("rounds", 16, 32, 8, 128, 16, (1024, 4096), 4, (32, 256), (64, 192), 3),
        # branches of one base session: forks, copy-on-write, ragged short prefills, 64-wide heads
        _branch("branches", 8, 4, 32, 8, 64, 16, 3001, (33, 200)),
    ]


def _loguniform(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    """One more case of the listed ranges: any head layout, page size and depth the kernels take, sizes
    spread over their logarithm, and no more work than the largest listed case."""
    top = work(listed()[5])
    while True:
        d = rng.choice([64, 128, 128])
        hq, hkv = rng.choice([(8, 8), (32, 8), (32, 8), (16, 4), (64, 8), (16, 16), (32, 4), (12, 12), (24, 3)])
        ps = rng.choice([8, 16, 16, 32, 64, 128])
        seed = rng.randrange(1, 1 << 20)
        kind = rng.choice(["prefill", "prefill", "prefill", "short", "decode", "deep", "rounds", "branch"])
        if kind == "prefill":
            t = _loguniform(rng, 400, 20480)
            keep = sorted(rng.uniform(0.05, 0.95) for _ in range(2))
            c = _replay("", _loguniform(rng, 1, 16), rng.choice([1, 1, 2]), hq, hkv, d, ps, (t, int(t * rng.uniform(1, 3))),
                        keep=tuple(round(k, 3) for k in keep), shape_seed=seed)
            c["t_hi"] = min(c["t_hi"], 24576)
            c["t_lo"] = min(c["t_lo"], c["t_hi"])
        elif kind == "short":
            t = _loguniform(rng, 2000, 40000)
            s = _loguniform(rng, 2, 64)
            c = _replay("", _loguniform(rng, 1, 16), rng.choice([1, 2, 4]), hq, hkv, d, ps, (t, t + rng.randrange(500)),
                        suffix=(s, s + rng.randrange(20)), shape_seed=seed)
        elif kind == "decode":
            t = _loguniform(rng, 700, 16000)
            c = _replay("", _loguniform(rng, 1, 48), 1, hq, hkv, d, ps, (t, 2 * t), suffix=(1, rng.choice([1, 1, 2])),
                        shape_seed=seed)
        elif kind == "deep":
            t = _loguniform(rng, 500, 12000)
            s = min(_loguniform(rng, 1, 700), t // 2)
            c = _replay("", 1, rng.choice([8, 16, 32]), hq, hkv, d, ps, (t, t), suffix=(s, s), prepared=True,
                        shape_seed=seed)
        elif kind == "rounds":
            p = _loguniform(rng, 300, 3000)
            c = _rounds("", _loguniform(rng, 1, 16), hq, hkv, d, ps, (p, 2 * p), rng.choice([1, 2, 3]), (20, 200),
                        (16, 80), rng.choice([0, 1]), shape_seed=seed)
            c["indep"] = min(c["indep"], c["turns"] - 1)
        else:
            t = _loguniform(rng, 800, 8000)
            c = _branch("", _loguniform(rng, 2, 12), rng.choice([1, 2, 4]), hq, hkv, d, ps, t, (20, 20 + rng.randrange(200)),
                        shape_seed=seed)
        w = work(c)
        if w["flops"] <= 0.9 * top["flops"] and w["bytes"] <= 0.9 * top["bytes"]:
            del c["name"]
            return c


# ------------------------------------------------------------------ shapes
def _agents(case):
    """[(P, S)] of the case's agents: kept and replayed tokens."""
    rng = random.Random(case["shape_seed"])
    out = []
    for _ in range(case["agents"]):
        if case["family"] == "rounds":
            p = rng.randint(case["p_lo"], case["p_hi"])
            out.append((p, sum(n for n, _ in _turns(case)[len(out)])))
            continue
        t = rng.randint(case["t_lo"], case["t_hi"])
        if case["family"] == "branch":
            s = rng.randint(case["s_lo"], case["s_hi"])
            out.append((rng.randint(max(1, t // 2), t), s))
        elif case["s_hi"] > 0:
            s = rng.randint(case["s_lo"], case["s_hi"])
            out.append((t - s, s))
        else:
            p = min(max(1, round(t * rng.uniform(case["keep_lo"], case["keep_hi"]))), t - 1)
            out.append((p, t - p))
    return out


def _turns(case):
    """Per agent the suffix's turns (length, kind)."""
    rng = random.Random(case["shape_seed"] + 1)
    out = []
    for _ in range(case["agents"]):
        indep = set(rng.sample(range(case["turns"] - 1), case["indep"])) if case["indep"] else set()
        turns = []
        for k in range(case["turns"]):
            turns.append((rng.randint(case["in_lo"], case["in_hi"]), TURN_INPUT))
            turns.append((rng.randint(case["out_lo"], case["out_hi"]), TURN_MODEL_INDEP if k in indep else TURN_MODEL_DEP))
        out.append(tuple(turns))
    return out


def _units(case):
    """Attention work as (queries, keys) pairs: the queries are the last ones of the keys."""
    if case["family"] != "rounds":
        return [(s, p + s) for p, s in _agents(case)]
    take, _ = replay_schedule(_turns(case), POLICY_SELECTIVE)
    lens = [p for p, _ in _agents(case)]
    units = []
    for row in take:
        for i, t in enumerate(row):
            if t:
                lens[i] += int(t)
                units.append((int(t), lens[i]))
    return units


def work(case):
    """Attention: every unmasked (query, key) pair, K and V of the visible keys read once per pass (per
    round, where a round stands for one generated position), Q read and the output written; append: the
    suffix K and V read and written."""
    hq, hkv, d = case["hq"], case["hkv"], case["d"]
    flops = bytes_ = 0.0
    for s, n in _units(case):
        flops += 4.0 * d * hq * (s * (n - s) + s * (s + 1) / 2)
        bytes_ += 2.0 * (2 * n * hkv * d + 2 * s * hq * d) + 4.0 * (2 * s * hkv * d)
    return {"bytes": bytes_ * case["layers"], "flops": flops * case["layers"]}


# ------------------------------------------------------------------ inputs
def _randn(shape, seed, stream):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    g = torch.Generator(device=dev).manual_seed(1000003 * seed + stream)
    x = torch.empty(shape, dtype=torch.bfloat16, device=dev)
    flat = x.view(-1)
    for lo in range(0, flat.numel(), 1 << 28):
        n = min(1 << 28, flat.numel() - lo)
        flat[lo:lo + n] = torch.randn(n, generator=g, device=dev)
    return x


def _tensors(case, seed):
    """Prefix K, V (packed over agents; of the one base session for branches), suffix K, V and Q."""
    L, hq, hkv, d = case["layers"], case["hq"], case["hkv"], case["d"]
    agents = _agents(case)
    n_pre = case["t_lo"] if case["family"] == "branch" else sum(p for p, _ in agents)
    n_suf = sum(s for _, s in agents)
    return (_randn((L, n_pre, hkv, d), seed, 1), _randn((L, n_pre, hkv, d), seed, 2),
            _randn((L, n_suf, hkv, d), seed, 3), _randn((L, n_suf, hkv, d), seed, 4),
            _randn((L, n_suf, hq, d), seed, 5))


def _cu(lengths):
    return [0] + [int(x) for x in np.cumsum(lengths)]


def prepare(case, seed):
    L, hkv, d, ps = case["layers"], case["hkv"], case["d"], case["ps"]
    agents = _agents(case)
    branch = case["family"] == "branch"
    kp, vp, K, V, Q = _tensors(case, seed)
    cu = _cu([s for _, s in agents])
    row = max(-(-(p + s) // ps) for p, s in agents) + 1
    if branch:
        row = max(row, -(-case["t_lo"] // ps) + 1)
    pages = row + sum(-(-s // ps) + 2 for _, s in agents) if branch else sum(-(-(p + s) // ps) for p, s in agents) + 64
    k_pool = torch.zeros((L, pages, hkv, ps, d), dtype=torch.bfloat16, device="cuda")
    v_pool = torch.zeros_like(k_pool)
    order = np.random.default_rng(seed).permutation(pages).astype(np.int32).tolist()
    cache = PagedKVCache(L, hkv, d, ps, pages, max_seqs=len(agents) + 1, max_pages_per_seq=row, init_free_order=order,
                         k_pool=k_pool, v_pool=v_pool)
    out = torch.empty_like(Q)
    st = {"family": case["family"], "layers": L, "cache": cache, "cu": cu, "K": K, "V": V, "Q": Q, "out": out,
          "taus": [p + 1 for p, _ in agents], "result": {"out": out, "k_pool": k_pool, "v_pool": v_pool},
          "Q_layers": [Q[i] for i in range(L)], "out_layers": [out[i] for i in range(L)]}
    if branch:
        st["base"] = cache.seq_create()
        cache.append_kv(st["base"], kp, vp)
        return st
    seqs = st["seqs"] = [cache.seq_create() for _ in agents]
    cache.append_kv_batch(seqs, kp, vp, _cu([p for p, _ in agents]))  # the kept part of the sessions ...
    if case["family"] == "rounds":
        st["take"], _ = replay_schedule(_turns(case), POLICY_SELECTIVE)
        return st
    cache.append_kv_batch(seqs, V, K, cu)  # ... and a contaminated suffix that the replay replaces
    if case["prepared"]:
        st["calls"] = [cache.prepare_crop_batch(seqs, st["taus"]), cache.prepare_append_kv_batch(seqs, K, V, cu)]
        st["calls"] += [cache.prepare_replay_attn_batch(seqs, i, Q[i], cu, out[i]) for i in range(L)]
    return st


def run(state):
    cache, cu = state["cache"], state["cu"]
    if "calls" in state:
        for call in state["calls"]:
            call()
        return state["result"]
    if state["family"] == "rounds":
        cache.crop_batch(state["seqs"], state["taus"])
        cache.replay_rounds(state["seqs"], state["take"], cu, state["K"], state["V"], state["Q"], out=state["out"])
        return state["result"]
    if state["family"] == "branch":
        seqs = [cache.seq_fork(state["base"]) for _ in state["taus"]]
    else:
        seqs = state["seqs"]
    cache.crop_batch(seqs, state["taus"])
    cache.append_kv_batch(seqs, state["K"], state["V"], cu)
    for layer in range(state["layers"]):
        cache.replay_attn_batch(seqs, layer, state["Q_layers"][layer], cu, out=state["out_layers"][layer])
    if state["family"] == "branch":
        for s in reversed(seqs):
            cache.seq_release(s)
    return state["result"]


# ------------------------------------------------------------------ how close results have to be
def tolerance(case):
    """bf16 outputs of fp32 sums: the output's rounding (2^-9) and the softmax weights' (2^-9 each,
    independent across keys).  Against exact() the listed and drawn cases are 2.2e-3 to 2.4e-3 off in
    the 2-norm; one output's largest difference is a few bf16 steps of it (2^-8 of a value of about 8
    root mean squares, 0.03)."""
    return {"rel": 0.01, "max": 0.12}


def exact(case, seed):
    """Attention of the suffix queries over prefix + suffix by its plain definition in 64 bits."""
    if work(case)["flops"] > 8e12:
        return None  # over about 20 seconds in 64 bits
    L, hq, hkv, d = case["layers"], case["hq"], case["hkv"], case["d"]
    g = hq // hkv
    agents = _agents(case)
    kp, vp, K, V, Q = _tensors(case, seed)
    cup = [0] * (len(agents) + 1) if case["family"] == "branch" else _cu([p for p, _ in agents])
    cu = _cu([s for _, s in agents])
    out = torch.empty(Q.shape, dtype=torch.float64, device=Q.device)
    for i, (p, s) in enumerate(agents):
        pos = torch.arange(p, p + s, device=Q.device)
        step = max(1, (1 << 27) // ((p + s) * hq))  # queries at a time
        for layer in range(L):
            k = torch.cat([kp[layer, cup[i]:cup[i] + p], K[layer, cu[i]:cu[i + 1]]]).double().permute(1, 2, 0)
            v = torch.cat([vp[layer, cup[i]:cup[i] + p], V[layer, cu[i]:cu[i + 1]]]).double().permute(1, 0, 2)
            for lo in range(0, s, step):
                hi = min(s, lo + step)
                n = p + hi
                q = Q[layer, cu[i] + lo:cu[i] + hi].double().reshape(hi - lo, hkv, g, d).permute(1, 2, 0, 3)
                x = torch.matmul(q.reshape(hkv, g * (hi - lo), d), k[:, :, :n]) * d ** -0.5
                mask = torch.arange(n, device=Q.device)[None, :] > pos[lo:hi, None]
                x = x.view(hkv, g, hi - lo, n).masked_fill_(mask, float("-inf"))
                x = torch.softmax(x, dim=-1).view(hkv, g * (hi - lo), n)
                o = torch.matmul(x, v[:, :n]).view(hkv, g, hi - lo, d).permute(2, 0, 1, 3)
                out[layer, cu[i] + lo:cu[i] + hi] = o.reshape(hi - lo, hq, d)
    return {"out": out, "k_pool": None, "v_pool": None}
