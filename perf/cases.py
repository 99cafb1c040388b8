"""Timing cases of the KV-eviction step, through the package's public entry points.

Every case is one call of a user's program on attention shapes of this repository's workloads (32 query
heads, 8 KV heads, head_dim 128). `way` names the calls that make up one pass:

  step      kv_evict_score, then kv_evict_select_gather: the eviction step at the end of a prefill
  lse       kv_evict_score_lse (the prefill hands over its rows' softmax normalisers), then
            kv_evict_select_gather
  attn      kv_evict_score_attn (the window rows' attention output comes with the score), then
            kv_evict_select_gather
  noalloc   kv_evict_score, kv_evict_select_noalloc, kv_evict_gather: an engine that cannot allocate at
            eviction time and keeps a token-major cache
  perq      the step with one selection per query head
  every     kv_evict_score, then kv_evict_select over every candidate
  profiles  kv_evict_select_profiles on given mu and sigma: one batch of a search over profiles

Integer outputs and the compact caches (copied bit for bit, returned as 16-bit words) are compared value
by value; mu, sigma and the window rows' output as numbers.
"""

from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2609_30738_gb300 import kv_evict, synth, workloads

HQ, HKV, D = 32, 8, 128
G = HQ // HKV
# the three-segment profile with a mid-layer sign flip of lambda2 (latent values, lambda = sinh(a))
SEGMENTS = ((0.3, 0.3, 0.3), (-0.8, 0.6, -0.8))


def _case(name, way, layers, lens, window=32, budget=64, lam="global", profiles=1, salient=0.0):
    c = dict(way=way, layers=layers, lens=",".join(str(x) for x in lens), window=window, budget=budget,
             lam=lam, profiles=profiles, salient=salient)
    return dict(c, name=name) if name else c


def listed():
    return [
        # one layer at a time, as a prefill that evicts each layer when it is done with it: latency
        _case("step-1layer-L2048", "step", 1, [2048]),
        # a short chat prompt of odd length with the paper's window of 8, in an engine that owns all memory
        _case("noalloc-32layer-L741-W8", "noalloc", 32, [741], window=8),
        # ordinary prompts: a whole model's step at 8k tokens
        _case("step-32layer-L8192", "step", 32, [8192]),
        # the paper's own timing: HotpotQA prompts of 15.6k tokens on average, window 8
        _case("step-32layer-L15611-W8", "step", 32, [15611], window=8, lam="paper"),
        # twice the budget and a profile by layer segments
        _case("step-32layer-L16384-B128", "step", 32, [16384], budget=128, lam="segments"),
        # the long-context step
        _case("step-32layer-L32768", "step", 32, [32768], salient=0.2),
        # a batch of ragged requests: the largest call
        _case("step-32layer-ragged6", "step", 32, [4099, 9473, 16001, 21250, 27777, 32705], lam="quadratic"),
        # a prefill that hands over its normalisers, at an odd length
        _case("lse-32layer-L20011", "lse", 32, [20011]),
        # the window rows' attention output from the same pass
        _case("attn-32layer-L8192", "attn", 32, [8192]),
        # the ablation with a selection per query head
        _case("perq-32layer-L4096", "perq", 32, [4096]),
        # the ablation with every token a candidate, both signs of lambda2 over the layers
        _case("every-6layer-L4096", "every", 6, [4096], lam="segments"),
        # a search over coefficient profiles re-selects for each
        _case("profiles14-32layer-L8192", "profiles", 32, [8192], lam="search", profiles=14),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    way = rng.choice(["step", "step", "step", "lse", "attn", "noalloc", "perq", "every", "profiles"])
    window = rng.choice([8, 32])
    budget = rng.choice([32, 64, 64, 128])
    lam = rng.choice(["global", "paper", "segments", "quadratic"])
    salient = rng.choice([0.0, 0.2])
    layers = rng.choice([1, _log_int(rng, 2, 32), 32])
    if way == "step":
        lens = [_log_int(rng, 700, 32768) for _ in range(rng.choice([1, 1, 2, 3]))]
        return _case(None, way, layers, lens, window, budget, lam, salient=salient)
    if way == "lse":
        return _case(None, way, layers, [_log_int(rng, 2000, 32768)], window, budget, lam, salient=salient)
    if way == "attn":
        return _case(None, way, layers, [_log_int(rng, 1000, 16384)], window, budget, lam, salient=salient)
    if way == "noalloc":
        return _case(None, way, layers, [_log_int(rng, 700, 16384)], window, budget, lam, salient=salient)
    if way == "perq":
        return _case(None, way, layers, [_log_int(rng, 700, 8192)], window, min(budget, 64), lam, salient=salient)
    if way == "every":
        return _case(None, way, min(layers, 6), [_log_int(rng, 1000, 4096)], window, min(budget, 64), lam)
    return _case(None, way, layers, [_log_int(rng, 1000, 16384)], window, min(budget, 64), "search",
                 profiles=rng.randint(2, 20))


def _spec(case):
    return dict(num_layers=case["layers"], num_q_heads=HQ, num_kv_heads=HKV, head_dim=D,
                window=case["window"], budget=case["budget"], pool_kernel=7,
                candidate_factor=0 if case["way"] == "every" else 4, norm_eps=1e-12,
                seq_lens=[int(x) for x in case["lens"].split(",")], salient_frac=case["salient"])


def _lambdas(case, seed):
    """The layer-wise coefficients: float32 [N_L] each, or [profiles, N_L] for a search."""
    n = case["layers"]
    t = np.arange(n) * 3 // n   # the layer's third
    if case["lam"] == "global":
        l1, l2 = np.full(n, 0.5), np.full(n, -0.5)
    elif case["lam"] == "paper":
        l1, l2 = np.zeros(n), np.full(n, -0.15)
    elif case["lam"] == "segments":
        l1, l2 = (np.sinh(np.asarray(a)[t]) for a in SEGMENTS)
    elif case["lam"] == "quadratic":
        mid = max((n - 1) / 2.0, 0.5)
        l1, l2 = np.full(n, 0.2), -0.6 + 1.2 * ((np.arange(n) - mid) / mid) ** 2 - 0.6
    else:
        rng = random.Random(seed)
        draws = [([rng.uniform(-0.5, 1.0) for _ in range(3)], [rng.uniform(-1.0, 0.6) for _ in range(3)])
                 for _ in range(case["profiles"])]
        l1 = np.stack([np.sinh(np.asarray(a)[t]) for a, _ in draws])
        l2 = np.stack([np.sinh(np.asarray(b)[t]) for _, b in draws])
    return np.ascontiguousarray(l1, dtype=np.float32), np.ascontiguousarray(l2, dtype=np.float32)


def _inputs(case, seed):
    return synth.make_batch(_spec(case), seed=seed, device="cuda")


def _logits(case, q_win, k, r, layer, dtype):
    """[Hkv, n, L] scaled window logits of one request and layer, -inf where the causal mask hides a key."""
    lens, w = [int(x) for x in case["lens"].split(",")], case["window"]
    off, length = sum(lens[:r]), lens[r]
    q = q_win[layer, r].reshape(HKV, G * w, D).to(dtype)
    x = torch.bmm(q, k[layer, :, off:off + length].to(dtype).transpose(1, 2)) / math.sqrt(D)
    last = (torch.arange(G * w, device=x.device) % w + (length - w))[:, None]
    return x.masked_fill_(torch.arange(length, device=x.device)[None, :] > last, float("-inf"))


def _mean_std(case, q_win, k, dtype, lse=None, v=None):
    """mu and sigma in the library's packed layout, from a plain softmax; the window rows' output with v."""
    lens, w, n = [int(x) for x in case["lens"].split(",")], case["window"], G * case["window"]
    mus, sigmas, outs = [], [], []
    off = 0
    for r, length in enumerate(lens):
        for layer in range(case["layers"]):
            x = _logits(case, q_win, k, r, layer, dtype)
            if lse is None:
                a = torch.softmax(x, dim=2)
            else:
                a = torch.exp(x - lse[layer, r].reshape(HKV, n, 1).to(dtype))
            del x
            if case["way"] == "perq":
                a = a.reshape(HQ, w, length)
            mus.append(a.mean(dim=1).reshape(-1))
            sigmas.append(a.std(dim=1).reshape(-1))
            if v is not None:
                outs.append(torch.bmm(a, v[layer, :, off:off + length].to(dtype)).reshape(HQ, w, D))
        off += length
    out = None if v is None else torch.stack(outs).reshape(len(lens), case["layers"], HQ, w, D).transpose(0, 1)
    return torch.cat(mus), torch.cat(sigmas), out


class _State:
    pass


def prepare(case, seed):
    s = _State()
    spec = _spec(case)
    batch = _inputs(case, seed)
    s.way = case["way"]
    s.l1, s.l2 = _lambdas(case, seed)
    s.q, s.k, s.v = batch["q_win"], batch["k"], batch["v"]
    strides = {}
    if s.way == "noalloc":
        # the engine's cache is token-major: [N_L][SL][Hkv][d]
        s.k, s.v = (t.permute(0, 2, 1, 3).contiguous().permute(0, 2, 1, 3) for t in (s.k, s.v))
        strides = dict(k_strides=s.k.stride()[:3], v_strides=s.v.stride()[:3])
    s.plan = kv_evict.Plan(spec, spec["seq_lens"], per_query_head=s.way == "perq", **strides)
    s.bufs = kv_evict.Buffers(s.plan, with_trace=False)
    s.k16, s.v16 = (t.view(torch.int16) for t in (s.bufs.k_out, s.bufs.v_out))
    if s.way == "lse":
        s.lse = torch.stack([torch.stack([torch.logsumexp(_logits(case, s.q, s.k, r, layer, torch.float32), dim=2)
                                          .reshape(HQ, case["window"]) for r in range(len(spec["seq_lens"]))])
                             for layer in range(case["layers"])]).contiguous()
    if s.way == "attn":
        s.o_win = torch.empty_like(s.q)
        s.attn_ws = torch.empty(s.plan.score_attn_workspace(), dtype=torch.uint8, device="cuda")
    if s.way == "profiles":
        s.mu, s.sigma, _ = _mean_std(case, s.q, s.k, torch.float32)
        s.indices = torch.empty((case["profiles"], s.plan.n_units, case["budget"]), dtype=torch.int32, device="cuda")
        s.ws = torch.empty(s.plan.select_profiles_workspace(case["profiles"]), dtype=torch.uint8, device="cuda")
    return s


def run(s):
    b, p = s.bufs, s.plan
    if s.way == "profiles":
        p.select_profiles(s.mu, s.sigma, s.k, s.l1, s.l2, s.indices, s.ws)
        return {"indices": s.indices}
    out = {"mu": b.mu, "sigma": b.sigma, "indices": b.indices, "k_out": s.k16, "v_out": s.v16}
    if s.way in ("step", "perq"):
        kv_evict.run_step(p, b, s.q, s.k, s.v, s.l1, s.l2)
    elif s.way == "lse":
        p.score_lse(s.q, s.k, s.lse, b.mu, b.sigma, b.ws)
        p.select_gather(b.mu, b.sigma, s.k, s.v, s.l1, s.l2, b.indices, b.k_out, b.v_out, b.ws)
    elif s.way == "attn":
        p.score_attn(s.q, s.k, s.v, b.mu, b.sigma, s.o_win, b.ws, s.attn_ws)
        p.select_gather(b.mu, b.sigma, s.k, s.v, s.l1, s.l2, b.indices, b.k_out, b.v_out, b.ws)
        out["o_win"] = s.o_win
    elif s.way == "noalloc":
        p.score(s.q, s.k, b.mu, b.sigma, b.ws)
        p.select_noalloc(b.mu, b.sigma, s.k, s.l1, s.l2, b.indices)
        p.gather(s.k, s.v, b.indices, b.k_out, b.v_out)
    else:
        p.score(s.q, s.k, b.mu, b.sigma, b.ws)
        p.select(b.mu, b.sigma, s.k, s.l1, s.l2, b.indices, b.ws)
        return {"mu": b.mu, "sigma": b.sigma, "indices": b.indices}
    return out


def work(case):
    """What one pass cannot do without: K read once, the window rows, mu and sigma, the kept rows read and
    written, one contraction of the window rows with the prefix (and one more for the output)."""
    lens, nl, w, b = [int(x) for x in case["lens"].split(",")], case["layers"], case["window"], case["budget"]
    tokens, uheads = sum(lens), HQ if case["way"] == "perq" else HKV
    units = len(lens) * nl * uheads
    kept = sum(min(b, x - w) + w for x in lens) * nl * uheads
    idx = 4.0 * units * b
    if case["way"] == "profiles":
        pool = sum(min(4 * b, x - w) for x in lens) * nl * uheads
        return {"bytes": 8.0 * nl * uheads * tokens + 2.0 * D * pool + idx * case["profiles"],
                "flops": 2.0 * D * pool * b * case["profiles"]}
    k_bytes = 2.0 * D * nl * HKV * tokens
    rows = 2.0 * D * nl * HQ * w * len(lens)
    nbytes = k_bytes + rows + 8.0 * nl * uheads * tokens + idx
    flops = 2.0 * D * nl * HQ * w * tokens
    if case["way"] == "every":
        return {"bytes": nbytes, "flops": flops}
    nbytes += 2 * 2 * 2.0 * D * kept
    if case["way"] == "lse":
        nbytes += 4.0 * nl * HQ * w * len(lens)
    if case["way"] == "attn":
        nbytes, flops = nbytes + k_bytes + rows, 2 * flops
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    if case["way"] == "attn":
        # the window output is rounded to bf16
        return {"rel": 1e-2, "max": 4e-2, "differ": 1e-2}
    # 32-bit sums of products, exponentials and their squares (2e-7 to 7e-7 off 64 bits; 3.4e-6 where the
    # normalisers are rounded to 32 bits on the way in); near ties of the greedy may fall either way
    return {"rel": 1e-5, "max": 1e-4, "differ": 1e-2}


def exact(case, seed):
    if case["way"] == "profiles":
        return None   # whole numbers only
    batch = _inputs(case, seed)
    q, k = batch["q_win"], batch["k"]
    lse = prepare(case, seed).lse if case["way"] == "lse" else None
    v = batch["v"] if case["way"] == "attn" else None
    mu, sigma, o_win = _mean_std(case, q, k, torch.float64, lse=lse, v=v)
    out = {"mu": mu, "sigma": sigma, "indices": None}
    if case["way"] == "every":
        return out
    out = dict(out, k_out=None, v_out=None)
    return out if o_win is None else dict(out, o_win=o_win.contiguous())
