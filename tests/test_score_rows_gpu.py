"""mu and sigma at every number of window rows that takes another path of the score kernel: up to 32
rows (keys on the lanes in both passes), up to 64 and up to 128, whole 32-row blocks and not, and the
per-query-head plans that take a KV head's four query heads in one unit. Lengths at the tile edges: a
single candidate, one key past a tile, window keys across two tiles, calls of few tiles (one tile per
item) and many (items of several tiles, several rounds)."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import kv_evict_oracle as O
from paper_2609_30738_gb300 import synth
from paper_2609_30738_gb300.workloads import WORKLOADS, scaled
from tests import parity as PT

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2609_30738_gb300 import kv_evict
    kv_evict.library()


def _check(spec, per_query_head, seed, zero_q=False, sigma_mu_floor=0.0):
    from paper_2609_30738_gb300 import kv_evict as K
    batch = synth.make_batch(spec, seed=seed, with_values=False)
    if zero_q:
        batch["q_win"].zero_()
    lens = batch["seq_lens"]
    plan = K.Plan(spec, lens, per_query_head=per_query_head)
    bufs = K.Buffers(plan)
    bufs.mu.fill_(float("nan"))
    bufs.sigma.fill_(float("nan"))
    plan.score(batch["q_win"].cuda(), batch["k"].cuda(), bufs.mu, bufs.sigma, bufs.ws)
    assert plan.status(bufs.ws) == K.KVE_OK
    mu, sigma = bufs.mu.cpu().numpy(), bufs.sigma.cpu().numpy()
    hq, hkv, W, nl = spec["num_q_heads"], spec["num_kv_heads"], spec["window"], spec["num_layers"]
    G = hq // hkv
    heads = hq if per_query_head else hkv
    q_bits, k_bits = PT.to_bits(batch["q_win"]), PT.to_bits(batch["k"])
    off = 0
    for r, L in enumerate(lens):
        for layer in range(nl):
            for h in range(heads):
                kv = h // G if per_query_head else h
                q, k = O.unit_slices(q_bits, k_bits, lens, r, layer, kv, hkv, W)
                if per_query_head:
                    q = q[(h % G) * W:(h % G + 1) * W]
                ref = O.score_unit(O.bf16_bits_to_f64(q), O.bf16_bits_to_f64(k), L, W, 1 if per_query_head else G)
                at = nl * heads * off + (layer * heads + h) * L
                PT.check_mu_sigma(mu[at:at + L], sigma[at:at + L], *ref, sigma_mu_floor=sigma_mu_floor)
        off += L


@pytest.mark.parametrize("per_query_head", [False, True])
@pytest.mark.parametrize("W", [1, 5, 8, 12, 16, 24, 32])
def test_window_rows(W, per_query_head):
    base = scaled(WORKLOADS["mistral-1layer-L2048"], window=W, budget=8, num_q_heads=8, num_kv_heads=2)
    _check(scaled(base, num_layers=1, seq_lens=[W + 1, 129, 128 + W // 2 + 1, 261, 1100]), per_query_head, 41)


@pytest.mark.parametrize("W,per_query_head", [(8, False), (16, False), (8, True), (32, True)])
def test_window_rows_many_items(W, per_query_head):
    base = scaled(WORKLOADS["mistral-1layer-L2048"], window=W, budget=8, num_q_heads=8, num_kv_heads=2)
    _check(scaled(base, num_layers=8, seq_lens=[9000, 2333]), per_query_head, 42)


@pytest.mark.parametrize("W,per_query_head", [(8, False), (16, False), (32, False), (8, True), (32, True)])
def test_equal_rows_take_the_exact_form(W, per_query_head):
    # zero queries: A = 1 / (visible keys), sigma / mu ~ W / L, the one-pass form cannot hold sigma
    # (the mu-proportional floor of tests/parity.py's derivation: 1e-4 mu)
    base = scaled(WORKLOADS["mistral-1layer-L2048"], window=W, budget=8, num_q_heads=8, num_kv_heads=2)
    _check(scaled(base, num_layers=1, seq_lens=[300, 1500]), per_query_head, 43, zero_q=True, sigma_mu_floor=1e-4)


@pytest.mark.parametrize("layers,L", [(12, 1500), (2, 9400), (3, 5000)])
def test_calls_of_few_tiles(layers, L):
    # items cut by the busiest CTA's load, on 152 CTAs: 288 and 304 items (two rounds), 144 (one)
    _check(scaled(WORKLOADS["mistral-1layer-L2048"], num_layers=layers, seq_lens=[L], budget=8), False, 44)
