"""Pool sizes at the edges of the selector's greedy: one half of 128 slots and two, a slot short of a
half and one past it, the largest pool whose dot products stand before the greedy (256) and the smallest
beyond it; equal scores and repeated keys, whose ties go to the lower position; and the every-candidate
selector's candidate counts around its warps' 32 rows and its block's 512, with both signs of lambda2;
very small, very large and zero keys.
Every admission is replayed through the oracle, margins included."""

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


def _check(L, B, factor, lam2, seed, flat=False, scale=1.0, dims=None):
    """Selection on given mu and sigma (flat: few distinct values, runs of equal keys; scale: of the keys; dims:
    the keys' first elements alone, at norm 1)."""
    from paper_2609_30738_gb300 import kv_evict as K
    W, nl, hkv = 8, 2, 2
    spec = scaled(WORKLOADS["mistral-1layer-L2048"], num_layers=nl, num_q_heads=4, num_kv_heads=hkv, window=W,
                  budget=B, candidate_factor=factor, seq_lens=[L])
    batch = synth.make_batch(spec, seed=seed, with_values=False)
    rng = np.random.default_rng(seed)
    mu = rng.random(nl * hkv * L).astype(np.float32) ** 4
    sigma = rng.random(nl * hkv * L).astype(np.float32) ** 4
    if flat:
        mu, sigma = np.round(mu * 2) / 2 + np.float32(0.25), np.round(sigma * 2) / 2
        batch["k"][:, :, 1::2] = batch["k"][:, :, 0:1]      # every other key is one and the same
    mu, sigma = mu.astype(np.float32), sigma.astype(np.float32)
    if dims:
        head = batch["k"][..., :dims].float()
        batch["k"].zero_()
        batch["k"][..., :dims] = head / head.norm(dim=-1, keepdim=True)
    if scale != 1.0:
        batch["k"] *= scale
        batch["k"][:, :, 5::7] = 0
    plan = K.Plan(spec, [L])
    bufs = K.Buffers(plan)
    bufs.mu.copy_(torch.from_numpy(mu))
    bufs.sigma.copy_(torch.from_numpy(sigma))
    bufs.ws.zero_()
    l1, l2 = np.full(nl, 0.5, np.float32), np.full(nl, lam2, np.float32)
    plan.select(bufs.mu, bufs.sigma, batch["k"].cuda(), l1, l2, bufs.indices, bufs.ws, bufs.order, bufs.margins)
    assert plan.status(bufs.ws) == K.KVE_OK
    order, indices = bufs.order.cpu().numpy(), bufs.indices.cpu().numpy()
    margins = bufs.margins.cpu().numpy()
    for u in range(nl * hkv):
        keys = O.bf16_bits_to_f64(PT.to_bits(batch["k"][u // hkv, u % hkv]))
        m64, s64 = mu[u * L:(u + 1) * L].astype(np.float64), sigma[u * L:(u + 1) * L].astype(np.float64)
        PT.check_selection(order[u], indices[u], m64, s64, keys, L, W, B, 0.5, lam2, candidate_factor=factor,
                           margins_gpu=margins[u])


@pytest.mark.parametrize("lam2", [-0.5, 0.6, 0.0])
@pytest.mark.parametrize("B,factor", [(127, 1), (64, 2), (43, 3), (51, 5), (64, 4), (257, 1)])
def test_pool_edges(B, factor, lam2):
    _check(1500, B, factor, lam2, seed=B)


@pytest.mark.parametrize("lam2", [-0.5, 0.0])
@pytest.mark.parametrize("L,B,factor", [(600, 32, 4), (600, 60, 4), (1500, 80, 4)])
def test_pool_ties(L, B, factor, lam2):
    _check(L, B, factor, lam2, seed=L + B, flat=True)


@pytest.mark.parametrize("lam2", [-0.5, 0.6])
@pytest.mark.parametrize("Lc", [513, 1023, 1025, 1056, 2081])
def test_every_candidate_edges(Lc, lam2):
    _check(Lc + 8, 24, 0, lam2, seed=Lc)


@pytest.mark.parametrize("B", [30, 60])
@pytest.mark.parametrize("scale", [2.0 ** -40, 2.0 ** -31, 2.0 ** 58])
def test_pool_key_scales(scale, B):
    """Squared norms below, around and above the range in which they are read from the dots; zero keys."""
    _check(700, B, 4, -0.5, seed=B, scale=scale)


@pytest.mark.parametrize("B", [30, 60])
@pytest.mark.parametrize("dims,scale", [(8, 2.0 ** -64.75), (None, 2.0 ** 60)])
def test_pool_key_scales_at_the_ends(dims, scale, B):
    """Norms whose inverses' product leaves the floats' range (every norm 2^-64.75), and norms near the
    largest whose squares still sum. At the small end a product of two elements keeps multiples of 2^-149:
    8 of them truncated move a dot by at most 2^-146, and rounded a squared norm by 2^-147, so that a cosine
    moves by (2^-146 + 2^-147) / 2^-129.5 = 1.6e-5 and two values' difference (lambda2 = -0.5) by as much:
    below the replay's 1e-4."""
    _check(700, B, 4, -0.5, seed=B, scale=scale, dims=dims)


@pytest.mark.parametrize("lam2", [-0.5, 0.6])
@pytest.mark.parametrize("Lc", [240, 500, 600, 2081])
def test_masked_tokens_come_last(Lc, lam2):
    """Tokens masked by mu = -inf, with fewer others than the budget: the others first, then the masked ones
    from the lowest position up, in each of the three selectors."""
    from paper_2609_30738_gb300 import kv_evict as K
    W, B = 8, 24
    spec = scaled(WORKLOADS["mistral-1layer-L2048"], num_layers=1, num_q_heads=4, num_kv_heads=1, window=W,
                  budget=B, candidate_factor=0, pool_kernel=1, seq_lens=[Lc + W])
    batch = synth.make_batch(spec, seed=Lc, with_values=False)
    rng = np.random.default_rng(Lc)
    kept = rng.choice(np.arange(3, Lc), size=10, replace=False)
    mu = np.full(Lc + W, -np.inf, np.float32)
    mu[kept] = rng.random(10).astype(np.float32) + 0.5
    plan = K.Plan(spec, [Lc + W])
    bufs = K.Buffers(plan)
    bufs.mu.copy_(torch.from_numpy(mu))
    bufs.sigma.fill_(0.25)
    bufs.ws.zero_()
    l1, l2 = np.full(1, 0.5, np.float32), np.full(1, lam2, np.float32)
    for margins in (bufs.margins, None):
        plan.select(bufs.mu, bufs.sigma, batch["k"].cuda(), l1, l2, bufs.indices, bufs.ws, bufs.order, margins)
        assert plan.status(bufs.ws) == K.KVE_OK
        order = bufs.order.cpu().numpy()[0]
        assert set(order[:10]) == set(kept)
        assert list(order[10:]) == [p for p in range(Lc) if p not in set(kept)][:B - 10]
        assert np.array_equal(bufs.indices.cpu().numpy()[0], np.sort(order))
