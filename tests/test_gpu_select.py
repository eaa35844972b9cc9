"""compresskv_select on given raw scores: pooled scores and indices bit by bit
against fp32 arithmetic in the kernel's order (the taps from the left, then one
division) and an exact top-k, on both sides of the lengths between which one
cluster of CTAs per unit pools and selects (up to 4 units: 8192 < n <= 16384; 80
and more: 12000 <= n <= 32768), where a CTA's bound keeps too few or too many
candidates and the search reads what the other CTAs of the cluster pooled (needs
a GB300)."""
import math

import numpy as np
import pytest
import torch

import paper_2606_24467_gb300 as ckv

pytestmark = pytest.mark.gpu

W = 32


def _raw(kind, n, rng):
    if callable(kind):
        return kind(kind, n, rng)
    if kind == "decades":  # scores as attention has them
        return np.exp(2.0 * rng.standard_normal(n)).astype(np.float32)
    if kind == "levels":  # four values: thousands of ties
        return (rng.integers(1, 5, n) * 0.25).astype(np.float32)
    if kind == "equal":
        return np.full(n, 0.37, np.float32)
    x = np.full(n, 1e-6, np.float32)  # few keys above a floor: bounds that keep too few
    x[rng.integers(0, max(n, 1), 40)] = rng.random(40, dtype=np.float32) + 1
    return x


def _pool(raw, P):
    r = (P - 1) // 2
    x = np.concatenate([np.zeros(r, np.float32), raw, np.zeros(r, np.float32)])
    acc = np.zeros(len(raw), np.float32)
    for t in range(P):
        acc = acc + x[t:t + len(raw)]
    return acc / np.float32(P)


def _select(lens, n_kv, P, kind, budgets, dev, pooled_out=True, seed=0):
    rng = np.random.default_rng(seed)
    cu = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    T = int(cu[-1])
    # (select reads the problem's shapes and not the keys)
    k = torch.empty((T, n_kv, 128), dtype=torch.bfloat16, device="meta")
    q = torch.empty((len(lens), n_kv, W, 128), dtype=torch.bfloat16, device="meta")
    prob = ckv.Problem(q, k, cu, W, P)
    n = [max(L - W, 0) for L in lens]
    pre = np.concatenate([[0], np.cumsum(n)])
    raw = np.concatenate([np.concatenate([_raw(kind, m, rng) for m in n])[None]
                          for _ in range(n_kv)])
    budgets = np.asarray(budgets, np.int32)
    kept = np.minimum(budgets, lens)
    out0 = np.concatenate([[0], np.cumsum(kept)])
    indices = torch.full((n_kv, int(out0[-1])), -1, dtype=torch.int32, device=dev)
    pooled = torch.full(raw.shape, -1.0, device=dev) if pooled_out else None
    ws = ckv.workspace(prob, dev)
    cu_out = ckv.select(prob, torch.from_numpy(raw).to(dev), budgets, indices, ws, pooled=pooled)
    torch.cuda.synchronize()
    assert ckv.read_device_status(ws) == 0
    assert cu_out.tolist() == out0.tolist()
    got = indices.cpu().numpy()
    for s, L in enumerate(lens):
        for g in range(n_kv):
            want = _pool(raw[g, pre[s]:pre[s + 1]], P)
            if pooled_out:
                assert np.array_equal(pooled[g, pre[s]:pre[s + 1]].cpu().numpy(), want), (s, g)
            top = int(kept[s]) - min(W, L)
            best = np.sort(np.argsort(-want, kind="stable")[:max(top, 0)])
            sel = np.concatenate([best, np.arange(n[s], L)]) if kept[s] < L else np.arange(L)
            assert np.array_equal(got[g, out0[s]:out0[s + 1]], sel), (s, g)


@pytest.mark.parametrize("n", [8192, 8193, 16001, 16384, 16385])
@pytest.mark.parametrize("P,pooled_out", [(1, True), (7, False), (63, True), (63, False)])
def test_lengths_and_widths(cuda_device, n, P, pooled_out):
    for rest in ([700], [0], [W], [W + 1], [n // 2 + W]):
        _select([n + W, *rest], 2, P, "decades", [512, 300], cuda_device, pooled_out)
    _select([n + W], 1, P, "decades", [W], cuda_device, pooled_out)


@pytest.mark.parametrize("n", [11999, 12000, 32768, 32769])
@pytest.mark.parametrize("P,pooled_out", [(7, True), (63, False)])
def test_many_units(cuda_device, n, P, pooled_out):
    """Clusters of one CTA and of two (slices of 16384 keys and their raw scores
    in shared memory), with short and empty sequences among them."""
    _select([n + W, 0, W + 1, 700, n // 2 + W], 16, P, "decades", [600, 40, 40, 300, 900],
            cuda_device, pooled_out)


@pytest.mark.parametrize("kind", ["levels", "equal", "few"])
@pytest.mark.parametrize("budget", [W + 1, 128, 4096 + W, 9000, 11999])
def test_bounds_that_keep_too_few_or_too_many(cuda_device, kind, budget):
    _select([12000, 10000], 2, 7, kind, [budget, min(budget, 9999)], cuda_device, budget != 128)


def test_second_sampled_bound(cuda_device):
    """Strong scores at eleven of the positions that the first CTA of a cluster
    samples (4 units of 9968 keys: 16 CTAs, slices of 640 keys, 16 evenly
    spaced samples each): the first bound is one of them, fewer than k = 96 keys
    reach it, and a second, looser one is taken."""
    n, n_kv, C, S = 10000 - W, 4, 16, 640
    at = [(t * S) // 16 for t in range(1, 12)]
    samples = []
    for c in range(C):
        lo, hi = min(n, c * S), min(n, (c + 1) * S)
        samples += [lo + (t * (hi - lo)) // 16 for t in range(16)]
    mu = 96 * len(samples) / n
    rank = min(len(samples), math.ceil(mu + 3 * math.sqrt(mu)) + 2)

    def planted(kind, m, rng):
        x = np.exp(rng.standard_normal(m)).astype(np.float32)
        x[at] = 1000.0 + np.arange(11, dtype=np.float32)
        assert (x >= np.sort(x[samples])[::-1][rank - 1]).sum() < 96
        return x

    _select([n + W], n_kv, 1, planted, [96 + W], cuda_device)
