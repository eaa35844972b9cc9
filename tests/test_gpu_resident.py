"""The persistent kernel for short prompts (logits kept in tensor memory) and
the line between it and the two-pass kernel, against the float64 oracle (needs
a GB300)."""
import numpy as np
import pytest
import torch

import oracle
import paper_2606_24467_gb300 as ckv
import workloads as wl
from oracle import compare
from test_gpu_fused import _block, _check_block, _pack, _run_call

pytestmark = pytest.mark.gpu

BLOCK_KEYS = ("raw", "pooled", "indices", "k_out", "v_out", "cu_out")


def _make(name, lens, **over):
    cfg = wl.get(name).scaled(seq_len=0, batch=len(lens), **over)
    masks = wl.srh_masks(cfg)
    budgets = wl.layer_budgets(cfg, lens)
    return cfg, [wl.make_layer(cfg, l, lengths=lens, masks=masks, budgets=budgets)
                 for l in range(cfg.n_layers)]


@pytest.mark.parametrize("window,heads,lens", [
    # tile edges in chunks of one tile (layers of at most 64 tiles), of two
    # (at most 256) and of four
    (16, (1, 1), [17, 127, 128, 129]),
    (32, (1, 2), [129, 600, 1153]),
    # the longest prompt whose scores the selection holds in shared memory
    # (6144 keys before the window)
    (16, (1, 1), [513, 4096, 4097, 6160, 6161, 8193]),
    # 32 and 64 rows: the line of both, from either side
    (32, (1, 2), [33, 16384, 49152]),
    (32, (1, 2), [33, 49153]),
    # pooling in pieces of 6144 keys (few units, a prompt above 12288), the last
    # of one key and of one row
    (16, (1, 1), [2 * 6144 + 17, 2 * 6144 + 48, 6160]),
    # 64, 128 and 192 rows in one call, 64 and 128, 32 to 96: their lines
    (64, (1, 3), [65, 4096]),
    (64, (1, 3), [65, 4097]),
    (64, (1, 2), [65, 8192]),
    (64, (1, 2), [65, 8193]),
    (32, (1, 3), [65, 12288]),
])
def test_sizes_around_tiles_chunks_and_the_kernels_line(cuda_device, window, heads, lens):
    cfg, layers = _make("c5", lens, n_layers=2, window=window, srh_per_group=heads,
                        budget_mean=300)
    big, cu_out, cu = _run_call(layers, cfg, cuda_device)
    for l, lay in enumerate(layers):
        _check_block(_block(big, cu_out, cu, l, cfg.batch, window), lay, cfg)
    alone, cu_out1, cu1 = _run_call(layers[1:], cfg, cuda_device)
    a = _block(alone, cu_out1, cu1, 0, cfg.batch, window)
    b = _block(big, cu_out, cu, 1, cfg.batch, window)
    for key in BLOCK_KEYS:
        assert np.array_equal(a[key], b[key]), key


@pytest.mark.parametrize("shift", [-90.0, 90.0])
def test_sums_outside_the_fixed_point_bins(cuda_device, shift):
    """Every other window row's logits moved by about `shift`: its sums of
    exponentials leave the range of the accumulators' bins, so it takes the
    second round; its neighbours don't.

    Bound: a logit is eight accumulations of at most |q| |k| in fp32, scaled
    once and rounded once against the exponent's reference, so off by at most
    10 ulp of |q| |k| / sqrt(d); a score is a ratio of two exponentials of it."""
    cfg, layers = _make("c2", [700, 5000], n_layers=1, srh_per_group=(1, 2), budget_mean=200)
    lay = layers[0]
    u = torch.sign(torch.randn(128, generator=torch.Generator().manual_seed(7)))
    dt = lay["k"].dtype
    lay["k"] = (lay["k"].float() + 2.0 * u).to(dt)
    q = lay["q_win"].float()
    q[:, :, ::2] += shift * 128 ** 0.5 / 256.0 * u
    lay["q_win"] = q.to(dt)
    out, cu_out, cu = _run_call(layers, cfg, cuda_device)
    blk = _block(out, cu_out, cu, 0, cfg.batch, cfg.window)
    res = oracle.compress_layer(lay["q_win"].float().numpy(), lay["k"].float().numpy(),
                                lay["v"].float().numpy(), lay["cu_seqlens"], lay["srh_mask"],
                                lay["budgets"], cfg.window, cfg.pool_width)
    norms = lay["q_win"].float().norm(dim=-1).max() * lay["k"].float().norm(dim=-1).max()
    rtol = 2 * 10 * 2.0 ** -23 * float(norms) / 128 ** 0.5 + 1e-5
    compare.check_scores("raw", blk["raw"], res.raw, rtol=rtol, atol=1e-8)
    compare.check_scores("pooled", blk["pooled"], res.pooled, rtol=rtol, atol=1e-8)


def test_chunk_sums_lose_no_bits(cuda_device):
    """Units whose keys are all alike: every chunk's sum of exponentials is a
    power of two times one exponential, just above a power of two at which the
    accumulators' bins could begin (2^24 for a unit of 20 chunks), so each
    score is 2^(z c) over an exactly known count of the same, however large.

    Bound: what remains is the rounding of D and of its reciprocal, of the
    product with it and of the sums over 16 rows, some six of at most 2^-24
    each and independent over the units: an rms below sqrt(6) 2^-24 =
    1.5e-7.  Sums kept to 20 bits are off by up to 8 / S, 2.3e-7 rms."""
    dev = cuda_device
    n_layers, n_kv, window, L, d = 64, 2, 16, 2560, 128
    scale = float(np.float32(0.125 / np.log2(np.e)))
    assert np.float32(scale * np.log2(np.e)) == 0.125  # z c exact
    k = torch.ones((n_layers * L, n_kv, d), dtype=torch.bfloat16, device=dev)
    q = torch.full((n_layers, n_kv, window, d), 1.0, dtype=torch.bfloat16, device=dev)
    frac = torch.arange(n_layers * n_kv, device=dev).view(n_layers, n_kv, 1) / 64.0
    q[..., 0] = 136.0 - 127.0 + 0.0  # z = 136 and a fraction, z c = 17 and up
    q[..., 1] = 1.0 + (frac % 1.0).to(torch.bfloat16)
    q[..., 2] = 1.0 + torch.floor(frac).to(torch.bfloat16) / 128.0
    z = q[:, :, 0].double().sum(-1)
    assert float(z.min()) >= 17 * 8 and float(z.max()) < 17.3 * 8
    cu = np.arange(n_layers + 1, dtype=np.int32) * L
    budgets = np.full(n_layers, window + 1, np.int32)
    prob = ckv.Problem(q, k, cu, window, 7, scale=scale)
    out = ckv.LayerOutputs(prob, budgets, d, k.dtype, dev, scores=True)
    ws = ckv.workspace(prob, dev)
    ckv.compress_layers(prob, n_layers, q, k, k, np.ones((n_layers, n_kv), np.uint8), budgets,
                        out.indices, out.k_out, out.v_out, ws, raw=out.raw, pooled=out.pooled)
    torch.cuda.synchronize()
    assert ckv.read_device_status(ws) == 0
    n = L - window
    want = sum(1.0 / (n + w + 1) for w in range(window))
    err = out.raw.double().view(n_kv, n_layers, n) / want - 1.0
    assert float(err.pow(2).mean().sqrt()) < 1.5e-7


@pytest.mark.parametrize("dtype,n,bias", [(torch.bfloat16, 8000, 0.8e-7),
                                          (torch.bfloat16, 26000, 0.8e-7),
                                          (torch.float16, 8000, 1.6e-7),
                                          (torch.float16, 26000, 1.6e-7)])
def test_truncated_logits_are_made_up_for(cuda_device, dtype, n, bias):
    """Given-LSE scores with LSE = 0 and W equal query rows are W e^z: the mean
    of (log(score / W) - z) / z over keys along the query, |z| from 3 to 9, in
    the resident (n <= 24576) and in the two-pass kernel.  The tensor cores'
    truncated sums alone give -1.2e-7 (bf16) and -2.0e-7 (f16); bound: half a
    unit of the fp32 scale's last place (0.6e-7) beside what the types differ
    from the mean correction."""
    dev, d, window, heads = cuda_device, 128, 16, 8
    gen = torch.Generator(device=dev)
    gen.manual_seed(3)
    q1 = 1.5 * torch.randn((1, heads, 1, d), generator=gen, device=dev)
    q = q1.expand(1, heads, window, d).contiguous().to(dtype)
    norm = q1[0, :, 0].norm(dim=-1, keepdim=True)
    along = torch.linspace(-9, 9, n + window, device=dev)[:, None, None] * (d ** 0.5 / norm)
    k = 0.5 * torch.randn((n + window, heads, d), generator=gen, device=dev)
    k = (k + along * (q1[0, :, 0] / norm)).to(dtype)
    budgets = np.array([window + 64], np.int32)
    prob = ckv.Problem(q, k, np.array([0, n + window], np.int32), window, 7)
    out = ckv.LayerOutputs(prob, budgets, d, dtype, dev, scores=True)
    ws = ckv.workspace(prob, dev)
    ckv.compress_layer_lse(prob, q, k, k, torch.zeros((1, heads, window), device=dev),
                           np.ones(heads, np.uint8), budgets, out.indices, out.k_out, out.v_out,
                           ws, raw=out.raw, pooled=out.pooled)
    torch.cuda.synchronize()
    assert ckv.read_device_status(ws) == 0
    z = torch.einsum("nhd,hd->hn", k[:n].double(), q[0, :, 0].double()) / d ** 0.5
    err = (torch.log(out.raw.double() / window) - z) / z
    assert abs(float(err[(z.abs() > 3) & (z.abs() < 9)].mean())) < bias


def test_calls_on_two_streams_at_once(cuda_device):
    """Two calls in flight on two streams with a workspace each (every one
    needs all its CTAs resident): the bits of the calls made one by one."""
    dev = cuda_device
    runs = []
    for seed, lens in enumerate(([1500, 3000], [900, 49153])):
        cfg, layers = _make("c2", lens, n_layers=2 + seed, budget_mean=200)
        want, _, _ = _run_call(layers, cfg, dev)
        q, k, v, cu, b, m = _pack(layers, dev)
        prob = ckv.Problem(q, k, cu, cfg.window, cfg.pool_width)
        out = ckv.LayerOutputs(prob, b, 128, k.dtype, dev, scores=True)
        runs.append((len(layers), prob, q, k, v, m, b, out, ckv.workspace(prob, dev), want,
                     torch.cuda.Stream()))
    torch.cuda.synchronize()
    for _ in range(10):
        for n, prob, q, k, v, m, b, out, ws, _, stream in runs:
            with torch.cuda.stream(stream):
                ckv.compress_layers(prob, n, q, k, v, m, b, out.indices, out.k_out, out.v_out, ws,
                                    raw=out.raw, pooled=out.pooled)
    torch.cuda.synchronize()
    for _, _, _, _, _, _, _, out, ws, want, _ in runs:
        assert ckv.read_device_status(ws) == 0
        for key in ("raw", "pooled", "indices", "k_out", "v_out"):
            assert torch.equal(getattr(out, key), getattr(want, key)), key


def test_layers_on_both_sides_of_the_line(cuda_device):
    """Layers of 64 and of 96 query rows at a length that the resident kernel
    takes for the former only: one call launches both kernels, and every layer
    has the bits of a call of its own (and, without scores, of the call without
    a workspace)."""
    dev = cuda_device
    lens = [13000, 0, 40, 32, 700]
    cfg = wl.get("c2").scaled(seq_len=0, n_layers=4, batch=len(lens), budget_mean=300)
    two = np.asarray(wl.srh_masks(cfg.scaled(srh_per_group=(2, 2))))
    three = np.asarray(wl.srh_masks(cfg.scaled(srh_per_group=(3, 3))))
    masks = np.stack([two[0], three[1], three[2], two[3]])
    budgets = wl.layer_budgets(cfg, lens)
    layers = [wl.make_layer(cfg, l, lengths=lens, masks=masks, budgets=budgets) for l in range(4)]
    big, cu_out, cu = _run_call(layers, cfg, dev)
    for l, lay in enumerate(layers):
        b = _block(big, cu_out, cu, l, cfg.batch, cfg.window)
        if l < 2:
            _check_block(b, lay, cfg)
        alone, cu_out1, cu1 = _run_call([lay], cfg, dev)
        a = _block(alone, cu_out1, cu1, 0, cfg.batch, cfg.window)
        for key in BLOCK_KEYS:
            assert np.array_equal(a[key], b[key]), (l, key)
    q, k, v, cu, b, m = _pack(layers, dev)
    trace = ckv.Trace(8)
    prob = ckv.Problem(q, k, cu, cfg.window, cfg.pool_width, trace=trace)
    out = ckv.LayerOutputs(prob, b, 128, k.dtype, dev, scores=False)
    ws = ckv.workspace(prob, dev)
    ckv.compress_layers(prob, 4, q, k, v, m, b, out.indices, out.k_out, out.v_out, ws)
    torch.cuda.synchronize()
    assert ckv.read_device_status(ws) == 0
    assert trace.struct.launches == 2
    assert torch.equal(out.indices, big.indices)
    prob = ckv.Problem(q, k, cu, cfg.window, cfg.pool_width)
    for _ in range(10):  # without the trace's events the two kernels overlap
        out.indices.zero_()
        out.k_out.zero_()
        ckv.compress_layers(prob, 4, q, k, v, m, b, out.indices, out.k_out, out.v_out, ws)
        torch.cuda.synchronize()
        assert ckv.read_device_status(ws) == 0
        assert torch.equal(out.indices, big.indices)
        assert torch.equal(out.k_out, big.k_out) and torch.equal(out.v_out, big.v_out)
    for l in (0, 1):
        one = layers[l]
        q, k, v = (one[x].to(dev) for x in ("q_win", "k", "v"))
        prob = ckv.Problem(q, k, np.asarray(one["cu_seqlens"], np.int32), cfg.window, cfg.pool_width)
        if ckv.workspace_size(prob) <= ckv.compresskv.STATIC_SCRATCH_BYTES:
            out = ckv.LayerOutputs(prob, one["budgets"], 128, k.dtype, dev, scores=True)
            ckv.compress_layer_noalloc(prob, q, k, v, masks[l], one["budgets"], out.indices,
                                       out.k_out, out.v_out, raw=out.raw, pooled=out.pooled)
            torch.cuda.synchronize()
            got = _block(out, np.concatenate([[0], np.cumsum(np.minimum(one["budgets"], lens))]),
                         np.asarray(one["cu_seqlens"]), 0, cfg.batch, cfg.window)
            want = _block(big, cu_out, cu, l, cfg.batch, cfg.window)
            for key in ("raw", "pooled", "indices", "k_out", "v_out"):
                assert np.array_equal(got[key], want[key]), (l, key)


def test_static_scratch_without_the_resident_area(cuda_device):
    """Many tiny units: the workspace is larger than the static scratch, which
    has no room for all units' sums, so the call without a workspace makes
    several launches: the same bits."""
    dev = cuda_device
    cfg, layers = _make("c2", [20] * 512, n_layers=1, num_q_heads=32, num_kv_heads=32, window=16,
                        srh_per_group=(1, 1), budget_mean=18)
    want, _, _ = _run_call(layers, cfg, dev)
    q, k, v, cu, b, m = _pack(layers, dev)
    prob = ckv.Problem(q, k, cu, cfg.window, cfg.pool_width)
    assert ckv.workspace_size(prob) > ckv.compresskv.STATIC_SCRATCH_BYTES
    out = ckv.LayerOutputs(prob, b, 128, k.dtype, dev, scores=True)
    status = torch.full((1,), -1, dtype=torch.int32, device=dev)
    ckv.compress_layer_noalloc(prob, q, k, v, m[0], b, out.indices, out.k_out, out.v_out,
                               raw=out.raw, pooled=out.pooled, device_status=status)
    torch.cuda.synchronize()
    assert int(status) == 0
    assert torch.equal(out.raw, want.raw) and torch.equal(out.pooled, want.pooled)
    assert torch.equal(out.indices, want.indices) and torch.equal(out.k_out, want.k_out)
