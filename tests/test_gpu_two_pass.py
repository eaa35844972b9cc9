"""The two-pass persistent kernel on layers beyond the resident kernel's line:
row counts that end in half a 32-column block on tiles before the window, odd
numbers of K tiles in a chunk, the given LSE, logits beyond the references'
range, the bounded wait (needs a GB300)."""
import numpy as np
import pytest
import torch

import oracle
import paper_2606_24467_gb300 as ckv
from oracle import compare
from test_gpu_fused import _block, _check_block, _pack, _run_call
from test_gpu_resident import BLOCK_KEYS, _make

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("window,heads,lens,dtype", [
    (16, (1, 1), [49153 + 128 * 5, 129], "bf16"),            # 16 rows
    (16, (3, 3), [49153, 2048 * 3 + 128], "fp16"),           # 48
    (16, (1, 4), [49200, 700], "bf16"),                      # 16 to 64
    (80, (1, 1), [12289 + 128 * 3, 2048 * 2 + 1], "bf16"),   # 80
    (32, (3, 3), [12289, 128 * 3 + 40], "fp16"),             # 96
    (48, (1, 3), [8193 + 40, 128], "bf16"),                  # 48 to 144
    (64, (1, 2), [8193, 65, 0, 64], "bf16"),                 # 64 and 128
    (80, (2, 2), [4097, 2048 + 128 * 5], "fp16"),            # 160
    (64, (3, 3), [2048 * 2 + 128 * 7 + 1, 2049], "bf16"),    # 192
])
def test_rows_and_odd_chunks(cuda_device, window, heads, lens, dtype):
    cfg, layers = _make("c5", lens, n_layers=2, window=window, srh_per_group=heads, dtype=dtype,
                        budget_mean=300)
    out, cu_out, cu = _run_call(layers, cfg, cuda_device)
    for l, lay in enumerate(layers):
        _check_block(_block(out, cu_out, cu, l, cfg.batch, window), lay, cfg)
    again, _, _ = _run_call(layers, cfg, cuda_device)
    alone, cu_out1, cu1 = _run_call(layers[1:], cfg, cuda_device)
    a = _block(alone, cu_out1, cu1, 0, cfg.batch, window)
    b = _block(out, cu_out, cu, 1, cfg.batch, window)
    for key in BLOCK_KEYS:
        assert np.array_equal(a[key], b[key]), key
        if key != "cu_out":
            assert torch.equal(getattr(again, key), getattr(out, key)), key


@pytest.mark.parametrize("window,heads,lens,n_layers", [
    (32, (1, 2), [24577, 300, 0], 1),          # pooled in pieces: few units
    (32, (1, 2), [24577 + 128 * 3], 20),       # ... and more units than SMs
    (64, (3, 3), [6145, 2049], 2),             # 192 rows: pooled by the selection
    (16, (3, 3), [24577 + 128 * 5, 129], 2),   # 48
    (80, (1, 1), [12289, 700], 2),             # 80
])
def test_given_lse(cuda_device, window, heads, lens, n_layers):
    dev = cuda_device
    cfg, layers = _make("c5", lens, n_layers=min(n_layers, 2), window=window, srh_per_group=heads,
                        budget_mean=300)
    layers = (layers * n_layers)[:n_layers]
    lse = torch.cat([torch.tensor(oracle.window_lse(lay["q_win"].float().numpy(),
                                                    lay["k"].float().numpy(), lay["cu_seqlens"],
                                                    window), dtype=torch.float32)
                     for lay in layers[:2]])
    lse = torch.cat([lse] * n_layers)[:n_layers * len(lens)].to(dev)
    q, k, v, cu, b, m = _pack(layers, dev)
    prob = ckv.Problem(q, k, cu, window, cfg.pool_width)
    out = ckv.LayerOutputs(prob, b, 128, k.dtype, dev, scores=True)
    ws = ckv.workspace(prob, dev)
    cu_out = ckv.compress_layers_lse(prob, n_layers, q, k, v, lse, m, b, out.indices, out.k_out,
                                     out.v_out, ws, raw=out.raw, pooled=out.pooled)
    torch.cuda.synchronize()
    assert ckv.read_device_status(ws) == 0
    blocks = [_block(out, cu_out, cu, l, cfg.batch, window) for l in range(n_layers)]
    for l in range(min(n_layers, 2)):
        _check_block(blocks[l], layers[l], cfg)
    for l in range(2, n_layers):  # the same layers again
        for key in BLOCK_KEYS:
            assert np.array_equal(blocks[l][key], blocks[l % 2][key]), key


@pytest.mark.parametrize("window,heads,lens", [(32, (1, 2), [49153, 700]),
                                               (64, (3, 3), [4200, 300])])
@pytest.mark.parametrize("shift", [-90.0, 90.0])
def test_logits_beyond_the_references(cuda_device, window, heads, lens, shift):
    """Every other window row's logits moved by about `shift`, and the keys of
    the second half of each chunk's tiles larger than those before: sums pass
    2^64 against their first reference, which is raised.  Bound: as in
    test_sums_outside_the_fixed_point_bins."""
    cfg, layers = _make("c5", lens, n_layers=1, window=window, srh_per_group=heads,
                        budget_mean=200)
    lay = layers[0]
    u = torch.sign(torch.randn(128, generator=torch.Generator().manual_seed(7)))
    dt = lay["k"].dtype
    grow = (torch.arange(lay["k"].shape[0]) // 1024 % 2)[:, None, None]
    lay["k"] = (lay["k"].float() + (1.0 + grow) * u).to(dt)
    q = lay["q_win"].float()
    q[:, :, ::2] += shift * 128 ** 0.5 / 256.0 * u
    lay["q_win"] = q.to(dt)
    out, cu_out, cu = _run_call(layers, cfg, cuda_device)
    blk = _block(out, cu_out, cu, 0, cfg.batch, window)
    res = oracle.compress_layer(lay["q_win"].float().numpy(), lay["k"].float().numpy(),
                                lay["v"].float().numpy(), lay["cu_seqlens"], lay["srh_mask"],
                                lay["budgets"], window, cfg.pool_width)
    norms = lay["q_win"].float().norm(dim=-1).max() * lay["k"].float().norm(dim=-1).max()
    rtol = 2 * 10 * 2.0 ** -23 * float(norms) / 128 ** 0.5 + 1e-5
    compare.check_scores("raw", blk["raw"], res.raw, rtol=rtol, atol=1e-8)
    compare.check_scores("pooled", blk["pooled"], res.pooled, rtol=rtol, atol=1e-8)


def test_bounded_wait_runs_out(cuda_device):
    """As test_bounded_wait_runs_out_and_the_workspace_recovers, for this
    kernel: the status of the stopped call, and the same workspace after
    workspace_init."""
    dev = cuda_device
    cfg, layers = _make("c5", [4500, 8000], n_layers=2, window=64, srh_per_group=(3, 3),
                        budget_mean=300)
    want, cu_out, cu = _run_call(layers, cfg, dev)
    _check_block(_block(want, cu_out, cu, 1, cfg.batch, cfg.window), layers[1], cfg)
    q, k, v, cu, b, m = _pack(layers, dev)
    prob = ckv.Problem(q, k, cu, cfg.window, cfg.pool_width)
    out = ckv.LayerOutputs(prob, b, 128, k.dtype, dev, scores=True)
    ws = ckv.workspace(prob, dev)

    def call():
        ckv.compress_layers(prob, len(layers), q, k, v, m, b, out.indices, out.k_out, out.v_out,
                            ws, raw=out.raw, pooled=out.pooled)
        torch.cuda.synchronize()
        return ckv.read_device_status(ws)

    ckv.debug_stall_next_fused_call(2_000_000)
    assert call() == ckv.compresskv.CKV_ERR_DEVICE_TIMEOUT
    ckv.compresskv._check(ckv.load().compresskv_workspace_init(ckv.compresskv._ptr(ws), ws.numel(),
                                                               None), "workspace_init")
    assert call() == 0
    for key in ("raw", "pooled", "indices", "k_out", "v_out"):
        assert torch.equal(getattr(out, key), getattr(want, key)), key
