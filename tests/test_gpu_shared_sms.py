"""The resident kernel where it does not get every SM: on a green context's
share, and while another kernel holds SMs.  Its results are the bits of the
call that has the GPU to itself (needs a GB300)."""
import ctypes
import time

import numpy as np
import pytest
import torch

import paper_2606_24467_gb300 as ckv
import workloads as wl
from test_gpu_fused import _pack
from test_gpu_resident import _make

pytestmark = pytest.mark.gpu

SM = 1  # CU_DEV_RESOURCE_TYPE_SM


class GreenStream:
    """A stream of a green context of at least n SMs."""

    def __init__(self, n):
        cu = ctypes.CDLL("libcuda.so.1")
        torch.zeros(1, device="cuda")

        def call(name, *args):
            rc = getattr(cu, name)(*args)
            if rc != 0:
                raise RuntimeError(f"{name}: {rc}")

        dev = ctypes.c_int()
        call("cuDeviceGet", ctypes.byref(dev), torch.cuda.current_device())
        whole, part, rest = (ctypes.create_string_buffer(512) for _ in range(3))
        call("cuDeviceGetDevResource", dev, whole, SM)
        groups = ctypes.c_uint(1)
        call("cuDevSmResourceSplitByCount", part, ctypes.byref(groups), whole, rest,
             ctypes.c_uint(0), ctypes.c_uint(n))
        # (type, 92 bytes, then the SM count)
        self.sms = ctypes.c_uint.from_buffer(part, 96).value
        desc, self._ctx, self._stream = ctypes.c_void_p(), ctypes.c_void_p(), ctypes.c_void_p()
        call("cuDevResourceGenerateDesc", ctypes.byref(desc), part, ctypes.c_uint(1))
        call("cuGreenCtxCreate", ctypes.byref(self._ctx), desc, dev, ctypes.c_uint(1))
        call("cuGreenCtxStreamCreate", ctypes.byref(self._stream), self._ctx, ctypes.c_uint(1),
             ctypes.c_int(0))
        self.stream = torch.cuda.ExternalStream(self._stream.value)


@pytest.fixture(scope="module")
def green():
    made = {}

    def get(n):
        if n not in made:
            try:
                made[n] = GreenStream(n)
            except (OSError, AttributeError, RuntimeError) as e:
                pytest.skip(f"no green contexts here: {e}")
        return made[n]

    return get


class Call:
    """compress_layers with its inputs, outputs and workspace."""

    def __init__(self, layers, cfg, dev, lse=None):
        self.q, self.k, self.v, cu, self.b, self.m = _pack(layers, dev)
        self.prob = ckv.Problem(self.q, self.k, cu, cfg.window, cfg.pool_width)
        self.out = ckv.LayerOutputs(self.prob, self.b, 128, self.k.dtype, dev, scores=True)
        self.ws = ckv.workspace(self.prob, dev)
        self.lse = lse
        torch.cuda.synchronize()

    def run(self, stream=None):
        o = self.out
        for t in (o.raw, o.pooled, o.indices):
            t.zero_()
        o.k_out.zero_()
        torch.cuda.synchronize()
        args = (o.indices, o.k_out, o.v_out, self.ws)
        kw = dict(raw=o.raw, pooled=o.pooled, stream=stream)
        if self.lse is None:
            ckv.compress_layers(self.prob, len(self.m), self.q, self.k, self.v, self.m, self.b,
                                *args, **kw)
        else:
            ckv.compress_layers_lse(self.prob, len(self.m), self.q, self.k, self.v, self.lse,
                                    self.m, self.b, *args, **kw)

    def result(self):
        torch.cuda.synchronize()
        assert ckv.read_device_status(self.ws) == 0
        o = self.out
        return [t.clone() for t in (o.raw, o.pooled, o.indices, o.k_out.view(torch.int16),
                                    o.v_out.view(torch.int16))]


def _same(a, b):
    for x, y in zip(a, b):
        assert torch.equal(x, y)


def _case(name, dev):
    if name == "wide":  # 64 to 192 rows, 1 to 32 chunks
        cfg, layers = _make("c5", [65, 4096, 0, 2000], n_layers=2, window=64,
                            srh_per_group=(1, 3), budget_mean=300)
    else:  # 32 and 64 rows, up to 96 chunks of four tiles
        cfg, layers = _make("c2", [49152, 33, 700], n_layers=2, srh_per_group=(1, 2),
                            budget_mean=300)
        if name == "large_logits":  # sums of every other row take the second round
            u = torch.sign(torch.randn(128, generator=torch.Generator().manual_seed(7)))
            for lay in layers:
                lay["k"] = (lay["k"].float() + 2.0 * u).to(lay["k"].dtype)
                q = lay["q_win"].float()
                q[:, :, ::2] += 90.0 * 128 ** 0.5 / 256.0 * u
                lay["q_win"] = q.to(lay["q_win"].dtype)
    lse = None
    if name == "lse":
        cfg, layers = _make("c2", [20000, 33], n_layers=2, srh_per_group=(1, 2), budget_mean=300)
        lse = torch.full((2 * 2, cfg.num_q_heads, cfg.window), 9.0, device=dev)
    return Call(layers, cfg, dev, lse)


@pytest.mark.parametrize("name", ["long", "wide", "large_logits", "lse"])
@pytest.mark.parametrize("sms", [120, 64, 32, 8])
def test_on_a_share_of_the_sms(cuda_device, green, name, sms):
    """A green context's stream: on few SMs a unit's logits do not fit tensor
    memory at once and K is read twice."""
    call = _case(name, cuda_device)
    call.run()
    want = call.result()
    g = green(sms)
    assert sms <= g.sms < 152
    for _ in range(2):
        call.run(g.stream)
        _same(call.result(), want)
    call.run()
    _same(call.result(), want)


@pytest.mark.parametrize("name", ["long", "wide", "large_logits", "lse"])
@pytest.mark.parametrize("held", [8, 64, 120])
def test_while_another_kernel_holds_sms(cuda_device, green, name, held):
    """A stalled call (its bounded wait limited to 0.4 s, the error in its own
    workspace) holds the SMs of a green context; a call that wants all SMs ends
    long before, with the same bits, and so does the next call on the same
    workspace with all SMs."""
    call = _case(name, cuda_device)
    call.run()
    want = call.result()
    cfg, layers = _make("c2", [4000], n_layers=2, budget_mean=200)
    holder = Call(layers, cfg, cuda_device)
    g = green(held)
    held_until, done = torch.cuda.Event(), torch.cuda.Event()
    side = torch.cuda.Stream()
    call.run(side)  # (every first use of a stream is behind us)
    call.result()
    ckv.debug_stall_next_fused_call(400_000_000)
    holder.run(g.stream)
    held_until.record(g.stream)
    time.sleep(0.02)
    o = call.out
    ckv.compress_layers(call.prob, len(call.m), call.q, call.k, call.v, call.m, call.b, o.indices,
                        o.k_out, o.v_out, call.ws, raw=o.raw, pooled=o.pooled, stream=side) \
        if call.lse is None else \
        ckv.compress_layers_lse(call.prob, len(call.m), call.q, call.k, call.v, call.lse, call.m,
                                call.b, o.indices, o.k_out, o.v_out, call.ws, raw=o.raw,
                                pooled=o.pooled, stream=side)
    done.record(side)
    t0 = time.time()
    while not done.query() and time.time() - t0 < 5.0:
        time.sleep(0.002)
    assert done.query() and not held_until.query()
    _same(call.result(), want)
    assert ckv.read_device_status(holder.ws) == ckv.compresskv.CKV_ERR_DEVICE_TIMEOUT
    call.run()
    _same(call.result(), want)
