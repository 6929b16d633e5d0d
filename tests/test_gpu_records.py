"""Where a call's record may live: qm_probe_layer, qm_metric, qm_tensor_stats and qm_quantize_error store every field once, from
their last kernel, so that `out` may be device memory or pinned host memory."""
import ctypes as C

import pytest
import torch

import paper_2408_02897_b200 as qm
from paper_2408_02897_b200 import binding

pytestmark = pytest.mark.gpu


def _calls():
    g = torch.Generator().manual_seed(11)
    x = torch.randn((300, 272), generator=g).to(torch.bfloat16).cuda()
    y = torch.randn((130, 272), generator=g).to(torch.bfloat16).cuda()
    lo, ro = qm.operand_of(x, -1), qm.operand_of(y, -1)
    a, b = x.float()[:, :80].contiguous(), y.float()[:, :80].contiguous()
    L, stream = qm.lib(), C.c_void_p(torch.cuda.current_stream().cuda_stream)
    ws = torch.empty(64 << 20, dtype=torch.uint8, device="cuda")
    w, n = C.c_void_p(ws.data_ptr()), ws.numel()
    m = [torch.randn(5000, generator=g).cuda() for _ in range(3)]
    delta = qm.qm_scale(lo, "e4m3", "channel")
    keep = (x, y, a, b, ws, m, delta)

    def probe(p, q, ref):
        cfg = binding._cfg("e4m3", "e4m3", "tensor", "channel", ref)
        return lambda out: L.qm_probe_layer(C.byref(p), C.byref(q), C.byref(cfg), out, w, n, stream)
    fp = [qm.operand_of(t, -1) for t in (a, b)]
    return keep, {
        "probe bf16": (binding.MetricResult, probe(lo, ro, "bf16")),
        "probe fp32": (binding.MetricResult, probe(*fp, "fp32")),
        "metric": (binding.MetricResult, lambda out: L.qm_metric(*[C.c_void_p(t.data_ptr()) for t in m], m[0].numel(), out, w, n, stream)),
        "statistics, dense": (binding.TensorStats, lambda out: L.qm_tensor_stats(C.byref(lo), out, w, n, stream)),
        "statistics, strided": (binding.TensorStats, lambda out: L.qm_tensor_stats(C.byref(qm.operand_of(x[:, :264], -2)), out, w, n, stream)),
        "error": (binding.QuantError, lambda out: L.qm_quantize_error(C.byref(lo), 1, 1, C.c_void_p(delta.data_ptr()), out, w, n, stream)),
    }


@pytest.mark.parametrize("name", ["probe bf16", "probe fp32", "metric", "statistics, dense", "statistics, strided", "error"])
def test_a_record_is_the_same_in_device_and_in_pinned_memory(name):
    keep, calls = _calls()
    kind, call = calls[name]
    got = []
    for fill in (0xA5, 0x3C):                        # whatever was there before is overwritten
        for kw in (dict(device="cuda"), dict(pin_memory=True)):
            buf = torch.full((C.sizeof(kind),), fill, dtype=torch.uint8, **kw)
            torch.cuda.synchronize()
            assert call(C.c_void_p(buf.data_ptr())) == 0
            torch.cuda.synchronize()
            got.append(bytes(buf.cpu().numpy().tobytes()))
    assert all(g == got[0] for g in got), got


def test_calls_under_a_default_device():
    """A program that lets torch put its tensors on the GPU by default makes the same calls."""
    g = torch.Generator().manual_seed(12)
    x = torch.randn((64, 272), generator=g).to(torch.bfloat16).cuda()
    op, m = qm.operand_of(x, -1), x.float().flatten()

    def records():
        probe, metric = qm.qm_probe_layer(op, op, "e4m3", "e4m3", "tensor", "tensor"), qm.qm_metric(m, m * 1.01, m.abs())
        return probe.record(), metric.record(), qm.qm_tensor_stats(op).derived(), qm.qm_quantize_error(op, "int8", "tensor").record()
    want = records()
    with torch.device("cuda"):
        assert records() == want
