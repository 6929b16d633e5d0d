"""Codes of rows under a scale each (a row spread over warps) and of ragged or pitched lines under one scale, bit for bit
against the oracle, at the lengths where the kernels' choices and last pieces change."""
import numpy as np
import pytest
import torch

import oracle
import paper_2408_02897_b200 as qm

pytestmark = pytest.mark.gpu


def tensor(rows, c, dtype, pad, seed):
    rng = np.random.default_rng(seed)
    x = torch.from_numpy(rng.standard_t(3, (rows, c)).astype(np.float32))
    x[0] = 0.0                                       # no scale of its own
    x[1] *= 1e-25                                    # a scale outside the range of the two-wide quotient
    x[-1, -1] = -40.0                                # the largest magnitude in the last piece of the last row
    out = torch.full((rows, c + pad), 1e30, dtype=dtype, device="cuda")[:, :c]
    return out.copy_(x.to(dtype))


def same_codes(codes, delta, x, fmt, gran, want_d=None):
    h = x.float().cpu().numpy()[None]
    if want_d is None:
        want_d = oracle.scale(h, fmt, gran)
        assert np.array_equal(delta.cpu().numpy().view(np.uint32), want_d.ravel().view(np.uint32))
    got = codes.cpu().numpy()
    assert np.array_equal(got[..., :h.shape[-1]], oracle.quantize(h, fmt, want_d))
    assert not got[..., h.shape[-1]:].any()


@pytest.mark.parametrize("c", [16, 256, 272, 512, 528, 1024, 1040, 2048, 2064, 4096, 4112, 8192, 8208])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("pad", [0, 8])
def test_rows_with_a_scale_each(c, dtype, pad):
    x = tensor(2500 if c <= 528 else 131, c, dtype, pad, c + pad)
    for fmt in ("int8", "e4m3", "e5m2"):
        codes, delta, _, _ = qm.qm_quantize(qm.operand_of(x, -1), fmt, "channel")
        same_codes(codes, delta, x, fmt, "channel")


@pytest.mark.parametrize("c", [1, 8, 15, 17, 100, 130, 1000, 1234])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
def test_lines_under_one_scale(c, dtype):
    x = tensor(301, c, dtype, -c % 8 + (8 if c == 1000 else 0), c)
    op = qm.operand_of(x, -1)
    for formats in (["e4m3"], ["int8"], ["e5m2", "int8"], ["e4m3", "e5m2", "int8"]):
        codes, deltas, _ = qm.qm_quantize_formats(op, formats, "tensor")
        for k, fmt in enumerate(formats):
            same_codes(codes[k], deltas[k], x, fmt, "tensor")
    # a scale from elsewhere: what saturates, and a product of value and reciprocal that overflows
    x[2, 0] = 3e30
    for given in (1e-2, 1e-18):
        d = torch.tensor([given], dtype=torch.float32, device="cuda")
        for fmt in ("int8", "e4m3", "e5m2"):
            codes, _, _, _ = qm.qm_quantize(op, fmt, "tensor", d)
            same_codes(codes, d, x, fmt, "tensor", np.full(1, given, np.float32))


@pytest.mark.parametrize("k", [16, 512, 1040, 4096, 8192, 8208])
def test_formats_of_rows_from_one_read(k):
    """Probes under channel scales in three formats: a batch prepares the rows in one pass (beyond 8192 elements in one of each
    format, on streams of their own), alone each has its own."""
    a, b = tensor(300, k, torch.bfloat16, 0, k), tensor(130, k, torch.bfloat16, 8, k + 1)
    probes = [(qm.operand_of(a, -1), qm.operand_of(b, -1), f, f, "channel", "channel") for f in ("int8", "e4m3", "e5m2")]
    batch = qm.ProbeBatch(probes)
    batch.launch()
    for p, r in zip(probes, batch.results()):
        want, got = qm.qm_probe_layer(*p).record(), r.record()
        assert r.device_error == 0 and got["count"] == want["count"] and got["max_be"] == want["max_be"]
        for key in ("sum_be", "sum_diff2", "sum_ref2", "sum_den2"):
            assert abs(got[key] - want[key]) <= 1e-12 * abs(want[key]), key


@pytest.mark.parametrize("dtype,c,per_block", [(torch.bfloat16, 1040, 4), (torch.bfloat16, 2064, 2), (torch.bfloat16, 4112, 1),
                                               (torch.float32, 272, 8), (torch.float32, 528, 4), (torch.float32, 1040, 2),
                                               (torch.float32, 2064, 1), (torch.float32, 4112, 1)])
def test_every_group_of_warps_takes_several_rows(dtype, c, per_block):
    """More than three rows for each group of one to eight warps (8 blocks an SM, per_block groups in each), the maxima of rows that
    follow one another far apart: a maximum left over from the row before, or the one before that, would show."""
    rows = 3 * 8 * torch.cuda.get_device_properties(0).multi_processor_count * per_block + 3
    g = torch.Generator(device="cuda").manual_seed(c)
    x = torch.randn((rows, c), generator=g, device="cuda") * torch.exp2(torch.arange(rows, device="cuda") * 5 % 23 - 11.0)[:, None]
    x = x.to(dtype)
    for fmt in ("int8", "e4m3") if dtype == torch.bfloat16 else ("e5m2",):
        codes, delta, _, _ = qm.qm_quantize(qm.operand_of(x, -1), fmt, "channel")
        same_codes(codes, delta, x, fmt, "channel")


@pytest.mark.parametrize("c", [17, 130, 1234])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
def test_lines_under_scales_outside_the_range_of_the_two_wide_quotient(c, dtype):
    for factor in (1e-25, 1e25):
        x = tensor(61, c, dtype, -c % 8, c)
        x *= factor
        codes, deltas, _ = qm.qm_quantize_formats(qm.operand_of(x, -1), ["e4m3", "e5m2", "int8"], "tensor")
        for k, fmt in enumerate(("e4m3", "e5m2", "int8")):
            same_codes(codes[k], deltas[k], x, fmt, "tensor")
    x = tensor(61, c, dtype, -c % 8, c)
    x[2, 0] = 3e30
    for given in (1e-22, 2.0 ** -60, 2.0 ** 60, 1e22):          # either side of the range and its ends
        d = torch.tensor([given], dtype=torch.float32, device="cuda")
        for fmt in ("int8", "e4m3", "e5m2"):
            codes, _, _, _ = qm.qm_quantize(qm.operand_of(x, -1), fmt, "tensor", d)
            same_codes(codes, d, x, fmt, "tensor", np.full(1, given, np.float32))
