"""The transposing quantize kernels at the edges of their 128 x 64 tiles, and the dense stochastic kernel: codes,
scales and contraction-major copies bit for bit against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import paper_2408_02897_b200 as qm
from paper_2408_02897_b200 import workloads

pytestmark = pytest.mark.gpu


def padded(rng, shape):
    """bf16 values in rows padded to a multiple of 8 with what must not be read as part of the matrix."""
    x = workloads.normal(rng, shape, 1e-3)
    wide = torch.full((*shape[:-1], (shape[-1] + 7) // 8 * 8), 1e4, dtype=torch.bfloat16)
    wide[..., :shape[-1]] = x
    return x, wide.cuda()[..., :shape[-1]]


def check(codes, delta, x, fmt, gran, K, rounding="rtne"):
    want_d = oracle.scale(x, fmt, gran)
    want = oracle.quantize(x, fmt, want_d, **({} if rounding == "rtne" else dict(rounding="stochastic", seed=7, stream=1)))
    assert np.array_equal(delta.cpu().numpy().ravel(), np.asarray(want_d, dtype=np.float32).ravel())
    got = codes.cpu().numpy()
    assert np.array_equal(got[..., :K].reshape(want.shape), want)
    assert not got[..., K:].any()                              # the padding of a row of codes is zero


# (the last three have tiles enough for the stochastic form of the tile kernel, the others take the general one)
@pytest.mark.parametrize("K,nc,batch", [(16, 1, 1), (128, 64, 1), (112, 63, 1), (144, 66, 1), (272, 130, 2), (2032, 70, 1),
                                        (1280, 640, 1), (2032, 450, 1), (144, 66, 26)])
@pytest.mark.parametrize("fmt", ["e4m3", "e5m2", "int8"])
@pytest.mark.parametrize("gran", ["tensor", "channel"])
@pytest.mark.parametrize("rounding", ["rtne", "stochastic"])
def test_strided_contraction(K, nc, batch, fmt, gran, rounding):
    x, d = padded(workloads._rng(K + nc), (K, nc) if batch == 1 else (batch, K, nc))
    codes, delta, _, copy = qm.qm_quantize(qm.operand_of(d, -2), fmt, gran, want_kmaj=True,
                                           stochastic=(7, 1) if rounding == "stochastic" else None)
    t = x.transpose(-1, -2).float().numpy()
    check(codes, delta, t, fmt, gran, K, rounding)
    assert np.array_equal(copy.float().cpu().numpy().reshape(t.shape), t)


@pytest.mark.parametrize("K,nc,batch", [(112, 63, 1), (272, 130, 2), (384, 64, 1)])
def test_strided_contraction_several_formats(K, nc, batch):
    x, d = padded(workloads._rng(K * nc), (K, nc) if batch == 1 else (batch, K, nc))
    formats = ["int8", "e4m3", "e5m2"]
    codes, deltas, copy = qm.qm_quantize_formats(qm.operand_of(d, -2), formats, "tensor", want_kmaj=True)
    t = x.transpose(-1, -2).float().numpy()
    for f, c, s in zip(formats, codes, deltas):
        check(c, s, t, f, "tensor", K)
    assert np.array_equal(copy.float().cpu().numpy().reshape(t.shape), t)


@pytest.mark.parametrize("rows,K", [(1, 16), (33, 48), (300, 1040)])
@pytest.mark.parametrize("fmt", ["e4m3", "e5m2", "int8"])
@pytest.mark.parametrize("gran", ["tensor", "channel"])
def test_dense_stochastic(rows, K, fmt, gran):
    x = workloads.normal(workloads._rng(rows), (rows, K), 1e-3)
    x[0, :8] = torch.tensor([0.0, -0.0, 1e-30, -1e-30, 3e-7, -3e-7, 1e-5, 0.02], dtype=torch.bfloat16)
    codes, delta, _, _ = qm.qm_quantize(qm.operand_of(x.cuda(), -1), fmt, gran, stochastic=(7, 1))
    check(codes, delta, x.float().numpy(), fmt, gran, K, "stochastic")
