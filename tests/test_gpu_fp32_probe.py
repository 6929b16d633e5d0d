"""The CUDA-core probe (fp32 reference) at the edges of its tile shapes: sizes that give each of the four,
ragged rows, columns and contractions, both storage orders of both operands, every format."""
import pytest
import torch

import oracle
import paper_2408_02897_b200 as qm
from paper_2408_02897_b200 import workloads

pytestmark = pytest.mark.gpu


def stored(rng, rows, K, cd, batch, dtype):
    """[rows, K] values in either storage order, rows padded to a multiple of 8 elements."""
    shape = (batch,) + ((rows, K) if cd == -1 else (K, rows))
    x = workloads.normal(rng, shape, dtype=dtype)
    wide = torch.full((*shape[:-1], (shape[-1] + 7) // 8 * 8 + 8), 77.0, dtype=dtype)      # what lies beside a row is not zero
    wide[..., :shape[-1]] = x
    d = wide.cuda()[..., :shape[-1]]
    return (x, d) if batch > 1 else (x[0], d[0])


# blocks of 64x64, 32x64, 32x32 and 16x32 outputs; contractions below, at and past their chunks of 32, 64 and 128
@pytest.mark.parametrize("M,N,K,batch", [(1, 1, 1, 1), (33, 65, 127, 1), (128, 256, 256, 1), (513, 511, 33, 1), (515, 770, 65, 1),
                                         (900, 1010, 129, 1), (70, 34, 31, 40)])
@pytest.mark.parametrize("cl,cr", [(-1, -2), (-2, -1), (-1, -1), (-2, -2)])
@pytest.mark.parametrize("fmt,gran", [("e4m3", "tensor"), ("int8", "channel"), ("e5m2", "channel")])
def test_fp32_probe_against_the_oracle(M, N, K, batch, cl, cr, fmt, gran):
    rng = workloads._rng(M + N + K)
    dtype = torch.bfloat16 if fmt == "e5m2" else torch.float32
    L, Ld = stored(rng, M, K, cl, batch, dtype)
    R, Rd = stored(rng, N, K, cr, batch, dtype)
    got = qm.qm_probe_layer(qm.operand_of(Ld, cl), qm.operand_of(Rd, cr), fmt, fmt, gran, gran, "fp32")
    Lo = L if cl == -1 else L.transpose(-1, -2)
    Ro = R.transpose(-1, -2) if cr == -1 else R                                # the oracle takes R as [.., K, N]
    want = oracle.probe(Lo.float().numpy(), Ro.float().numpy(), fmt, fmt, gran, gran)
    rec = got.record()
    assert got.device_error == 0 and rec["count"] == want["count"]
    # fp32 FMA chains of at most 129 terms: each output within K 2^-24 of its magnitude scale D, so within 1e-5 of
    # it, and BE, a quotient by D, within 1e-5 absolutely; sums over many outputs far closer
    n = rec["count"]
    assert abs(rec["sum_be"] - want["sum_be"]) <= 1e-5 * (n if n < 100 else want["sum_be"])
    assert abs(rec["max_be"] - want["max_be"]) <= 1e-5
    for k in ("sum_diff2", "sum_ref2", "sum_den2"):
        assert abs(rec[k] - want[k]) <= 2e-5 * want["sum_den2" if n < 100 else k], k


# extents at which the tile shape changes: just over one block for an SM in one shape, and what is taken instead
@pytest.mark.parametrize("M,N,K", [(700, 400, 68), (704, 448, 36), (350, 350, 40), (1030, 1030, 20), (17, 33, 300), (4000, 30, 24),
                                   (640, 960, 63), (640, 960, 64), (900, 900, 95), (900, 900, 96)])
@pytest.mark.parametrize("fmt,gran", [("e4m3", "tensor"), ("int8", "channel")])
def test_tile_shapes_against_the_oracle(M, N, K, fmt, gran):
    rng = workloads._rng(M + N)
    L, R = workloads.normal(rng, (M, K), 1.0, torch.float32), workloads.normal(rng, (N, K), 0.05, torch.float32)
    pad = lambda t: torch.nn.functional.pad(t, (0, -t.shape[1] % 8)).cuda()[:, :t.shape[1]]
    Ld, Rd = pad(L), pad(R)
    got = qm.qm_probe_layer(qm.operand_of(Ld, -1), qm.operand_of(Rd, -1), fmt, fmt, gran, gran, "fp32").record()
    want = oracle.probe(L.numpy(), R.T.numpy(), fmt, fmt, gran, gran)
    # fp32 sums of up to 300 terms in parts: outputs within 1e-5 of their magnitude scale
    assert got["count"] == want["count"] and abs(got["max_be"] - want["max_be"]) <= 2e-5
    for k in ("sum_be", "sum_diff2", "sum_ref2", "sum_den2"):
        assert abs(got[k] - want[k]) <= 2e-5 * want[k], k
