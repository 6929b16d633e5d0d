"""The two-launch preparation of a single probe against the general kernels, which prepare the operands of a
batch: the same records over storage orders, types, odd sizes, formats, granularities and roundings."""
import pytest
import torch

import oracle
import paper_2408_02897_b200 as qm
from paper_2408_02897_b200 import binding, workloads

pytestmark = pytest.mark.gpu

FIELDS = ("sum_be", "max_be", "sum_diff2", "sum_ref2", "sum_den2")


def stored(rng, rows, K, cd, batch, dtype):
    shape = (rows, K) if cd == -1 else (K, rows)
    shape = shape if batch == 1 else (batch, *shape)
    x = workloads.normal(rng, shape, 1e-2, dtype)
    wide = torch.full((*shape[:-1], (shape[-1] + 7) // 8 * 8), 1e4, dtype=dtype)      # what must not be read
    wide[..., :shape[-1]] = x
    return x, wide.cuda()[..., :shape[-1]]


# (the last two: either side of the line in rows, and of the one in elements)
@pytest.mark.parametrize("M,N,K,batch", [(1, 1, 16, 1), (130, 67, 144, 1), (300, 64, 16, 3), (64, 770, 2032, 1), (1024, 1000, 1040, 1),
                                         (2048, 2049, 48, 1), (2000, 2161, 1008, 1)])
@pytest.mark.parametrize("cl,cr", [(-1, -2), (-2, -1), (-1, -1), (-2, -2)])
@pytest.mark.parametrize("fl,fr", [("e4m3", "e4m3"), ("e4m3", "e5m2"), ("e5m2", "e4m3"), ("e5m2", "e5m2"), ("int8", "int8")])
@pytest.mark.parametrize("gran", ["tensor", "channel"])
def test_same_records_as_the_general_kernels(M, N, K, batch, cl, cr, fl, fr, gran):
    rng = workloads._rng(M + 3 * N + K)
    Ld, Rd = stored(rng, M, K, cl, batch, torch.bfloat16)[1], stored(rng, N, K, cr, batch, torch.bfloat16)[1]
    Lo, Ro = qm.operand_of(Ld, cl), qm.operand_of(Rd, cr)
    for rounding in ("rtne", "stochastic_l", "stochastic_r"):
        plan = qm.ProbePlan(Lo, Ro, fl, fr, gran, gran, "bf16", rounding, seed=11)
        plan.ws.fill_(0xA5)                                    # nothing may depend on what a workspace held
        plan.launch(Lo, Ro)
        b = qm.ProbeBatch([(Lo, Ro, fl, fr, gran, gran)])
        b.cfg[0].round, b.cfg[0].seed = binding.ROUND[rounding], 11
        b.launch()
        torch.cuda.synchronize()
        got, other = plan.result(), b.results()[0]
        assert got.device_error == other.device_error == 0
        assert got.record()["count"] == other.record()["count"] == M * N * batch
        for k in FIELDS:
            assert abs(got.record()[k] - other.record()[k]) <= 1e-12 * abs(other.record()[k]), (k, rounding)


# fp32 operands, contractions off every vector: the general 64 x 64 tiles and ragged chunks of the same kernels
@pytest.mark.parametrize("M,N,K", [(5, 3, 1), (70, 131, 147), (200, 33, 1043)])
@pytest.mark.parametrize("cl,cr", [(-1, -2), (-2, -1)])
@pytest.mark.parametrize("fmt,gran,rounding", [("e4m3", "tensor", "rtne"), ("int8", "channel", "rtne"), ("e5m2", "tensor", "stochastic_l")])
def test_fp32_operands_against_the_oracle(M, N, K, cl, cr, fmt, gran, rounding):
    rng = workloads._rng(M + N + K)
    L, Ld = stored(rng, M, K, cl, 1, torch.float32)
    R, Rd = stored(rng, N, K, cr, 1, torch.float32)
    plan = qm.ProbePlan(qm.operand_of(Ld, cl), qm.operand_of(Rd, cr), fmt, fmt, gran, gran, "fp32", rounding, seed=11)
    plan.ws.fill_(0xA5)
    plan.launch(qm.operand_of(Ld, cl), qm.operand_of(Rd, cr))
    got = plan.result().record()
    l = (L if cl == -1 else L.T).numpy()
    r = (R.T if cr == -1 else R).numpy()                       # the oracle takes R as [K, N]
    want = oracle.probe(l, r, fmt, fmt, gran, gran, **({} if rounding == "rtne" else dict(round_l="stochastic", seed=11)))
    assert got["count"] == want["count"]
    # fp32 sums of up to 1043 terms in sixteenths or eighths: outputs within 1e-5 of their magnitude scale
    assert abs(got["max_be"] - want["max_be"]) <= 2e-5
    assert abs(got["sum_be"] - want["sum_be"]) <= 2e-5 * max(want["sum_be"], 1.0 if M * N < 100 else 0.0)
    for k in ("sum_diff2", "sum_ref2", "sum_den2"):
        assert abs(got[k] - want[k]) <= 2e-5 * (want["sum_den2"] if M * N < 100 else want[k]), k


@pytest.mark.parametrize("gran", ["tensor", "channel"])
@pytest.mark.parametrize("where", [0, 1])
@pytest.mark.parametrize("cd", [-1, -2])
def test_non_finite_operands_are_flagged(gran, where, cd):
    x, y = torch.randn(96, 64).bfloat16(), torch.randn(64, 64).bfloat16()
    (x, y)[where][3, 5] = float("inf")
    shape = lambda t: t.cuda() if cd == -1 else t.T.contiguous().cuda()
    a, b = shape(x), shape(y)
    r = qm.qm_probe_layer(qm.operand_of(a, cd), qm.operand_of(b, cd), "e4m3", "e4m3", gran, gran)
    assert r.device_error & 1


# The one-launch form: operands of 256 KB and just above (of 512 KB before), of 128 KB and above where lines are ragged, strips of 64 columns
# whole and ragged with fewer rows than blocks of a cluster, contractions of 2048, 4096 and just above.  Under channel scales 960 x 960 x 32 has a block
# to each of the 240 flags and 968 x 960 x 32 more than there are; 3 x 65 x 16 and 130 x 65 x 16 launch 24 and 40 blocks, so that the first
# block's clearing of the unused flags splits a warp right ahead of a cluster's barrier.
@pytest.mark.parametrize("M,N,K,batch", [(512, 511, 512, 1), (512, 513, 512, 1), (256, 255, 512, 1), (256, 257, 512, 1), (131, 64, 496, 1), (131, 64, 512, 1),
                                         (65, 3, 16, 1), (3, 129, 2048, 1), (3, 129, 2064, 1), (3, 129, 4096, 1), (3, 129, 4112, 1),
                                         (960, 128, 32, 1), (960, 960, 32, 1), (968, 960, 32, 1),
                                         (70, 40, 112, 4), (3, 65, 16, 1), (130, 65, 16, 1)])
@pytest.mark.parametrize("cl,cr", [(-1, -2), (-2, -1)])
@pytest.mark.parametrize("fmt,gran_l,gran_r", [("e4m3", "tensor", "channel"), ("int8", "channel", "tensor"), ("e5m2", "channel", "channel"),
                                               ("e4m3", "tensor", "tensor")])
def test_small_operands_either_side_of_the_one_launch_form(M, N, K, batch, cl, cr, fmt, gran_l, gran_r):
    rng = workloads._rng(M + 5 * N + K)
    Ld, Rd = stored(rng, M, K, cl, batch, torch.bfloat16)[1], stored(rng, N, K, cr, batch, torch.bfloat16)[1]
    Lo, Ro = qm.operand_of(Ld, cl), qm.operand_of(Rd, cr)
    plan = qm.ProbePlan(Lo, Ro, fmt, fmt, gran_l, gran_r)
    plan.ws.fill_(0xA5)
    plan.launch(Lo, Ro)
    b = qm.ProbeBatch([(Lo, Ro, fmt, fmt, gran_l, gran_r)])
    b.launch()
    torch.cuda.synchronize()
    got, other = plan.result(), b.results()[0]
    assert got.device_error == other.device_error == 0
    for k in FIELDS:
        assert abs(got.record()[k] - other.record()[k]) <= 1e-12 * abs(other.record()[k]), k
    # a value that is not finite is flagged wherever it lies, also by the last block; the next call starts afresh
    for t in (Ld, Rd):
        at = tuple(s - 1 for s in t.shape)
        old = t[at].clone()
        t[at] = float("nan")
        plan.launch(Lo, Ro)
        assert plan.result().device_error & 1
        t[at] = old
    plan.launch(Lo, Ro)
    assert plan.result().device_error == 0
