"""Probes of the same operands in one batch share their reference and denominator products: every record
must be the one the probe gives on its own (which the other form of the fused kernel evaluates), for every
number of formats and granularities per product, and whatever else is in the batch."""
import pytest
import torch

import oracle
import paper_2408_02897_b200 as qm
from paper_2408_02897_b200 import binding, workloads

pytestmark = pytest.mark.gpu

FIELDS = ("sum_be", "max_be", "sum_diff2", "sum_ref2", "sum_den2")
VARIANTS = [("e4m3", "tensor", "rtne"), ("int8", "channel", "rtne"), ("e5m2", "tensor", "stochastic_r"), ("int8", "tensor", "rtne"),
            ("e4m3", "channel", "rtne"), ("e5m2", "channel", "rtne"), ("e5m2", "channel", "stochastic_both")]


def operands(M, N, K, batch, seed):
    rng = workloads._rng(seed)
    shape = (lambda r: (r, K)) if batch == 1 else (lambda r: (batch, r, K))
    return workloads.normal(rng, shape(M)), workloads.normal(rng, shape(N), 0.02)


def as_batch(Lo, Ro, variants):
    b = qm.ProbeBatch([(Lo, Ro, f, f, g, g) for f, g, _ in variants])
    for c, (_, _, r) in zip(b.cfg, variants):
        c.round, c.seed = binding.ROUND[r], 5
    b.launch()
    torch.cuda.synchronize()
    return b.results()


# 1 .. 7 variants (six fill a unit, the seventh starts another); contraction below, at and past a block of 64 and
# of 128, more blocks than the ring has stages, outputs at most 64 wide, ragged edges, several tiles per CTA pair
@pytest.mark.parametrize("n_var", [1, 2, 3, 4, 5, 6, 7])
@pytest.mark.parametrize("M,N,K,batch", [(256, 128, 64, 1), (130, 40, 80, 1), (300, 200, 128, 1), (257, 129, 1040, 1),
                                         (96, 64, 48, 200), (512, 96, 192, 60)])
def test_records_do_not_depend_on_what_shares_the_products(n_var, M, N, K, batch):
    L, R = operands(M, N, K, batch, 100 + n_var)
    Ld, Rd = L.cuda(), R.cuda()
    Lo, Ro = qm.operand_of(Ld, -1), qm.operand_of(Rd, -1)
    got = as_batch(Lo, Ro, VARIANTS[:n_var])
    for (f, g, r), rec in zip(VARIANTS, got):
        alone = qm.qm_probe_layer(Lo, Ro, f, f, g, g, "bf16", rounding=r, seed=5).record()
        assert rec.device_error == 0 and rec.record()["count"] == alone["count"] == M * N * batch
        for k in FIELDS:     # the same fp32 terms; only the order of the fp64 additions over tiles may differ
            assert abs(rec.record()[k] - alone[k]) <= 1e-12 * abs(alone[k]), (f, g, r, k)


def test_shared_products_against_the_oracle():
    L, R = operands(300, 200, 272, 1, 7)
    Ld, Rd = L.cuda(), R.cuda()
    variants = [v for v in VARIANTS if v[2] == "rtne"]
    got = as_batch(qm.operand_of(Ld, -1), qm.operand_of(Rd, -1), variants)
    for (f, g, _), rec in zip(variants, got):
        want = oracle.probe(L.float().numpy(), R.float().numpy().T, f, f, g, g)
        for k in FIELDS:     # the tolerances of the one-probe tests: fp32 accumulation with truncation
            assert abs(rec.record()[k] - want[k]) <= (1e-3 if k == "max_be" else 1e-4) * abs(want[k]), (f, g, k)


# Products asked for once beside one asked for in three formats: 26 of four tiles each fill the GPU and take the side-by-side
# kernel (24 to a launch), three do not and ride along with the others
@pytest.mark.parametrize("n_single,launches", [(26, 3), (3, 1)])
def test_products_of_one_probe_beside_shared_ones(n_single, launches):
    keep, probes = [], []
    for i in range(n_single):
        L, R = (t.cuda() for t in operands(300, 200, 64 + 16 * (i % 9), 1, 300 + i))
        keep.append((L, R))
        f, g, _ = VARIANTS[(0, 1, 3)[i % 3]]
        probes.append((qm.operand_of(L, -1), qm.operand_of(R, -1), f, f, g, g))
    L, R = (t.cuda() for t in operands(513, 130, 272, 1, 299))
    Lo, Ro = qm.operand_of(L, -1), qm.operand_of(R, -1)
    probes[1:1] = [(Lo, Ro, f, f, g, g) for f, g, r in VARIANTS[:4] if r == "rtne"]
    b = qm.ProbeBatch(probes)
    binding.profile_enable(True)
    try:
        b.launch()
        torch.cuda.synchronize()
        assert binding.profile_read()[1] == launches
    finally:
        binding.profile_enable(False)
    for p, rec in zip(probes, b.results()):
        alone = qm.qm_probe_layer(*p, "bf16").record()
        assert rec.device_error == 0 and rec.record()["count"] == alone["count"]
        for k in FIELDS:
            assert abs(rec.record()[k] - alone[k]) <= 1e-12 * abs(alone[k]), k


# Operands with a strided contraction are used as they lie by probes of both granularities and roundings, which share their
# products, and what is written of one operand beyond a probe's own buffers goes to one workspace: the two bytes an element that
# every workspace has for it stay untouched in all but the first
@pytest.mark.parametrize("cl,cr", [(-2, -2), (-2, -1), (-1, -2)])
def test_one_copy_of_a_strided_operand_whatever_the_scales(cl, cr):
    M, N, K, fill = 304, 200, 272, -0x5A5A5A5B          # (strided rows are a multiple of 8 elements apart)
    L, R = operands(M, N, K, 1, 8)
    Ld, Rd = (t.cuda() if c == -1 else t.T.contiguous().cuda() for t, c in ((L, cl), (R, cr)))
    Lo, Ro = qm.operand_of(Ld, cl), qm.operand_of(Rd, cr)
    b = qm.ProbeBatch([(Lo, Ro, f, f, g, g) for f, g, _ in VARIANTS])
    for c, (_, _, r) in zip(b.cfg, VARIANTS):
        c.round, c.seed = binding.ROUND[r], 5
    for w in b._ws:
        w.view(torch.int32).fill_(fill)
    b.launch()
    torch.cuda.synchronize()
    copies = 2 * K * ((M if cl == -2 else 0) + (N if cr == -2 else 0))
    untouched = [4 * int((w.view(torch.int32) == fill).sum()) for w in b._ws]
    assert untouched[0] < copies and all(u >= copies for u in untouched[1:]), (untouched, copies)
    for (f, g, r), rec in zip(VARIANTS, b.results()):
        alone = qm.qm_probe_layer(Lo, Ro, f, f, g, g, "bf16", rounding=r, seed=5).record()
        assert rec.device_error == 0
        for k in FIELDS:
            assert abs(rec.record()[k] - alone[k]) <= 1e-12 * abs(alone[k]), (f, g, r, k)


@pytest.mark.parametrize("gran", ["tensor", "channel"])
def test_records_hold_the_last_tile_of_every_unit(gran):
    """Units of one probe that ride along in a launch of shared products, most of them a tile per CTA pair: a unit's last tile
    counts in every sum.  The per-row sums of the same launch leave each tile by another way (atomics from the registers)."""
    shapes = [(256, 128, 64), (130, 40, 80), (256, 64, 16), (20, 128, 128), (257, 129, 208), (256, 256, 64)]
    ops = [[t.cuda() for t in operands(M, N, K, 1, 300 + i)] for i, (M, N, K) in enumerate(shapes)]
    probes = [(qm.operand_of(L, -1), qm.operand_of(R, -1), f, f, gran, gran)
              for i, (L, R) in enumerate(ops) for f in (("e4m3", "int8", "e5m2") if i == 0 else (("int8", "e4m3")[i & 1],))]
    b = qm.ProbeBatch(probes, row_stats=True)
    for _ in range(8):
        b.launch()
        torch.cuda.synchronize()
        for p, rec, rows in zip(probes, b.results(), b.row_stats):
            alone, rows = qm.qm_probe_layer(*p).record(), rows.cpu().numpy()
            want = dict(zip(FIELDS, rows.sum(axis=0)), max_be=rows[:, 1].max())
            assert rec.device_error == 0
            for k in FIELDS:     # fp64 additions of the same terms in another order
                assert abs(rec.record()[k] - want[k]) <= 1e-12 * abs(want[k]), k
                assert abs(rec.record()[k] - alone[k]) <= 1e-12 * abs(alone[k]), k


# |R| is written by the converters up to two blocks of the contraction with one probe to a unit and up to six with several, by warps
# of its own beyond, and in a whole launch as soon as one of its units is longer
@pytest.mark.parametrize("lengths", [(128,), (144,), (128, 144), (16, 1040)])
@pytest.mark.parametrize("formats", [("e4m3",), ("int8", "e5m2")])
@pytest.mark.parametrize("cl,cr", [(-1, -1), (-2, -2)])
def test_records_do_not_depend_on_who_writes_the_magnitudes(lengths, formats, cl, cr):
    if len(formats) > 1:
        lengths = tuple({128: 384, 144: 400}.get(k, k) for k in lengths)
    probes, want = [], []
    for i, K in enumerate(lengths):
        L, R = operands(264, 136, K, 1, 400 + i)
        Lo, Ro = (qm.operand_of(t.cuda() if c == -1 else t.T.contiguous().cuda(), c) for t, c in ((L, cl), (R, cr)))
        for f in formats:
            probes.append((Lo, Ro, f, f, "tensor", "channel"))
            want.append(oracle.probe(L.float().numpy(), R.float().numpy().T, f, f, "tensor", "channel"))
    b = qm.ProbeBatch(probes)
    b.launch()
    torch.cuda.synchronize()
    for p, rec, w in zip(probes, b.results(), want):
        alone = qm.qm_probe_layer(*p).record()
        assert rec.device_error == 0
        for k in FIELDS:
            assert abs(rec.record()[k] - alone[k]) <= 1e-12 * abs(alone[k]), k
            assert abs(rec.record()[k] - w[k]) <= (1e-3 if k == "max_be" else 1e-4) * abs(w[k]), k
