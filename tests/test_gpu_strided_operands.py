"""Operands whose contraction is strided go to the tensor cores as they lie in memory, their codes in the same order:
the record has to be the one of the same values stored contraction-major, to the rounding of the final sums (the codes,
scales and products are the same numbers, summed in the same order within a tile's row)."""
import itertools

import pytest
import torch

import oracle
import paper_2408_02897_b200 as qm
from paper_2408_02897_b200 import binding
from helpers import assert_record_close

pytestmark = pytest.mark.gpu
FORMATS = ("e4m3", "e5m2", "int8")


def stored(x, strided):
    """x [.., rows, K] in memory with K contiguous or strided, rows padded to whole 16 bytes; the operand."""
    t = x.transpose(-1, -2) if strided else x
    pad = -t.shape[-1] % 8
    out = torch.full((*t.shape[:-1], t.shape[-1] + pad), 7.0, dtype=torch.bfloat16, device="cuda")[..., :t.shape[-1]]
    out.copy_(t)
    return out, qm.operand_of(out, -2 if strided else -1)


def draw(shape, seed, scale=1.0):
    g = torch.Generator().manual_seed(seed)
    x = torch.randn(shape, generator=g) * scale
    x[..., 0] *= 9.0                                  # (channel scales that differ from one another)
    return x.to(torch.bfloat16).cuda()


def same(a, b):
    ra, rb = a.record(), b.record()
    assert a.device_error == b.device_error == 0 and ra["count"] == rb["count"]
    assert ra["max_be"] == rb["max_be"]
    for k in ("sum_be", "sum_diff2", "sum_ref2", "sum_den2"):
        assert abs(ra[k] - rb[k]) <= 1e-12 * abs(rb[k]), (k, ra[k], rb[k])


# edges of the tiles (256 x 128, narrow 64), of the 64- and 128-deep blocks, of the 16-byte rows; several units of tiles
SHAPES = [(1, 1, 16, 1), (257, 129, 80, 1), (130, 64, 48, 3), (64, 40, 208, 2), (520, 392, 144, 1), (300, 1000, 1040, 1), (2048, 1536, 512, 1)]


@pytest.mark.parametrize("m,n,k,batch", SHAPES)
@pytest.mark.parametrize("gran", ["tensor", "channel"])
@pytest.mark.parametrize("formats", [("e4m3",), ("int8",), FORMATS])
def test_strided_operands_give_the_record_of_contiguous_ones(m, n, k, batch, gran, formats):
    shape = (lambda r: (r, k) if batch == 1 else (batch, r, k))
    L, R = draw(shape(m), 1), draw(shape(n), 2, 0.05)
    want = None
    for sl, sr in itertools.product((False, True), repeat=2):
        (keep_l, lo), (keep_r, ro) = stored(L, sl), stored(R, sr)
        b = qm.ProbeBatch([(lo, ro, f, f, gran, gran) for f in formats])
        b.launch()
        got = b.results()
        alone = [qm.qm_probe_layer(lo, ro, f, f, gran, gran) for f in formats]
        torch.cuda.synchronize()
        if want is None:
            want = got
            # (C - Q of one output carries the fp32 rounding of C, some 6e-8 D against an error of 1e-3 D and less: the
            # helper's 1e-4 is for sums over many outputs, so a lone one is held to the contiguous form only)
            if m * n * batch > 4096 and m * n * k * batch < 1 << 24:
                for f, g in zip(formats, got):
                    assert_record_close(g.record(), oracle.probe(L.float().cpu().numpy(), R.float().cpu().numpy().swapaxes(-1, -2), f, f, gran, gran))
        for g, a, w in zip(got, alone, want):
            same(g, w)
            same(a, w)


@pytest.mark.parametrize("m,n,k", [(257, 129, 80), (770, 1000, 2032), (4096, 768, 256)])
def test_rounding_and_orientation_mixed_in_a_batch(m, n, k):
    """The same values stored strided and contiguous, rounded to nearest and stochastically, under both kinds of scales: shared
    preparation gives every probe the record it has alone, and strided operands that of contiguous ones."""
    L, R = draw((m, k), 3), draw((n, k), 4, 0.05)
    (_k0, ls), (_k1, rs), (_k2, lc), (_k3, rc) = stored(L, True), stored(R, True), stored(L, False), stored(R, False)
    kinds = [("e4m3", "e5m2", "tensor", "rtne"), ("e4m3", "e5m2", "tensor", "stochastic_r"), ("int8", "int8", "channel", "stochastic_l"),
             ("e5m2", "e5m2", "channel", "rtne"), ("e5m2", "e4m3", "tensor", "rtne")]
    probes = [(lo, ro, fl, fr, g, g, rnd) for lo, ro in ((ls, rs), (lc, rc)) for fl, fr, g, rnd in kinds]
    b = qm.ProbeBatch([p[:6] for p in probes])
    for i, p in enumerate(probes):
        b.cfg[i] = binding._cfg(*p[2:6], "bf16", p[6], 5)
    b.launch()
    got = b.results()
    for i, (fl, fr, g, rnd) in enumerate(kinds):
        same(got[i], got[i + len(kinds)])
        same(got[i], qm.qm_probe_layer(ls, rs, fl, fr, g, g, rounding=rnd, seed=5))


@pytest.mark.parametrize("groups", [1, 2])
def test_scales_shared_along_the_batch(groups):
    L, R = draw((4, 130, 96), 6), draw((4, 72, 96), 7, 0.05)
    (_a, ls), (_b, rs), (_c, lc), (_d, rc) = stored(L, True), stored(R, True), stored(L, False), stored(R, False)
    same(*[qm.qm_probe_layer(lo, ro, "e4m3", "e4m3", "channel", "channel", groups=(groups, groups)) for lo, ro in ((ls, rs), (lc, rc))])


def test_a_nonfinite_value_is_flagged_in_either_order():
    L, R = draw((300, 64), 8), draw((64, 64), 9)
    L[299, 63] = float("nan")
    for gran in ("tensor", "channel"):
        (_a, ls), (_b, rs) = stored(L, True), stored(R, True)
        assert qm.qm_probe_layer(ls, rs, "e4m3", "e4m3", gran, gran).device_error & 1


def kept_codes(ws, scales, rows, ld):
    """The codes of the left operand where the workspace of a probe has them: behind the control block and the max|x| words and
    scales of both operands (one of each per column here), every part on 256 bytes."""
    pad = lambda b: (b + 255) & ~255
    n_l, n_r = scales
    at = 256 + 2 * (pad(4 * n_l) + pad(4 * n_r))
    return ws[at:at + rows * ld].view(rows, ld).cpu().numpy()


# columns: whole blocks of 256, 128 and 64, one more, few, not a multiple of eight; contraction entries: below and past the rows
# that a block's lanes cover at once (8 to 32) and in one step of four, past the 64 rows of a block of the two-launch preparation
@pytest.mark.parametrize("m,k", [(256, 64), (257, 1040), (128, 272), (130, 80), (64, 1040), (72, 304), (40, 16), (12, 96), (1000, 48)])
@pytest.mark.parametrize("gran", ["tensor", "channel"])
@pytest.mark.parametrize("fmt", FORMATS)
def test_codes_in_the_operands_own_order(m, k, gran, fmt):
    """Bit for bit the oracle's, transposed, prepared alone and in a batch; beside ordinary columns some of zeros (a scale of 1) and
    some whose scale lies outside the range of the two-wide quotient, on either side."""
    L, R = draw((m, k), 20), draw((24, k), 21)
    if gran == "channel":
        L[3], L[m - 1], L[8] = 0.0, L[m - 1] * 1e-25, L[8] * 1e25
    (_k, lo), (_r, ro) = stored(L, True), stored(R, True)
    x = L.float().cpu().numpy()[None]
    delta = oracle.scale(x, fmt, gran)
    want = oracle.quantize(x, fmt, delta)[0].T
    plan = qm.ProbePlan(lo, ro, fmt, fmt, gran, gran)
    plan.launch(lo, ro)
    batch = qm.ProbeBatch([(lo, ro, fmt, fmt, gran, gran), (ro, lo, fmt, fmt, gran, gran)])
    batch.launch()
    torch.cuda.synchronize()
    n = (m, 24) if gran == "channel" else (1, 1)
    for ws in (plan.ws, batch._ws[0]):
        assert (kept_codes(ws, n, k, qm.binding.qm_code_ld(m))[:, :m] == want).all()


@pytest.mark.parametrize("m,n,k", [(300, 72, 96), (1040, 40, 4096)])
def test_columns_without_an_ordinary_scale_in_the_record(m, n, k):
    L, R = draw((m, k), 22), draw((n, k), 23, 0.05)
    L[5], L[17], R[2] = 0.0, L[17] * 1e-25, 0.0
    (_k, lo), (_r, ro) = stored(L, True), stored(R, True)
    for f in FORMATS:
        want = oracle.probe(L.float().cpu().numpy(), R.float().cpu().numpy().T, f, f, "channel", "channel")
        got = qm.qm_probe_layer(lo, ro, f, f, "channel", "channel")
        assert got.device_error == 0
        assert_record_close(got.record(), want)


@pytest.mark.parametrize("a,b", [(272, 80), (1040, 528)])
def test_one_memory_in_both_orientations(a, b):
    """The same tensor contracted over either dimension in one batch, one use rounded stochastically, as the left and as the right
    operand: what is shared (max|x|, the codes rounded to nearest) must be right for each."""
    T, U, V = draw((a, b), 24), draw((136, b), 25, 0.05), draw((136, a), 26, 0.05)
    (_t, over_b), (_u, u), (_v, v) = stored(T, False), stored(U, False), stored(V, True)
    over_a = qm.operand_of(_t, -2)
    uses = [(over_b, u, "rtne"), (over_a, v, "rtne"), (over_a, v, "stochastic_l"), (over_b, u, "stochastic_l"), (v, over_a, "stochastic_r"),
            (u, over_b, "rtne"), (v, over_a, "rtne"), (over_b, u, "stochastic_both")]
    probes = [(lo, ro, f, f, g, g, rnd) for f, g in (("e4m3", "tensor"), ("int8", "tensor"), ("e5m2", "channel")) for lo, ro, rnd in uses]
    batch = qm.ProbeBatch([p[:6] for p in probes])
    for i, p in enumerate(probes):
        batch.cfg[i] = binding._cfg(*p[2:6], "bf16", p[6], 9)
    batch.launch()
    t = T.float().cpu().numpy()
    against = {id(u): U.float().cpu().numpy().T, id(v): V.float().cpu().numpy().T}
    for p, got in zip(probes, batch.results()):
        same(got, qm.qm_probe_layer(*p[:6], rounding=p[6], seed=9))
        if p[6] == "rtne" and p[0] in (over_a, over_b):
            assert_record_close(got.record(), oracle.probe(t if p[0] is over_b else t.T, against[id(p[1])], *p[2:6]))
