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
    """One tensor as it lies and flipped, rounded to nearest and stochastically, under both kinds of scales: shared
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
