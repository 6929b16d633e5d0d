"""Timed workloads of the quantized-matmul error probe, through the package's public entry points.

`listed()` holds the workloads that stand for the library's use: the measurement passes over the
matmuls of an encoder layer (probes issued together), single probes from the smallest to ragged
ones, and the steps of the probe on their own (quantize, tensor analysis, stand-alone products).
`draw(rng)` gives further ones of the same kinds and ranges.
"""
import math

import torch

from paper_2408_02897_b200 import binding as qm

LARGEST = 16384 * 4096 * 1024          # multiply-adds of one product, at most
GRAD_STD = 1e-3                        # upstream gradients, as in workloads.py
WEIGHT_STD = 0.02


# ------------------------------------------------------------------------------- the workloads
def listed():
    return [
        # The smallest call: one fp32 product of a layer being looked at by itself, per-tensor
        # E4M3 against an fp32 reference, in a loop that keeps its workspace.
        dict(name="probe fp32 128x256x256", kind="probe", m=128, n=256, k=256, batch=1, dtype="fp32", direction="forward",
             left="e4m3", right="e4m3", gran="tensor", rounding="rtne", values="normal", planned=True),
        # The worked example of the method: Student-t matrices, a scale per vector, from a notebook or
        # script that makes the one call and reads the record.
        dict(name="probe Student-t 512", kind="probe", m=512, n=512, k=512, batch=1, dtype="bf16", direction="forward",
             left="int8", right="int8", gran="channel", rounding="rtne", values="student-t", planned=False),
        # A weight gradient with extents off every tile edge; the gradient operand is rounded
        # stochastically, both operands are stored with the contraction strided.
        dict(name="probe wgrad ragged", kind="probe", m=770, n=3078, k=2032, batch=1, dtype="bf16", direction="wgrad",
             left="e4m3", right="e5m2", gran="tensor", rounding="stochastic_r", values="normal", planned=True),
        # BERT-base forward matmuls, batch 8 x seq 512, E4M3 and INT8: an ordinary pass.
        dict(name="pass BERT-base forward", kind="pass", examples=8, seq=512, hidden=768, ffn=3072, heads=0,
             formats="e4m3,int8", directions="forward", weights="tensor", host=False),
        # One BERT-large layer forward and backward in one format, per-channel scales on the weights.
        dict(name="pass BERT-large layer", kind="pass", examples=32, seq=512, hidden=1024, ffn=4096, heads=0,
             formats="e4m3", directions="all", weights="channel", host=False),
        # One layer of the full sweep: every projection and attention product, forward and backward,
        # in all three formats: the largest pass.
        dict(name="pass sweep layer", kind="pass", examples=32, seq=512, hidden=1024, ffn=4096, heads=16,
             formats="e4m3,e5m2,int8", directions="all", weights="tensor", host=False),
        # The BERT-base pass over tensors that another program left in pinned host memory.
        dict(name="pass BERT-base from host", kind="pass", examples=8, seq=512, hidden=768, ffn=3072, heads=0,
             formats="e4m3,int8", directions="forward", weights="tensor", host=True),
        # Outlier study of one product: heavy-tailed activations with scaled feature channels, each
        # format with both scale granularities.
        dict(name="outliers FFN1", kind="outliers", tokens=16384, hidden=1024, ffn=4096),
        # Scale + quantize of activations, one scale per token (contraction contiguous).
        dict(name="quantize rows 16384x4096", kind="quantize", rows=16384, cols=4096, dtype="bf16", strided=False,
             formats="int8", gran="channel", stochastic=False, values="normal"),
        # Scale + quantize of a gradient for a weight-gradient product: the contraction is the strided
        # dimension, stochastic rounding, the contraction-major bf16 copy wanted beside the codes.
        dict(name="quantize gradient strided", kind="quantize", rows=16384, cols=1024, dtype="bf16", strided=True,
             formats="e5m2", gran="tensor", stochastic=True, values="gradient"),
        # Statistics of a tensor and its element-wise quantization error: the input of FFN2 (behind the GELU).
        dict(name="analyse 16384x4096", kind="analyse", rows=16384, cols=4096, dtype="bf16", fmt="e4m3", gran="tensor"),
        # The steps apart: 8-bit product, reference, denominator, then the metric on the written matrices.
        dict(name="products 4096x3072x768", kind="products", m=4096, n=3072, k=768, batch=1, fmt="e4m3", gran="channel"),
    ]


def _log(rng, lo, hi, step=1):
    """An integer in [lo, hi], even over the logarithm, a multiple of step."""
    x = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return max(lo, min(hi, int(round(x / step)) * step))


def draw(rng):
    kind = rng.choice(["probe"] * 4 + ["pass"] * 3 + ["outliers", "quantize", "quantize", "analyse", "products"])
    fmts = ("e4m3", "e5m2", "int8")
    if kind == "probe":
        fp32 = rng.random() < 0.3
        direction = rng.choice(["forward", "dgrad", "wgrad"])
        fmt = rng.choice(fmts)
        grad = "int8" if fmt == "int8" else "e5m2"
        c = dict(kind=kind, m=_log(rng, 32, 1024 if fp32 else 16384), n=_log(rng, 32, 1024 if fp32 else 4096),
                 k=_log(rng, 32, 1024) if fp32 else _log(rng, 32, 4096, 16), batch=1, dtype="fp32" if fp32 else "bf16",
                 direction=direction, left=grad if direction == "dgrad" else fmt, right=grad if direction == "wgrad" else fmt,
                 gran=rng.choice(["tensor", "channel"]), rounding="rtne", values=rng.choice(["normal", "student-t"]),
                 planned=rng.random() < 0.6)
        if direction != "forward" and rng.random() < 0.5:
            c["rounding"] = "stochastic_l" if direction == "dgrad" else "stochastic_r"
        if not fp32 and rng.random() < 0.25:         # a batched product of attention
            s, d = _log(rng, 64, 512, 16), 64
            c.update(m=s, n=rng.choice([s, d]), batch=_log(rng, 8, 512))
            c["k"] = d if c["n"] == s else s
        while c["m"] * c["n"] * c["k"] * c["batch"] > LARGEST:
            c["m"] = max(32, c["m"] // 2)
        return c
    if kind == "pass":
        heads = _log(rng, 4, 16)
        host = rng.random() < 0.25
        seq = _log(rng, 64, 512, 16)
        return dict(kind=kind, examples=max(1, _log(rng, 256, 4096 if host else 16384) // seq), seq=seq, hidden=64 * heads,
                    ffn=256 * heads, heads=heads if rng.random() < 0.5 else 0,
                    formats=rng.choice(["e4m3", "int8", "e4m3,int8", "e4m3,e5m2", "e4m3,e5m2,int8"]),
                    directions=rng.choice(["forward", "all"]), weights=rng.choice(["tensor", "channel"]), host=host)
    if kind == "outliers":
        return dict(kind=kind, tokens=_log(rng, 256, 16384), hidden=_log(rng, 256, 1024, 16), ffn=_log(rng, 512, 4096, 8))
    if kind == "quantize":
        stochastic = rng.random() < 0.35
        return dict(kind=kind, rows=_log(rng, 128, 16384), cols=_log(rng, 128, 4096), dtype=rng.choice(["bf16", "bf16", "fp32"]),
                    strided=rng.random() < 0.5, formats=rng.choice(fmts) if stochastic else rng.choice(fmts + ("e4m3,e5m2,int8",)),
                    gran=rng.choice(["tensor", "channel"]), stochastic=stochastic, values="gradient" if stochastic else "normal")
    if kind == "analyse":
        return dict(kind=kind, rows=_log(rng, 128, 16384), cols=_log(rng, 128, 4096), dtype=rng.choice(["bf16", "fp32"]),
                    fmt=rng.choice(fmts), gran=rng.choice(["tensor", "channel"]))
    return dict(kind=kind, m=_log(rng, 64, 8192), n=_log(rng, 64, 4096), k=_log(rng, 64, 4096, 16), batch=1, fmt=rng.choice(fmts),
                gran=rng.choice(["tensor", "channel"]))


# ------------------------------------------------------------------------------- inputs
_DTYPE = {"bf16": torch.bfloat16, "fp32": torch.float32}


class _Inputs:
    """Seeded tensors on the GPU, rows padded to a multiple of 8 elements as the library asks."""

    def __init__(self, seed):
        self.g = torch.Generator(device="cuda")
        self.g.manual_seed(seed)

    def _randn(self, *shape):
        return torch.randn(shape, generator=self.g, device="cuda")

    def tensor(self, shape, values, dtype="bf16"):
        if values == "student-t":                    # three degrees of freedom
            x = self._randn(*shape) / torch.sqrt(sum(self._randn(*shape).square_() for _ in range(3)) / 3.0)
        elif values == "outliers":                   # the same, 1 % of the feature columns times 50
            x = self.tensor(shape, "student-t", "fp32").contiguous()
            cols = torch.randperm(shape[-1], generator=self.g, device="cuda")[:max(1, shape[-1] // 100)]
            x[:, cols] *= 50.0
        elif values == "gelu":
            x = torch.nn.functional.gelu(self._randn(*shape))
        else:
            x = self._randn(*shape)
            if values in ("gradient", "weight"):
                x *= GRAD_STD if values == "gradient" else WEIGHT_STD
        pad = -shape[-1] % 8
        out = torch.zeros(*shape[:-1], shape[-1] + pad, dtype=_DTYPE[dtype], device="cuda")[..., :shape[-1]]
        return out.copy_(x)


# L.R of a forward, dgrad or wgrad product: which dimension contracts, and what the operands hold
_LAYOUT = {"forward": (-1, -2), "dgrad": (-1, -1), "wgrad": (-2, -2)}
_HOLDS = {"forward": ("normal", "weight"), "dgrad": ("gradient", "weight"), "wgrad": ("normal", "gradient")}


def _stored(rows, contract, contract_dim, batch):
    shape = (rows, contract) if contract_dim == -1 else (contract, rows)
    return shape if batch == 1 else (batch, *shape)


def _pass_products(c):
    """The products of a pass: (tensor of L, contracting dim, tensor of R, contracting dim, M, N, K, batch)
    with the tensors by name, and {name: (shape, values)}."""
    M, H, F, S = c["examples"] * c["seq"], c["hidden"], c["ffn"], c["seq"]
    back = c["directions"] == "all"
    tensors = {"X": ((M, H), "normal"), "X2": ((M, F), "normal")}
    products = []
    for name, x, k, n in (("qkv", "X", H, 3 * H), ("attn_out", "X", H, H), ("ffn1", "X", H, F), ("ffn2", "X2", F, H)):
        w, g = "W_" + name, "dY_" + name
        tensors[w] = ((k, n), "weight")
        products.append((x, -1, w, -2, M, n, k, 1))
        if back:
            tensors[g] = ((M, n), "gradient")
            products.append((g, -1, w, -1, M, k, n, 1))
            products.append((x, -2, g, -2, k, n, M, 1))
    if c["heads"]:
        B, D = c["examples"] * c["heads"], H // c["heads"]
        for t in "QKV":
            tensors[t] = ((B, S, D), "normal")
        tensors["P"] = ((B, S, S), "probabilities")
        products += [("Q", -1, "K", -1, S, S, D, B), ("P", -1, "V", -2, S, D, S, B)]
        if back:
            tensors["dS"], tensors["dO"] = ((B, S, S), "gradient"), ((B, S, D), "gradient")
            products += [("dS", -1, "K", -2, S, D, S, B), ("dS", -2, "Q", -2, S, D, S, B),
                         ("dO", -1, "V", -1, S, S, D, B), ("P", -2, "dO", -2, S, D, S, B)]
    return products, tensors


def _format_of(tensor, fmt):
    return "e5m2" if tensor[0] == "d" and fmt != "int8" else fmt       # gradients: E5M2 in an FP8 pass


def _pass_probes(c, operand):
    """operand(name, contracting dim) -> what the batch takes for an operand (a tuple of arguments)."""
    products, _ = _pass_products(c)
    formats = c["formats"].split(",")
    # the formats of a product next to one another where the tensors come from the host, else one format
    # after the other over the whole layer, as sweep.py issues them
    order = [(p, f) for p in products for f in formats] if c["host"] else [(p, f) for f in formats for p in products]
    gran = {True: c["weights"], False: "tensor"}
    return [(*operand(l, cl), *operand(r, cr), _format_of(l, f), _format_of(r, f), "tensor", gran[r[0] == "W"], "bf16")
            for (l, cl, r, cr, *_), f in order]


def _record_views(out, n):
    """The records of a plan's result buffer, field by field, as views of it."""
    f = out.view(torch.float64).view(n, 7)
    names = ("sum_be", "max_be", "sum_diff2", "sum_ref2", "sum_den2")
    d = {k: f[:, i] for i, k in enumerate(names)}
    d["count"] = out.view(torch.int64).view(n, 7)[:, 5]
    d["device_error"] = out.view(torch.int32).view(n, 14)[:, 12]
    return d


# ------------------------------------------------------------------------------- what a program has in hand
def prepare(case, seed):
    make = _Inputs(seed)
    kind = case["kind"]
    if kind == "probe":
        cl, cr = _LAYOUT[case["direction"]]
        vl, vr = _HOLDS[case["direction"]]
        if case["values"] == "student-t":
            vl = vr = "student-t"
        L = make.tensor(_stored(case["m"], case["k"], cl, case["batch"]), vl, case["dtype"])
        R = make.tensor(_stored(case["n"], case["k"], cr, case["batch"]), vr, case["dtype"])
        s = dict(case=case, L=L, R=R, cl=cl, cr=cr, ref="fp32" if case["dtype"] == "fp32" else "bf16")
        s["args"] = (case["left"], case["right"], case["gran"], case["gran"])
        if case["planned"]:
            s["Lo"], s["Ro"] = qm.operand_of(L, cl), qm.operand_of(R, cr)
            s["plan"] = qm.ProbePlan(s["Lo"], s["Ro"], *s["args"], s["ref"], case["rounding"], seed=7)
            s["out"] = _record_views(s["plan"].out, 1)
        return s
    if kind == "pass":
        tensors = {}
        for name, (shape, values) in _pass_products(case)[1].items():
            if values == "probabilities":
                scores = torch.matmul(tensors["Q"], tensors["K"].transpose(1, 2)).float() / math.sqrt(tensors["Q"].shape[-1])
                tensors[name] = torch.softmax(scores, dim=-1).to(torch.bfloat16)
            else:
                tensors[name] = make.tensor(shape, values)
        if case["host"]:
            tensors = {k: t.cpu().pin_memory() for k, t in tensors.items()}
            return dict(case=case, tensors=tensors, batch=qm.HostProbeBatch(_pass_probes(case, lambda t, cd: (tensors[t], cd))))
        batch = qm.ProbeBatch(_pass_probes(case, lambda t, cd: (qm.operand_of(tensors[t], cd),)))
        return dict(case=case, tensors=tensors, batch=batch, out=_record_views(batch.out, batch.n))
    if kind == "outliers":
        X = make.tensor((case["tokens"], case["hidden"]), "outliers")
        W = make.tensor((case["hidden"], case["ffn"]), "weight")
        Xo, Wo = qm.operand_of(X, -1), qm.operand_of(W, -2)
        batch = qm.ProbeBatch([(Xo, Wo, f, f, g, g) for f in ("e4m3", "e5m2", "int8") for g in ("tensor", "channel")])
        return dict(case=case, X=X, W=W, batch=batch, out=_record_views(batch.out, batch.n))
    if kind in ("quantize", "analyse"):
        x = make.tensor((case["rows"], case["cols"]), case.get("values", "gelu"), case["dtype"])
        s = dict(case=case, x=x, op=qm.operand_of(x, -2 if case.get("strided") else -1))
        if kind == "analyse":
            s["ws"] = torch.empty(qm.lib().qm_stats_workspace_bytes(), dtype=torch.uint8, device="cuda")
        return s
    # products: the codes and scales of both operands, and the bf16 operands with their magnitudes
    l, r = (make.tensor((case["batch"], case[d], case["k"]), v) for d, v in (("m", "normal"), ("n", "weight")))
    cl, dl, al, _ = qm.qm_quantize(qm.operand_of(l, -1), case["fmt"], case["gran"], want_abs=True)
    cr, dr, ar, _ = qm.qm_quantize(qm.operand_of(r, -1), case["fmt"], case["gran"], want_abs=True)
    return dict(case=case, l=l, r=r, al=al, ar=ar, cl=cl, dl=dl, cr=cr, dr=dr)


# ------------------------------------------------------------------------------- one pass
def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "probe":
        if case["planned"]:
            s["plan"].launch(s["Lo"], s["Ro"])
            return s["out"]
        rec = qm.qm_probe_layer(qm.operand_of(s["L"], s["cl"]), qm.operand_of(s["R"], s["cr"]), *s["args"], s["ref"],
                                rounding=case["rounding"], seed=7)
        return {**rec.record(), "device_error": rec.device_error}
    if kind == "pass" and case["host"]:
        recs = s["batch"].run()
        rows = [list(r.record().values()) + [r.device_error] for r in recs]
        names = list(recs[0].record()) + ["device_error"]
        return {k: torch.tensor(v, dtype=torch.float64 if isinstance(v[0], float) else torch.int64)
                for k, v in zip(names, map(list, zip(*rows)))}
    if kind in ("pass", "outliers"):
        s["batch"].launch()
        return s["out"]
    if kind == "quantize":
        formats = case["formats"].split(",")
        if len(formats) > 1:
            codes, deltas, _ = qm.qm_quantize_formats(s["op"], formats, case["gran"])
            return {"codes": codes, "delta": deltas}
        copy = case["strided"] and case["dtype"] == "bf16"
        codes, delta, _, kmaj = qm.qm_quantize(s["op"], formats[0], case["gran"], want_kmaj=copy,
                                               stochastic=(7, 1) if case["stochastic"] else None)
        return {"codes": codes, "delta": delta, "copy": kmaj}
    if kind == "analyse":
        stats = qm.qm_tensor_stats(s["op"], s["ws"])
        err = qm.qm_quantize_error(s["op"], case["fmt"], case["gran"], ws=s["ws"])
        return {"sum1": stats.sum1, "sum2": stats.sum2, "sum3": stats.sum3, "sum4": stats.sum4, "max_abs": stats.max_abs,
                **stats.derived(), "error": err.record(), "device_error": stats.device_error | err.device_error}
    q, _ = qm.qm_gemm(s["cl"], case["fmt"], s["dl"], case["gran"], s["cr"], case["fmt"], s["dr"], case["gran"], case["k"])
    c = qm.qm_gemm_ref(s["l"], s["r"])
    d = qm.qm_gemm_ref(s["al"], s["ar"])
    rec = qm.qm_metric(c, q, d)
    return {"q": q, "c": c, "d": d, **rec.record(), "device_error": rec.device_error}


# ------------------------------------------------------------------------------- work and tolerance
_SIZE = {"bf16": 2, "fp32": 4}


def work(case):
    """Inputs read once, outputs written once; multiply-adds of the products that the records need: a
    product's reference and denominator once, an 8-bit product per format (and granularity)."""
    kind = case["kind"]
    if kind == "probe":
        m, n, k, b = case["m"], case["n"], case["k"], case["batch"]
        return dict(bytes=(m + n) * k * b * _SIZE[case["dtype"]] + 56, flops=3 * 2 * m * n * k * b)
    if kind == "pass":
        products, tensors = _pass_products(case)
        nf = len(case["formats"].split(","))
        return dict(bytes=sum(2 * math.prod(shape) for shape, _ in tensors.values()) + 56 * nf * len(products),
                    flops=sum(2 * m * n * k * b * (2 + nf) for *_, m, n, k, b in products))
    if kind == "outliers":
        m, n, k = case["tokens"], case["ffn"], case["hidden"]
        return dict(bytes=2 * (m + n) * k + 6 * 56, flops=2 * m * n * k * (2 + 6))
    if kind == "quantize":
        r, c = case["rows"], case["cols"]
        nf = len(case["formats"].split(","))
        nc, kk = (c, r) if case["strided"] else (r, c)
        copy = 2 * r * c if case["strided"] and case["dtype"] == "bf16" and nf == 1 else 0
        scales = 4 * (nc if case["gran"] == "channel" else 1)
        return dict(bytes=r * c * _SIZE[case["dtype"]] + nf * (nc * qm.qm_code_ld(kk) + scales) + copy, flops=0)
    if kind == "analyse":
        return dict(bytes=case["rows"] * case["cols"] * _SIZE[case["dtype"]], flops=0)
    m, n, k, b = case["m"], case["n"], case["k"], case["batch"]
    return dict(bytes=b * ((m + n) * k * (1 + 2 + 2) + 3 * 4 * m * n), flops=3 * 2 * m * n * k * b)


def tolerance(case):
    """Codes, scales and copies are exact.  Records: four times what they were seen to differ from the
    same arithmetic in 64 bits.  The tensor cores accumulate in fp32 with truncation, so that sums over
    all-positive products are low by an amount that grows with the contraction (sum D^2: 2e-6 at K = 512,
    2.7e-5 at 4096, 1.7e-4 at 16384), and max BE is one element whose numerator cancels (2e-5 at K = 1024,
    9e-5 at 3072, 1.4e-4 at 16384).  fp32 reference: 2e-6.  Tensor analysis: 1e-7 (fp32 terms, fp64 sums)."""
    kind = case["kind"]
    if kind == "quantize":
        return "exact"
    if kind == "analyse":
        return {"rel": 1e-6}
    if case.get("dtype") == "fp32":
        return {"rel": 1e-5}
    if kind == "pass":
        k = max(p[6] for p in _pass_products(case)[0])
    else:
        k = case["hidden"] if kind == "outliers" else case["k"]
    return {"rel": min(7e-4, max(4e-5, 1.2e-7 * k))}


# ------------------------------------------------------------------------------- in 64 bits, plain torch
_QMAX = {"int8": 127.0, "e4m3": 448.0, "e5m2": 57344.0}


def _oriented(t, contract_dim):
    """The operand as [batch, non-contracting, contracting]."""
    t = t.cuda()
    t = t if t.dim() == 3 else t.unsqueeze(0)
    return t if contract_dim == -1 else t.transpose(1, 2)


def _uniform(shape, seed, stream):
    """Draw of every element in C order: word i mod 4 of Philox4x32-10 on block i div 4, its upper 24 bits."""
    n, mask = math.prod(shape), 0xFFFFFFFF
    i = torch.arange((n + 3) // 4, device="cuda", dtype=torch.int64)
    c = [i & mask, i >> 32, torch.full_like(i, stream), torch.zeros_like(i)]
    k0, k1 = seed & mask, (seed >> 32) & mask

    def product(m, x):                               # high and low word of the 64-bit product, in halves
        a, b = (m >> 16) * x, (m & 0xFFFF) * x
        s = ((a & 0xFFFF) << 16) + (b & mask)
        return ((a >> 16) + (b >> 32) + (s >> 32)) & mask, s & mask
    for _ in range(10):
        (h0, l0), (h1, l1) = product(0xD2511F53, c[0]), product(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    return ((torch.stack(c, 1).reshape(-1)[:n] >> 8).double() / 2.0 ** 24).reshape(shape)


def _quantized(x, fmt, gran, draw=None):
    """(values of the codes as float64, scales, the fp32 quotients) of an oriented operand."""
    x = x.float()
    top = x.abs().amax(-1, keepdim=True) if gran == "channel" else x.abs().amax().reshape(1, 1, 1)
    delta = torch.where(top > 0, top / torch.tensor(_QMAX[fmt], device="cuda"), torch.ones_like(top))
    t = x / delta
    a = t.clamp(-_QMAX[fmt], _QMAX[fmt])
    if draw is not None:
        m, emin = {"int8": (0, 0), "e4m3": (3, -6), "e5m2": (2, -14)}[fmt]
        d = a.abs().double()
        e = torch.frexp(d).exponent.double() - 1
        step = torch.ones_like(d) if fmt == "int8" else torch.exp2(e.clamp(min=emin) - m)
        lo = torch.floor(d / step) * step
        v = torch.copysign(lo + step * (draw * step < d - lo), a.double())
    elif fmt == "int8":
        v = a.round().double()
    else:
        v = a.to(torch.float8_e4m3fn if fmt == "e4m3" else torch.float8_e5m2).double()
    return v, delta.double(), t


def _reduce(c, q, d):
    diff = (c - q).abs()
    be = torch.where(d > 0, diff / d, torch.zeros_like(d))
    return [be.sum(), be.max(), (diff * diff).sum(), (c * c).sum(), (d * d).sum()]


def _exact_record(l, r, ql, qr):
    """Eq. 3 sums of oriented operands and their quantized values, blocks of output rows at a time."""
    (vl, dl, _), (vr, dr, _) = ql, qr
    vl, vr = vl * dl, vr * dr
    l, r = l.double(), r.double()
    total = None
    rows = max(1, (1 << 27) // r.shape[1])
    for b in range(0, l.shape[0], max(1, rows // l.shape[1])):
        bs = slice(b, b + max(1, rows // l.shape[1]))
        for i in range(0, l.shape[1], rows):
            x = l[bs, i:i + rows]
            rt = r[bs].transpose(1, 2)
            part = _reduce(x @ rt, vl[bs, i:i + rows] @ vr[bs].transpose(1, 2), x.abs() @ rt.abs())
            total = part if total is None else [max(p, t) if k == 1 else p + t for k, (p, t) in enumerate(zip(part, total))]
    return [float(t) for t in total]


def _record_dict(rows, counts):
    names = ("sum_be", "max_be", "sum_diff2", "sum_ref2", "sum_den2")
    d = {k: torch.tensor([row[i] for row in rows], dtype=torch.float64) for i, k in enumerate(names)}
    d["count"] = torch.tensor(counts, dtype=torch.int64)
    d["device_error"] = torch.zeros(len(rows), dtype=torch.int32)
    return d


def exact(case, seed):
    """What run() returns for these inputs, in 64 bits.  None for the quantize cases: their outputs are bytes
    and fp32 scales that are compared bit for bit."""
    kind = case["kind"]
    if kind == "quantize":
        return None
    with torch.no_grad():
        s = prepare({**case, "planned": False} if kind == "probe" else case, seed)
        if kind == "probe":
            l, r = _oriented(s["L"], s["cl"]), _oriented(s["R"], s["cr"])
            ql = _quantized(l, case["left"], case["gran"], _uniform(l.shape, 7, 0) if case["rounding"] == "stochastic_l" else None)
            qr = _quantized(r, case["right"], case["gran"], _uniform(r.shape, 7, 1) if case["rounding"] == "stochastic_r" else None)
            d = _record_dict([_exact_record(l, r, ql, qr)], [l.shape[0] * l.shape[1] * r.shape[1]])
            return d if case["planned"] else {k: float(v[0]) for k, v in d.items()}
        if kind in ("pass", "outliers"):
            if kind == "pass":
                products = _pass_probes(case, lambda t, cd: (t, cd))
                tensors = s["tensors"]
            else:
                tensors = s
                products = [("X", -1, "W", -2, f, f, g, g) for f in ("e4m3", "e5m2", "int8") for g in ("tensor", "channel")]
            rows, counts = [], []
            for l, cl, r, cr, fl, fr, gl, gr, *_ in products:
                x, y = _oriented(tensors[l], cl), _oriented(tensors[r], cr)
                rows.append(_exact_record(x, y, _quantized(x, fl, gl), _quantized(y, fr, gr)))
                counts.append(x.shape[0] * x.shape[1] * y.shape[1])
            return _record_dict(rows, counts)
        if kind == "analyse":
            x = _oriented(s["x"], -1)
            v, delta, t = _quantized(x, case["fmt"], case["gran"])
            x = x.double()
            n, mean = x.numel(), x.mean()
            m2, m3, m4 = (((x - mean) ** k).mean() for k in (2, 3, 4))
            err, nz = (x - v * delta).abs(), x != 0
            over = nz & (t.abs().double() > _QMAX[case["fmt"]])
            under = nz & ~over & (v == 0)
            mid = nz & ~over & ~under
            re = torch.where(nz, err / x.abs(), torch.zeros_like(x))
            e2 = err * err
            sums = {"sum%d" % k: float((x ** k).sum()) for k in (1, 2, 3, 4)}
            f = {"sum_re": re.sum(), "sum_re_round": re[mid].sum(), "max_re_round": re[mid].max(), "err2_round": e2[mid].sum(),
                 "err2_overflow": e2[over].sum(), "err2_underflow": e2[under].sum(), "sum_x2": (x * x).sum()}
            counts = {"count": n, "n_nonzero": int(nz.sum()), "n_overflow": int(over.sum()), "n_underflow": int(under.sum())}
            return {**sums, "max_abs": float(x.abs().max()), "mean": float(mean), "variance": float(m2),
                    "skew": float(m3 / m2 ** 1.5), "kurtosis": float(m4 / m2 ** 2),
                    "error": {**{k: float(w) for k, w in f.items()}, **counts}, "device_error": 0}
        l, r = s["l"], s["r"]
        (vl, dl, _), (vr, dr, _) = _quantized(l, case["fmt"], case["gran"]), _quantized(r, case["fmt"], case["gran"])
        l, r = l.double(), r.double()
        c, d = l @ r.transpose(1, 2), l.abs() @ r.abs().transpose(1, 2)
        q = (vl * dl) @ (vr * dr).transpose(1, 2)
        names = ("sum_be", "max_be", "sum_diff2", "sum_ref2", "sum_den2")
        return {"q": q, "c": c, "d": d, **{k: float(w) for k, w in zip(names, _reduce(c, q, d))}, "count": c.numel(),
                "device_error": 0}
