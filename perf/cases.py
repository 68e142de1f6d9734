"""Performance cases of the library: what a program that serves or quantizes a model has it do, call by call.

A case is a dict of plain values. Its "kind" says which entry points one pass goes through:

  gemv      goq_gemv, decode linears called one by one (the caller's attention and norms sit in between, so every linear
            has an input of its own). With "inner" > 0 the pass is a whole decoder layer: q, k, v, o, gate, up, down
            (hidden k, key/value width n, MLP width inner); otherwise one n x k linear.
  chain     goq_gemv_sequence, a decode step of "layers" decoder layers in one call: k and v read what q reads, o reads v's
            output, gate and up read o's, down reads up's, the next layer's q, k, v read down's.
  gemm      goq_gemm on bf16 activations: prefill, or a decode batch above what goq_gemv takes. Shapes as for gemv.
  a8        the integer path on a vision transformer's linears: fp32 activations quantized to int8 per token
            (goq_quantize_activations) and one integer linear n x k; with "inner" > 0 the MLP block: quantize, k -> inner
            with the requantising epilogue (goq_gemm_i8_requant), inner -> n (goq_gemm).
  quantize  goq_quantize_geo and goq_pack of one fp32 weight matrix: the path from a checkpoint to packed weights.
  ref       goq_solve_ref: REF-mode coefficients of one weight matrix from m calibration rows.
"""
import math

import torch

from paper_2605_26092_b200 import goq

# ---------------------------------------------------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------------------------------------------------


def listed():
    return [
        # the smallest call: one 256 x 256 linear, group 64, a batch of 8; launches and host work are all there is
        {"name": "gemv 256x256 b8", "kind": "gemv", "n": 256, "k": 256, "inner": 0, "m": 8, "wbits": 3, "group": 64, "out": "f32"},
        # a decoder layer of the 7B shapes, one sequence, call by call: single-user decoding
        {"name": "gemv 7B layer b1", "kind": "gemv", "n": 4096, "k": 4096, "inner": 11008, "m": 1, "wbits": 3, "group": 128, "out": "bf16"},
        # the same layer with 16 sequences in flight, the largest batch of the decode entry point
        {"name": "gemv 7B layer b16", "kind": "gemv", "n": 4096, "k": 4096, "inner": 11008, "m": 16, "wbits": 3, "group": 128, "out": "bf16"},
        # a decoder layer of the 70B shapes (grouped key/value heads) at four bits, four sequences
        {"name": "gemv 70B layer W4 b4", "kind": "gemv", "n": 1024, "k": 8192, "inner": 28672, "m": 4, "wbits": 4, "group": 128, "out": "f32"},
        # the decode step of the whole 32-layer 7B stack in one call: the library's headline workload
        {"name": "chain 7B 32 layers b1", "kind": "chain", "n": 4096, "k": 4096, "inner": 11008, "layers": 32, "m": 1, "wbits": 3, "group": 128},
        # a few layers of it (a pipeline stage) for four sequences
        {"name": "chain 7B 4 layers b4", "kind": "chain", "n": 4096, "k": 4096, "inner": 11008, "layers": 4, "m": 4, "wbits": 3, "group": 128},
        # continuous batching: 64 decode tokens through the 70B layer, between decode and prefill
        {"name": "gemm 70B layer m64", "kind": "gemm", "n": 1024, "k": 8192, "inner": 28672, "m": 64, "wbits": 3, "group": 128, "out": "bf16"},
        # prefill of a 2048-token prompt through a 7B layer
        {"name": "gemm 7B layer m2048", "kind": "gemm", "n": 4096, "k": 4096, "inner": 11008, "m": 2048, "wbits": 3, "group": 128, "out": "bf16"},
        # a ragged prompt through a narrow four-bit linear (key/value projection of grouped heads)
        {"name": "gemm 1024x8192 W4 m777", "kind": "gemm", "n": 1024, "k": 8192, "inner": 0, "m": 777, "wbits": 4, "group": 128, "out": "f32"},
        # the MLP block of ViT-B/16 on a batch of 64 images of 197 tokens, int8 activations
        {"name": "a8 ViT MLP 64 images", "kind": "a8", "n": 768, "k": 768, "inner": 3072, "m": 64 * 197, "wbits": 3, "group": 64, "out": "bf16"},
        # quantizing a checkpoint: one 7B MLP matrix from fp32 to packed
        {"name": "quantize 11008x4096", "kind": "quantize", "n": 11008, "k": 4096, "m": 0, "wbits": 3, "group": 128},
        # REF-mode refinement of one 7B attention matrix on 256 calibration rows
        {"name": "ref 4096x4096 m256", "kind": "ref", "n": 4096, "k": 4096, "m": 256, "wbits": 3, "group": 128},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _width(rng, lo, hi, step):
    """A size between lo and hi, log-uniform; a multiple of `step`."""
    return max(step, _log_int(rng, lo, hi) // step * step)


def draw(rng):
    """One more case of the same ranges: any output width (odd ones among them), any input width the group size allows."""
    kind = rng.choice(["gemv", "gemv", "gemv", "chain", "chain", "gemm", "gemm", "gemm", "a8", "a8", "quantize", "ref"])
    group = rng.choice([32, 64, 64, 128, 128, 128])
    wbits = rng.choice([2, 3, 3, 4])
    out = rng.choice(["f32", "bf16"])
    if kind == "gemv":
        layer = rng.random() < 0.3
        k = _width(rng, 256, 8192 if layer else 16384, group)
        n = _log_int(rng, 256, 28672) if not layer else _width(rng, max(128, k // 8), k, 128)
        inner = _width(rng, 2 * k, 3.5 * k, group) if layer else 0
        return {"kind": kind, "n": n, "k": k, "inner": inner, "m": rng.randint(1, 16), "wbits": wbits, "group": group, "out": out}
    if kind == "chain":
        k = _width(rng, 512, 4096, 128)
        return {"kind": kind, "n": _width(rng, max(128, k // 4), k, 128), "k": k, "inner": _width(rng, 2 * k, 2.9 * k, 128),
                "layers": _log_int(rng, 1, 24), "m": rng.randint(1, 4), "wbits": rng.choice([2, 3]), "group": group}
    if kind == "gemm":
        k, n = _width(rng, 512, 11008, group), _log_int(rng, 512, 16384)
        m = min(_log_int(rng, 17, 4096), 400_000_000_000 // (n * k))
        return {"kind": kind, "n": n, "k": k, "inner": 0, "m": m, "wbits": wbits, "group": group, "out": out}
    if kind == "a8":
        k = rng.choice([192, 384, 768, 1024])
        group = rng.choice([32, 64])
        images = _log_int(rng, 1, 64)
        if wbits == 4 or rng.random() < 0.5:   # one linear; at four bits the int32 bound ends the widths at 1040
            return {"kind": kind, "n": rng.choice([k, 3 * k, 4 * k, 1000]), "k": k, "inner": 0, "m": images * 197, "wbits": wbits,
                    "group": group, "out": out}
        return {"kind": kind, "n": k, "k": k, "inner": 4 * k, "m": images * 197, "wbits": wbits, "group": group, "out": out}
    k = _width(rng, 512, 8192, group)
    n = _log_int(rng, 512, 8192)
    m = _log_int(rng, 32, 512) if kind == "ref" else 0
    return {"kind": kind, "n": n, "k": k, "m": m, "wbits": wbits, "group": group}


def _linears(case):
    """(n, k, input) of the linears of one pass; linears with the same `input` share their activations."""
    n, k, inner = case["n"], case["k"], case["inner"]
    if not inner:
        return [(n, k, 0)]
    return [(k, k, 0), (n, k, 0), (n, k, 0), (k, k, 1), (inner, k, 2), (inner, k, 2), (k, inner, 3)]


# ---------------------------------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------------------------------


def _rng(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _codes(w, group, wbits):
    """Codes of the weights w [n][k]: nearest state of the asymmetric lattice after scaling by the group's largest.
    Returns the codes [n][k] and the mean square of the states."""
    emax = (1 << (wbits - 1)) - 1
    neg = [-2.0 ** -e for e in range(emax + 1)]                    # code 2^(b-1) + e
    pos = [2.0 ** -e for e in range(emax)]                         # code e; code emax is the zero
    states = torch.tensor(neg + [0.0] + pos[::-1], device="cuda")  # ascending
    code = torch.tensor([(1 << (wbits - 1)) + e for e in range(emax + 1)] + [emax] + list(range(emax))[::-1],
                        dtype=torch.uint8, device="cuda")
    edges = (states[1:] + states[:-1]) / 2
    v = w.view(-1, group)
    at = torch.bucketize(v / v.abs().amax(dim=1, keepdim=True), edges, out_int32=True)
    return code[at].view(w.shape), float(states[at].square().mean())


def _fields(n, k, group, wbits, gen, w=None):
    """Quantizer output of one matrix (normally distributed if none is given): codes, exchange records (any of the 64),
    coefficients of a layer with unit gain."""
    codes, ms = _codes(torch.randn((n, k), device="cuda", generator=gen) if w is None else w, group, wbits)
    meta = torch.randint(0, 64, (n, k // 8), dtype=torch.uint8, device="cuda", generator=gen)
    c = torch.randn((n, k // group, 2), device="cuda", generator=gen)
    c[..., 0] = 1.0 + 0.1 * c[..., 0]   # the first coefficient follows the group's scale, the second is a correction
    c[..., 1] *= 0.3
    coef = (c * (1.1 * ms * k) ** -0.5).to(torch.float16)
    return codes, meta, coef


def _packed(n, k, group, wbits, gen):
    codes, meta, coef = _fields(n, k, group, wbits, gen)
    d = goq.desc(n, k, group, wbits)
    packed = torch.empty(goq.packed_bytes(d), dtype=torch.uint8, device="cuda")
    goq.pack(d, codes, meta, coef, packed)
    return d, packed, coef


def _workspace(nbytes):
    if not nbytes:
        return None
    ws = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    goq.workspace_init(ws)
    return ws


def _weights(n, k, gen):
    """fp32 weights ~N(0, 0.02), one input channel in a hundred scaled by 20 (outlier channels)."""
    w = torch.randn((n, k), device="cuda", generator=gen) * 0.02
    hot = torch.rand(k, device="cuda", generator=gen) < 0.01
    return w * torch.where(hot, 20.0, 1.0)


def _int_coefficients(coef):
    """8-bit symmetric coefficient integers with one fp32 scale per output channel and basis."""
    c = coef.float()
    sc = c.abs().amax(dim=1) / 127.0                                # [n][2]
    return torch.round(c / sc[:, None, :]).clamp(-127, 127).to(torch.int8), sc.contiguous()


_TORCH = {"f32": torch.float32, "bf16": torch.bfloat16}
_GOQ = {"f32": goq.F32, "bf16": goq.BF16}


def prepare(case, seed):
    gen = _rng(seed)
    kind, m, group, wbits = case["kind"], case["m"], case["group"], case["wbits"]
    if kind in ("gemv", "gemm"):
        out = case["out"]
        linears = _linears(case)
        xs = {i: torch.randn((m, k), device="cuda", generator=gen).to(torch.bfloat16) for _, k, i in linears}
        op = goq.OP_GEMV if kind == "gemv" else goq.OP_GEMM
        calls, need = [], 0
        for n, k, i in linears:
            d, packed, _ = _packed(n, k, group, wbits, gen)
            need = max(need, goq.workspace_bytes(d, op, m))
            calls.append((d, packed, xs[i], torch.empty((m, n), dtype=_TORCH[out], device="cuda")))
        return {"kind": kind, "m": m, "out": _GOQ[out], "calls": calls, "ws": _workspace(need)}
    if kind == "chain":
        x = torch.randn((m, case["k"]), device="cuda", generator=gen).to(torch.bfloat16)
        widths = [n for n, _, _ in _linears(case)] * case["layers"]
        block = torch.zeros(m * sum(widths), dtype=torch.bfloat16, device="cuda")   # every linear's output, one after another
        ys = [y.view(m, -1) for y in torch.split(block, [m * w for w in widths])]
        items, keep = [], [x]
        for layer in range(case["layers"]):
            q, k_, v, o, gate, up, down = ys[7 * layer:7 * layer + 7]
            first = x if layer == 0 else ys[7 * layer - 1]
            # o reads v's output (attention is the caller's); a narrower v is topped up from q, which has o's input width
            reads = [first, first, first, v if case["n"] == case["k"] else q, o, o, up]
            for (n, k, _), src, y in zip(_linears(case), reads, (q, k_, v, o, gate, up, down)):
                d, packed, _ = _packed(n, k, group, wbits, gen)
                keep.append(packed)
                items.append((d, packed, src, m, y, goq.BF16, False))
        return {"kind": kind, "seq": goq.make_sequence(items), "ws": _workspace(goq.sequence_workspace_bytes(len(items))),
                "block": block, "keep": keep}
    if kind == "a8":
        x = torch.randn((m, case["k"]), device="cuda", generator=gen)
        shapes = [(case["inner"], case["k"]), (case["n"], case["inner"])] if case["inner"] else [(case["n"], case["k"])]
        layers = []
        for n, k in shapes:
            d, packed, coef = _packed(n, k, group, wbits, gen)
            cq, sc = _int_coefficients(coef)
            layers.append((d, packed, cq, sc))

        def empty(shape, dtype):
            return torch.empty(shape, dtype=dtype, device="cuda")
        s = {"kind": kind, "m": m, "k": case["k"], "x": x, "layers": layers, "out": _GOQ[case["out"]],
             "xq": empty((m, case["k"]), torch.int8), "sx": empty((m,), torch.float32), "y": empty((m, case["n"]), _TORCH[case["out"]])}
        if case["inner"]:
            s.update(h=empty((m, case["inner"]), torch.float32), amax=empty((m,), torch.float32),
                     hq=empty((m, case["inner"]), torch.int8), sh=empty((m,), torch.float32))
        return s
    n, k = case["n"], case["k"]
    w = _weights(n, k, gen)
    d = goq.desc(n, k, group, wbits)
    if kind == "quantize":
        return {"kind": kind, "d": d, "w": w,
                "codes": torch.empty((n, k), dtype=torch.uint8, device="cuda"),
                "meta": torch.empty((n, k // 8), dtype=torch.uint8, device="cuda"),
                "coef": torch.empty((n, k // group, 2), dtype=torch.float16, device="cuda"),
                "packed": torch.empty(goq.packed_bytes(d), dtype=torch.uint8, device="cuda")}
    codes, meta, _ = _fields(n, k, group, wbits, gen, w)
    xc = torch.randn((m, k), device="cuda", generator=gen)
    return {"kind": kind, "d": d, "w": w, "codes": codes, "meta": meta, "x": xc, "m": m,
            "coef": torch.empty((n, k // group, 2), dtype=torch.float16, device="cuda"),
            "c": torch.empty((n, k // group, 2), dtype=torch.float64, device="cuda")}


# ---------------------------------------------------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------------------------------------------------


def run(s):
    kind = s["kind"]
    if kind == "gemv":
        for d, packed, x, y in s["calls"]:
            goq.gemv(d, packed, x, s["m"], y, s["out"], ws=s["ws"])
        return [y for _, _, _, y in s["calls"]]
    if kind == "gemm":
        for d, packed, x, y in s["calls"]:
            goq.gemm(d, packed, x, s["m"], goq.BF16, y=y, y_dtype=s["out"], ws=s["ws"])
        return [y for _, _, _, y in s["calls"]]
    if kind == "chain":
        goq.gemv_sequence(s["seq"], s["ws"])
        return s["block"]
    if kind == "a8":
        goq.quantize_activations(s["x"], goq.F32, s["m"], s["k"], s["xq"], s["sx"])
        x, sx = s["xq"], s["sx"]
        if len(s["layers"]) == 2:
            d, packed, cq, sc = s["layers"][0]
            goq.gemm_i8_requant(d, packed, x, s["m"], sx, cq, sc, s["h"], s["amax"], s["hq"], s["sh"])
            x, sx = s["hq"], s["sh"]
        d, packed, cq, sc = s["layers"][-1]
        goq.gemm(d, packed, x, s["m"], goq.I8, y=s["y"], y_dtype=s["out"], sx=sx, cq=cq, sc=sc)
        return {"xq": s["xq"], "sx": s["sx"], "y": s["y"], **({"hq": s["hq"], "sh": s["sh"]} if len(s["layers"]) == 2 else {})}
    if kind == "quantize":
        goq.quantize_geo(s["d"], s["w"], s["codes"], s["meta"], s["coef"])
        goq.pack(s["d"], s["codes"], s["meta"], s["coef"], s["packed"])
        return {"codes": s["codes"], "meta": s["meta"], "coef": s["coef"], "packed": s["packed"]}
    goq.solve_ref(s["d"], s["w"], s["codes"], s["meta"], s["x"], s["m"], 1e-4, s["coef"], s["c"])
    return {"coef": s["coef"], "c": s["c"]}


# ---------------------------------------------------------------------------------------------------------------------
# what a pass cannot do without, and how far two correct implementations can be apart
# ---------------------------------------------------------------------------------------------------------------------


def work(case):
    """Weights at the format's own bits per weight (wbits + 0.75 + 32 / group), activations and outputs once each."""
    kind, m, group, wbits = case["kind"], case["m"], case["group"], case["wbits"]

    def weights(n, k):
        return goq.algorithmic_bytes(goq.desc(n, k, group, wbits))
    if kind in ("gemv", "gemm", "chain"):
        linears = _linears(case)
        out = 4 if case.get("out") == "f32" else 2
        times = case.get("layers", 1)
        inputs = sum(m * k * 2 for k in {i: k for _, k, i in linears}.values())
        nbytes = times * (sum(weights(n, k) + m * n * out for n, k, _ in linears) + inputs)
        return {"bytes": nbytes, "flops": times * sum(2 * m * n * k for n, k, _ in linears)}
    if kind == "a8":
        n, k, inner = case["n"], case["k"], case["inner"]
        out = 4 if case["out"] == "f32" else 2
        nbytes = m * k * 4 + m * k + m * 4 + m * n * out
        shapes = [(inner, k), (n, inner)] if inner else [(n, k)]
        nbytes += sum(weights(a, b) for a, b in shapes) + (m * inner * 4 + m * inner if inner else 0)
        return {"bytes": nbytes, "flops": sum(4 * m * a * b for a, b in shapes)}   # two integer accumulators
    n, k = case["n"], case["k"]
    fields = n * k + n * (k // 8) + n * (k // group) * 4
    if kind == "quantize":
        return {"bytes": 4 * n * k + fields + weights(n, k), "flops": 0}
    return {"bytes": 4 * n * k + fields + 4 * m * k + 16 * n * (k // group), "flops": 6 * min(m, group) * n * k}


def tolerance(case):
    kind, m = case["kind"], case["m"]
    if kind == "gemv":
        # fp32 outputs: exact or 2^-15-rounded products, fp32 sums. bf16 outputs: results that far apart round to
        # neighbouring values now and then
        return {"rel": 2e-5, "max": 1e-3} if case["out"] == "f32" else {"rel": 3e-3, "max": 1e-2}
    if kind == "chain":
        # each linear reads bf16 outputs of an earlier one: roundings that differ once stay different, 2^-9 / sqrt(3) per
        # linear of the longest path (four a layer), added in squares and twice (two implementations)
        return {"rel": min(2e-2, 1.2e-3 * math.sqrt(2 * 4 * case["layers"])), "max": 0.2}
    if kind == "gemm":
        # 16-bit weight operand: 2^-12 / sqrt(3) per weight, independent; bf16 outputs as above
        return {"rel": 5e-4 if case["out"] == "f32" else 3e-3, "max": 1e-2}
    if kind == "a8":
        # integers are exact up to the last step, s_x 2^-emax (s_1 ACC_1 + s_2 ACC_2) in fp32; a hidden value on a rounding
        # boundary may then go to the other int8, and bf16 outputs to a neighbour
        return {"rel": 3e-3 if case["out"] == "bf16" else 1e-4, "max": 1e-2, "differ": 1e-4}
    if kind == "quantize":
        # float64 throughout: codes agree; a record whose scores agree to the last bits, or a coefficient on a rounding
        # boundary of fp16, may differ
        return {"rel": 1e-6, "max": 2e-3, "differ": 1e-6}
    # float64 normal equations: the fp16 pair differs only where the float64 value sits on a rounding boundary
    return {"rel": 1e-5, "max": 1e-3}
