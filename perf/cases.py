"""Performance cases of the MoLE library: the calls a program makes, at the sizes it makes them.

Kinds (every case names one):
  layer     one lookup layer, what a model calls between its attention blocks: decode batches of a few tokens up
            to prefills of thousands
  step      the L lookup layers of one decode step in one call
  host      the same step for a caller whose activations live in pinned host memory
  offload   the same step with the tables in pinned host memory and only the looked-up rows crossing the link
  build     the table of one layer from its experts' FFNs (once per model)
  quantize  a table to NF4 / NF3 records (once per model)

Shapes are the repository's workload shapes (inputs.SHAPES) and, for drawn cases, widths and expert counts around
them.  Id streams are Zipf(1.1) over the vocabulary, as in the benchmark.  Where the tables of a full-vocabulary model
would not fit a GPU three times over, the vocabulary is cut; a step looks up the same number of rows either way.
"""
import math

import numpy as np
import torch

from paper_2503_15798_b200 import binding as mole
from paper_2503_15798_b200 import inputs

DEV = "cuda"
FORMATS = {"bf16": mole.LUT_PLAIN, "f32": mole.LUT_PLAIN, "nf4": mole.LUT_NF4, "nf3": mole.LUT_NF3}
TABLE_BYTES = 40e9          # resident tables of a case
HOST_TABLE_BYTES = 1.7e9    # pinned tables of an offload case
OFFLOAD_CONTEXT_TOKENS = 256  # an offload context is made once, for the largest batch a program serves
EPS = 1e-6


def listed():
    s160, s410, s1b, tiny = (inputs.SHAPES[k] for k in ("160m", "410m", "1b", "tiny"))

    def case(name, kind, sh, M, **more):
        return dict({"name": name, "kind": kind, "V": sh.V, "d": sh.d, "N": sh.N, "M": M, "table": sh.dtype}, **more)

    return [
        # the tiny fp32 model the tests build from its FFNs: two small layers, all call overhead
        case("tiny-f32-step-64", "step", tiny, 64, L=tiny.L, mode="auto", norm=False),
        # one token of one layer: the shortest call of an interactive decode; ids as torch makes them (int64)
        case("160m-layer-1", "layer", s160, 1, norm=False, residual=False, ids64=True),
        # prefill of 8 prompts of 2048 tokens through one layer
        case("410m-layer-prefill-16384", "layer", s410, 16384, norm=False, residual=False, ids64=False),
        # a ragged prefill chunk through the widest layer, in the decoder-layer form: the router reads the normalised
        # state, the residual already holds the shared expert's output
        case("1b-layer-prefill-2999-norm", "layer", s1b, 2999, norm=True, residual=True, ids64=True),
        # the benchmark's decode step: one launch per layer, each feeding the next
        case("160m-step-256-chained", "step", s160, 256, L=s160.L, mode="chained", norm=False),
        # a decode step the way the library likes to run it, with a normalised router in every layer
        case("410m-step-64-norm", "step", s410, 64, L=s410.L, mode="auto", norm=True),
        # a small interactive batch of the widest model (a third of its vocabulary)
        dict(case("1b-step-16", "step", s1b, 16, L=s1b.L, mode="auto", norm=False), V=16384),
        # the same decode over tables quantised to a quarter
        dict(case("160m-step-64-nf4", "step", s160, 64, L=s160.L, mode="auto", norm=False), table="nf4", block=768),
        # activations in, activations out, through pinned host memory; the caller waits for every step
        case("160m-host-256", "host", s160, 256, L=s160.L),
        # tables off the GPU: a small decode batch over 24 layers (part of the vocabulary)
        dict(case("410m-offload-8", "offload", s410, 8, L=s410.L, hot=0), V=2048),
        # once per model: the tables from the experts, and their quantised form
        dict(case("160m-build", "build", s160, 0, D=4 * s160.d, norm=False)),
        dict(case("160m-quantize-nf3", "quantize", s160, 0), table="nf3", block=128),
    ]


# ---- drawn cases ----------------------------------------------------------------------------------------------------

def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))))


def _shape(rng, quant):
    """(N, d, V): half the time one of the repository's shapes, otherwise a width and expert count around them; a
    quantised layer takes widths in multiples of 128, and so do the many-expert ones (their rows are cut into pieces)."""
    if rng.random() < 0.5:
        sh = inputs.SHAPES[rng.choice(("160m", "410m", "1b"))]
        return sh.N, sh.d, sh.V
    N = rng.choice((4, 8, 16, 32) if quant else (4, 8, 12, 16, 24, 32, 64))
    unit = 128 if quant or N > 16 else rng.choice((8, 64, 128))
    d = max(unit, _log_int(rng, 128, 1024 if N > 32 else 2048) // unit * unit)
    return N, d, rng.choice((8192, 32000, 50304))


def _block(rng, d, fmt):
    if fmt == "nf4":  # the paper quantises whole rows of 768
        return 1024 if d % 1024 == 0 else d
    return 128


def draw(rng):
    kind = rng.choice(("layer", "layer", "step", "step", "host", "offload", "build", "quantize"))
    table = rng.choice(("bf16", "bf16", "bf16", "nf4", "nf3", "f32"))
    if kind in ("host", "build") or (kind == "offload" and table == "f32"):
        table = "bf16"
    if kind == "quantize":
        table = rng.choice(("nf4", "nf3"))
    quant = table in ("nf4", "nf3")
    N, d, V = _shape(rng, quant)
    if table == "f32":  # the small fp32 models
        N, d, V = rng.choice((4, 8, 16)), 4 * _log_int(rng, 16, 256), rng.choice((512, 4096, 32000))
    c = {"kind": kind, "V": V, "d": d, "N": N, "M": 0, "table": table}
    if quant:
        c["block"] = _block(rng, d, table)
    row = _row_bytes(c)
    if kind == "layer":
        c.update(M=_log_int(rng, 1, 16384), norm=rng.random() < 0.4, residual=rng.random() < 0.4, ids64=rng.random() < 0.5)
        if row * c["M"] > 16384 * 32768:  # no more work than the largest prefill listed
            c["M"] = 16384 * 32768 // row
    elif kind in ("step", "host"):
        c.update(M=_log_int(rng, 1, 1024), L=rng.randint(2, 24))
        if kind == "step":
            c.update(mode=rng.choice(("auto", "chained")), norm=rng.random() < 0.4)
        c["V"] = max(512, min(V, int(TABLE_BYTES / (row * c["L"]))))
    elif kind == "offload":
        c.update(M=_log_int(rng, 1, 128), L=rng.randint(4, 24))
        c["V"] = max(128, min(2048, int(HOST_TABLE_BYTES / (row * c["L"]))))
        c["hot"] = rng.choice((0, 0, c["V"] // 8))
    elif kind == "build":
        D = 4 * d
        most = int(7.5e12 / (4 * N * d * D))  # no more work than the listed table
        c.update(V=_log_int(rng, 64, max(64, min(V, most))), D=D, norm=rng.random() < 0.5)
    else:
        c["V"] = _log_int(rng, 1000, max(1000, min(V, int(1.2e9 / (2 * N * d)))))
    return c


# ---- sizes ----------------------------------------------------------------------------------------------------------

def _elem(c):
    return 4 if c["table"] == "f32" else 2


def _row_bytes(c):
    """bytes gathered per token and layer"""
    if c["table"] in ("nf4", "nf3"):
        return mole.quant_record_bytes(c["N"], c["d"], FORMATS[c["table"]], c["block"])
    return c["N"] * c["d"] * _elem(c)


def _distinct(c):
    """expected number of distinct ids among M Zipf(1.1) draws"""
    p = inputs.zipf_probs(c["V"])
    return float(-np.expm1(c["M"] * np.log1p(-p)).sum())


def work(case):
    c = case
    N, d, M, e = c["N"], c["d"], c["M"], _elem(c)
    if c["kind"] == "build":
        weights = 2 * N * c["D"] * d * 2
        return {"bytes": c["V"] * d * 2 + weights + c["V"] * N * d * 2, "flops": 4.0 * c["V"] * N * d * c["D"]}
    if c["kind"] == "quantize":
        return {"bytes": c["V"] * (N * d * 2 + _row_bytes(c)), "flops": 0}
    L = c.get("L", 1)
    ids = M * (8 if c.get("ids64") else 4)
    layer = _distinct(c) * _row_bytes(c) + d * N * e + (d * e if c.get("norm") else 0)
    act = M * d * e * (3 if c.get("residual") else 2)
    return {"bytes": L * layer + act + ids, "flops": 4.0 * L * M * N * d}


def tolerance(case):
    if case["kind"] == "quantize":
        return "exact"
    if case["table"] == "f32":
        return {"rel": 1e-5}
    # outputs are rounded to bf16 once per layer; another order of the fp32 sums moves a rounding now and then
    return {"rel": 5e-3, "max": 3e-2}


# ---- one case -------------------------------------------------------------------------------------------------------

def _normal(gen, shape, std, dtype):
    t = torch.empty(shape, dtype=dtype, device=DEV)
    return t.normal_(0.0, std, generator=gen)


def _tables(gen, c, L):
    """the tables of L layers: a bf16 / fp32 tensor [L][V][N][d], or the records of a quantised table"""
    V, N, d = c["V"], c["N"], c["d"]
    dtype = torch.float32 if c["table"] == "f32" else torch.bfloat16
    if c["table"] in ("bf16", "f32"):
        return _normal(gen, (L, V, N, d), 0.05, dtype)
    fmt, block = FORMATS[c["table"]], c["block"]
    packed = torch.zeros((L, V, _row_bytes(c)), dtype=torch.uint8, device=DEV)
    plain = torch.empty((V, N, d), dtype=dtype, device=DEV)
    for l in range(L):
        plain.normal_(0.0, 0.05, generator=gen)
        mole.QuantTable.quantize(plain, fmt, block, out=packed[l])
    return mole.QuantTable(packed, N, d, fmt, block)


def prepare(case, seed):
    c = case
    V, N, d, M, L = c["V"], c["N"], c["d"], c["M"], c.get("L", 1)
    dtype = torch.float32 if c["table"] == "f32" else torch.bfloat16
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    s = {"case": c}
    if c["kind"] == "build":
        s["x"] = _normal(gen, (V, d), 1.0, dtype)
        s["w1"] = _normal(gen, (N, c["D"], d), 1.0 / math.sqrt(d), dtype)
        s["w2"] = _normal(gen, (N, d, c["D"]), 1.0 / math.sqrt(c["D"]), dtype)
        s["norm"] = 1.0 + _normal(gen, (d,), 0.1, dtype) if c["norm"] else None
        s["out"] = torch.empty((V, N, d), dtype=dtype, device=DEV)
        return s
    if c["kind"] == "quantize":
        s["lut"] = _normal(gen, (V, N, d), 0.05, dtype)
        s["out"] = torch.zeros((V, _row_bytes(c)), dtype=torch.uint8, device=DEV)
        return s

    ids = torch.from_numpy(inputs.zipf_ids(M, V, seed=seed))
    ids = ids.to(torch.int64) if c.get("ids64") else ids
    hidden = _normal(gen, (M, d), 1.0, dtype)
    s["wr"] = _normal(gen, (L, d, N), 0.02, dtype)
    s["norm"] = 1.0 + _normal(gen, (L, d), 0.1, dtype) if c.get("norm") else None
    s["out"] = torch.empty_like(hidden)
    if c["kind"] == "layer":
        t = _tables(gen, c, 1)
        s["lut"] = t.layer(0) if isinstance(t, mole.QuantTable) else t[0]
        s["hidden"], s["ids"] = hidden, ids.to(DEV)
        s["residual"] = _normal(gen, (M, d), 1.0, dtype) if c["residual"] else None
        s["wr"], s["norm"] = s["wr"][0], s["norm"][0] if c["norm"] else None
    elif c["kind"] == "step":
        s["luts"] = _tables(gen, c, L)
        s["hidden"], s["ids"], s["tmp"] = hidden, ids.to(DEV), torch.empty_like(hidden)
        s["mode"] = {"auto": mole.STEP_AUTO, "chained": mole.STEP_CHAINED}[c["mode"]]
    elif c["kind"] == "host":
        s["luts"] = _tables(gen, c, L)
        s["hidden_host"], s["ids_host"] = hidden.cpu().pin_memory(), ids.pin_memory()
        s["out_host"] = torch.empty_like(s["hidden_host"], device="cpu", pin_memory=True)
        s["dev"] = [torch.empty_like(hidden), torch.empty(M, dtype=torch.int32, device=DEV), torch.empty_like(hidden),
                    torch.empty_like(hidden)]
    else:
        t = _tables(gen, c, L)
        t = t.packed if isinstance(t, mole.QuantTable) else t
        s["luts_host"] = torch.empty(t.shape, dtype=t.dtype, pin_memory=True)
        s["luts_host"].copy_(t)
        s["ctx"] = mole.OffloadContext(OFFLOAD_CONTEXT_TOKENS, N, d, V, lut_format=FORMATS[c["table"]], lut_block=c.get("block", 0))
        if c["hot"]:
            s["ctx"].set_hot_rows(inputs.zipf_hot_ids(V, c["hot"]), s["luts_host"])
        s["side"] = torch.cuda.Stream()
        s["hidden"], s["ids"], s["tmp"] = hidden, ids.to(DEV), torch.empty_like(hidden)
    return s


def run(state):
    s, c = state, state["case"]
    kind = c["kind"]
    if kind == "layer":
        return mole.layer_forward(s["hidden"], s["ids"], s["lut"], s["wr"], s["out"], residual=s["residual"], norm_weight=s["norm"],
                                  norm_eps=EPS)
    if kind == "step":
        return mole.decode_step_args(s["hidden"], s["ids"], s["luts"], s["wr"], s["out"], s["tmp"], mode=s["mode"],
                                     norm_weights=s["norm"], norm_eps=EPS)
    if kind == "host":
        out = mole.decode_step_host(s["hidden_host"], s["ids_host"], s["out_host"], *s["dev"], s["luts"], s["wr"])
        torch.cuda.current_stream().synchronize()  # the caller's next token depends on it
        return out
    if kind == "offload":
        return s["ctx"].decode_step(s["hidden"], s["ids"], s["luts_host"], s["wr"], s["out"], s["tmp"], side_stream=s["side"])
    if kind == "build":
        return mole.build_lut(s["x"], s["w1"], s["w2"], norm_weight=s["norm"], norm_eps=EPS, out=s["out"])
    return mole.QuantTable.quantize(s["lut"], FORMATS[c["table"]], c["block"], out=s["out"]).packed
