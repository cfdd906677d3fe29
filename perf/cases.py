"""Performance cases of the framework: the calls a user's program makes, over the sizes it makes them at.

Kinds of case (key "kind"):
  call      one mat-vec (lw.matvec), 1 to 16 activation columns
  step      every mat-vec of a decode step as one chain (lw.matvec_sequence, lw.matvec_sequence_batch for several
            columns, the _host form where the step's input and logits live in host memory)
  attn      decode attention of one token over a block-quantised KV cache (lw.attn_decode)
  dequant   blocks to fp32 on the device (lw.dequant)
  quantize  fp32 to blocks on the host (lw.quantize)

Weights are blocks that the framework's own quantiser makes from N(0, std^2) values (for the K-quants 1 % of them ten
times larger, as in trained weights): a pool of 2^20 weights is quantised per format and width, and matrices are
drawn from the pool's blocks on the GPU.  The standard deviation is 1 / sqrt(cols), so that a chain of mat-vecs keeps
the size of its activations.
"""
import math

import numpy as np
import torch

from paper_2605_20706_b200 import lw

KQUANTS = ("q4_K", "q6_K", "q5_K", "q2_K")
POOL_WEIGHTS = 1 << 20

# hidden, kv width, ffn, vocabulary, layers of the two decode steps that the benchmark replays
STEP_1B = {"hidden": 2048, "kv": 512, "ffn": 8192, "vocab": 128256, "layers": 16}
STEP_8B = {"hidden": 4096, "kv": 1024, "ffn": 14336, "vocab": 128256, "layers": 32}


def listed():
    return [
        # the smallest call: one projection of a small model; launch latency and host time
        {"name": "call_q8_0_2048", "kind": "call", "fmt": "q8_0", "rows": 2048, "cols": 2048, "batch": 1, "overlap": 0},
        # an output head in the format that mixed quantisations give it, width no multiple of 2048
        {"name": "call_q6_K_head", "kind": "call", "fmt": "q6_K", "rows": 32000, "cols": 3072, "batch": 1, "overlap": 0},
        # sizes that fit no tile: an odd number of rows, a width of whole 32-weight blocks only
        {"name": "call_q4_0_ragged", "kind": "call", "fmt": "q4_0", "rows": 11007, "cols": 2848, "batch": 1, "overlap": 0},
        # a few sequences decoded together, one call per matrix: the gate projection of the 8B step
        {"name": "call_q5_1_batch5", "kind": "call", "fmt": "q5_1", "rows": 14336, "cols": 4096, "batch": 5, "overlap": 0},
        # decode steps of one sequence as one chain: a small model in 4 bits, the same in f16 with the step's input
        # and logits in host memory, the benchmark's default workload
        dict(STEP_1B, name="step_1b_q4_0", kind="step", fmt="q4_0", batch=1, host=False, overlap=0),
        dict(STEP_1B, name="step_1b_f16_host", kind="step", fmt="f16", batch=1, host=True, overlap=0),
        dict(STEP_8B, name="step_8b_q4_K", kind="step", fmt="q4_K", batch=1, host=False, overlap=0),
        # eight sequences decoded together; the weights are parameters, so copies of them may start early
        dict(STEP_8B, name="step_8b_q4_K_batch8", kind="step", fmt="q4_K", batch=8, host=False, overlap=2),
        # attention of one token: a long conversation of the 8B shape, a short odd one of the 1B shape
        {"name": "attn_8b_q8_0_32k", "kind": "attn", "fmt": "q8_0", "heads": 32, "kv_heads": 8, "dim": 128, "pos": 32768, "overlap": 0},
        {"name": "attn_1b_f16_1021", "kind": "attn", "fmt": "f16", "heads": 32, "kv_heads": 8, "dim": 64, "pos": 1021, "overlap": 0},
        # decode and encode: a model's weights to fp32 on the device, one matrix to blocks on the host
        {"name": "dequant_q4_K", "kind": "dequant", "fmt": "q4_K", "n": 1 << 28, "overlap": 0},
        {"name": "quantize_q4_K", "kind": "quantize", "fmt": "q4_K", "n": 1024 * 4096, "overlap": 0},
    ]


def _log(rng, lo, hi, quantum=1):
    """A multiple of `quantum` between lo and hi, spread evenly over the logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / quantum)) * quantum))


def draw(rng):
    kind = rng.choice(["call"] * 8 + ["step"] * 6 + ["attn"] * 4 + ["dequant", "quantize"])
    fmt = rng.choice(["q4_K", "q4_K", "q4_0", "q4_0", "q8_0", "q8_0", "f16", "q6_K", "q5_K", "q2_K", "q4_1", "q5_0", "q5_1"])
    if kind == "call":
        # one width in three is a whole number of blocks and no more; one matrix in three has any number of rows
        quantum = 256 if fmt in KQUANTS or rng.random() < 0.67 else 32
        rows = _log(rng, 512, 131072, 1 if rng.random() < 0.33 else 128)
        return {"kind": kind, "fmt": fmt, "rows": rows, "cols": _log(rng, 1024, 14336, quantum),
                "batch": rng.choice([1, 1, 1, 1, 2, 3, 4, 6, 8, 13, 16]), "overlap": 0}
    if kind == "step":
        hidden = _log(rng, 1024, 4096, 256)
        c = {"hidden": hidden, "kv": max(256, hidden // rng.choice([2, 4, 4, 8]) // 64 * 64),
             "ffn": _log(rng, 2 * hidden, 4 * hidden, 256), "vocab": _log(rng, 8192, 131072, 8), "layers": _log(rng, 4, 32)}
        batch = rng.choice([1, 1, 1, 2, 4, 5, 8, 16])
        c.update(kind=kind, fmt=fmt, batch=batch, host=rng.random() < 0.25, overlap=2 if batch > 1 else 0)
        most = work(next(k for k in listed() if k["name"] == "step_8b_q4_K_batch8"))
        while c["layers"] > 1 and (work(c)["bytes"] > most["bytes"] or work(c)["flops"] > most["flops"]):
            c["layers"] -= 1
        return c
    if kind == "attn":
        kv = rng.choice([2, 4, 8, 8, 8])
        return {"kind": kind, "fmt": rng.choice(["f16", "q8_0", "q4_0"]), "heads": kv * rng.choice([1, 3, 4, 4, 4, 8]), "kv_heads": kv,
                "dim": rng.choice([64, 64, 128, 128, 256]), "pos": _log(rng, 100, 131072), "overlap": 0}
    if kind == "dequant":
        return {"kind": kind, "fmt": fmt, "n": _log(rng, 1 << 20, 1 << 28, 256), "overlap": 0}
    return {"kind": kind, "fmt": fmt, "n": _log(rng, 1 << 18, 1 << 22, 256), "overlap": 0}


def _matrices(c):
    """(rows, cols, input, starts a phase) of every mat-vec of a step; input is the index of the matrix whose
    result it reads, -1 for the step's input.  o reads q's result and down reads gate's: the operations between
    them (attention, activation function) are other kernels' work and keep the width."""
    out, last = [], -1
    for _ in range(c["layers"]):
        j = len(out)
        out += [(c["hidden"], c["hidden"], last, True), (c["kv"], c["hidden"], last, False), (c["kv"], c["hidden"], last, False),
                (c["hidden"], c["hidden"], j, True),
                (c["ffn"], c["hidden"], j + 3, True), (c["ffn"], c["hidden"], j + 3, False),
                (c["hidden"], c["ffn"], j + 4, True)]
        last = j + 6
    out.append((c["vocab"], c["hidden"], last, True))
    return out


def work(case):
    c, kind = case, case["kind"]
    fmt = lw.FORMATS[c["fmt"]]
    if kind in ("call", "step"):
        mats = [(c["rows"], c["cols"])] if kind == "call" else [(r, k) for r, k, _, _ in _matrices(c)]
        weights = sum(r * k for r, k in mats)
        b = sum(r * lw.row_bytes(fmt, k) + 4 * c["batch"] * (r + k) for r, k in mats)
        return {"bytes": b, "flops": 2 * weights * c["batch"]}
    if kind == "attn":
        width = c["kv_heads"] * c["dim"]
        b = 2 * c["pos"] * lw.row_bytes(fmt, width) + 8 * c["heads"] * c["dim"]
        return {"bytes": b, "flops": 4 * c["heads"] * c["dim"] * c["pos"]}
    return {"bytes": 4 * c["n"] + lw.row_bytes(fmt, c["n"]), "flops": 2 * c["n"]}


def tolerance(case):
    c, kind = case, case["kind"]
    if kind in ("dequant", "quantize"):
        return "exact"                      # every product is exact, every rounding is prescribed
    if kind == "attn":
        return {"rel": 2e-5, "max": 8e-4}   # fp32 sums over the positions, most of them cancelling
    # fp32 sums, and from two columns on activations of 16 significant bits (2^-16 each, errors of either sign).  The
    # mat-vecs of a chain add their errors up: 225 of them with activations of 16 bits differ by 2e-4 between two runs
    # that only add in another order
    one = 1e-5 if c["batch"] == 1 else 2e-5
    return {"rel": one} if kind == "call" else {"rel": 2e-5 if c["batch"] == 1 else 3e-4}


def _pool(name, std, seed):
    """2^20 quantised weights as (blocks, bytes per block / 2) int16 on the GPU; f16 counts runs of 32 as blocks."""
    fmt = lw.FORMATS[name]
    gen = np.random.default_rng(seed)
    w = gen.standard_normal(POOL_WEIGHTS, dtype=np.float32)
    if name in KQUANTS:
        w[gen.integers(0, POOL_WEIGHTS, POOL_WEIGHTS // 100)] *= np.float32(10.0)
        std /= math.sqrt(1.99)
    blocks = lw.quantize(fmt, w * np.float32(std))
    return torch.from_numpy(blocks.view(np.int16).reshape(-1, _block(fmt)[1] // 2)).cuda()


def _block(fmt):
    """Weights and bytes of the pool's blocks."""
    return (lw.block_elems(fmt), lw.block_bytes(fmt)) if fmt != lw.F16 else (32, 64)


def _from_pool(pool, out, blocks, gen):
    """Fills `out` (int16) with blocks drawn from the pool, a part at a time."""
    out = out.view(blocks, pool.shape[1])
    for at in range(0, blocks, 1 << 23):
        n = min(1 << 23, blocks - at)
        idx = torch.randint(0, pool.shape[0], (n,), device="cuda", generator=gen)
        torch.index_select(pool, 0, idx, out=out[at:at + n])


def prepare(case, seed):
    c, kind = case, case["kind"]
    fmt = lw.FORMATS[c["fmt"]]
    be, bb = _block(fmt)
    s = {"kind": kind, "fmt": fmt, "case": c}
    if kind == "quantize":
        gen = np.random.default_rng(seed)
        s["src"] = gen.standard_normal(c["n"], dtype=np.float32) * np.float32(0.02)
        s["src"][gen.integers(0, c["n"], c["n"] // 100)] *= np.float32(10.0)
        s["dst"] = np.zeros(lw.row_bytes(fmt, c["n"]), dtype=np.uint8)
        return s
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    lw.set_overlap(c["overlap"])
    if kind == "dequant":
        s["W"] = torch.empty(c["n"] // be * bb // 2, dtype=torch.int16, device="cuda")
        _from_pool(_pool(c["fmt"], 0.02, seed), s["W"], c["n"] // be, gen)
        s["out"] = torch.zeros(c["n"], device="cuda")
        return s
    if kind == "attn":
        width = c["kv_heads"] * c["dim"]
        pool = _pool(c["fmt"], 1.0, seed)
        for key in ("K", "V"):
            s[key] = torch.empty(c["pos"] * lw.row_bytes(fmt, width) // 2, dtype=torch.int16, device="cuda")
            _from_pool(pool, s[key], c["pos"] * width // be, gen)
        s["q"] = torch.randn(c["heads"] * c["dim"], device="cuda", generator=gen)
        s["out"] = torch.zeros_like(s["q"])
        s["ws"] = torch.empty(lw.attn_workspace_bytes(c["heads"], c["kv_heads"], c["dim"], c["pos"]), dtype=torch.uint8, device="cuda")
        s["scale"] = 1.0 / math.sqrt(c["dim"])
        return s
    mats = [(c["rows"], c["cols"], -1, True)] if kind == "call" else _matrices(c)
    batch = c["batch"]
    pools = {}
    for k in sorted({k for _, k, _, _ in mats}):
        pools[k] = _pool(c["fmt"], 1.0 / math.sqrt(k), seed + k)
    s["W"] = []
    for r, k, _, _ in mats:
        w = torch.empty(r * lw.row_bytes(fmt, k) // 2, dtype=torch.int16, device="cuda")
        _from_pool(pools[k], w, r * k // be, gen)
        s["W"].append(w)
    s["X"] = torch.randn(batch * mats[0][1], device="cuda", generator=gen)
    # results one behind the other, each on a 16-byte boundary
    starts, size = [], 0
    for r, _, _, _ in mats:
        starts.append(size)
        size += (batch * r + 3) // 4 * 4
    s["Y"] = torch.zeros(size, device="cuda")
    if kind == "call":
        return s
    Y = [s["Y"][at:at + batch * m[0]] for at, m in zip(starts, mats)]
    s["items"] = lw.seq_items([(w, r, k, s["X"] if src < 0 else Y[src], y, lw.SEQ_DEPENDENT if first else 0)
                               for w, (r, k, src, first), y in zip(s["W"], mats, Y)])
    s["logits"] = Y[-1]
    s["ws"] = torch.zeros(lw.matvec_sequence_workspace_bytes(), dtype=torch.uint8, device="cuda")
    if c["host"]:
        s["X_host"] = s["X"].cpu().pin_memory()
        s["logits_host"] = torch.zeros(Y[-1].numel(), pin_memory=True)
    return s


def run(s):
    c, fmt = s["case"], s["fmt"]
    if s["kind"] == "call":
        lw.matvec(fmt, s["W"][0], c["rows"], c["cols"], s["X"], s["Y"], c["batch"])
        return s["Y"]
    if s["kind"] == "step":
        host = c["host"] and (s["X_host"], s["X"], 4 * s["X"].numel(), s["logits"], s["logits_host"], 4 * s["logits"].numel())
        if c["batch"] == 1:
            if not host:
                lw.matvec_sequence(fmt, s["items"], s["ws"])
                return s["Y"]
            lw.matvec_sequence_host(fmt, s["items"], *host, s["ws"])
        else:
            if not host:
                lw.matvec_sequence_batch(fmt, s["items"], c["batch"])
                return s["Y"]
            lw.matvec_sequence_batch_host(fmt, s["items"], c["batch"], *host)
        return [s["logits_host"], s["Y"]]
    if s["kind"] == "attn":
        lw.attn_decode(fmt, s["K"], s["V"], s["q"], s["out"], c["heads"], c["kv_heads"], c["dim"], c["pos"], s["scale"], s["ws"])
        return s["out"]
    if s["kind"] == "dequant":
        lw.dequant(fmt, s["W"], c["n"], s["out"])
        return s["out"]
    lw.quantize(fmt, s["src"], s["dst"])
    return s["dst"]
