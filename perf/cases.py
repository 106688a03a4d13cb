"""Performance cases of the codec: calls that a user's program makes through
the package's public entry points, each as a dict of plain values.

A case names a direction (``op``), how the call is made (``form``), the values
that the tensors hold (``kind``) and the sizes:

form  "one"    one tensor through ``compress_into`` / ``decompress`` into
               buffers that the caller keeps (a serving or checkpointing loop)
      "call"   the one-line call ``compress(x)``, which allocates the container
               and reads its size back (scripts, converters)
      "plan"   all tensors of a model through a captured plan, launched once
               per pass (a trainer that compresses every checkpoint, a loader)
      "batch"  the same without a plan: ``BatchCompressor`` / ``batch_decompress``
kind  "bf16", "fp16", "fp32", "u8"   weights in that type: N(0, 0.02); FP32
               with per-row scales and 2% zeros; U8 as int8 quantised weights
      "clean_fp32", "clean_fp16"     BF16 values held in a wider type
      "delta_bf16", "delta_fp32"     a checkpoint against the one before it
      "model"  a decoder-only model in BF16 (``workloads.llama8b_specs``)
      "mixed"  a model of BF16, int8, FP16 and FP32 tensors in one batch

Outputs are bytes: containers, and decoded tensors viewed as integers (the
codec is lossless, so they have one right value).
"""
from __future__ import annotations

import math

import torch

from paper_2411_05239_gb300 import workloads as W
from paper_2411_05239_gb300 import zipnn as Z

CHUNK = Z.DEFAULT_CHUNK

# Container bytes per original byte, for `work` (measured; the container is an
# output whose size depends on the values, here only on their distribution).
RATIO = {"bf16": 0.670, "fp16": 0.858, "fp32": 0.859, "u8": 0.803, "clean_fp32": 0.338,
         "clean_fp16": 0.69, "delta_bf16": 0.138, "delta_fp32": 0.10, "model": 0.670,
         "mixed": 0.71}
ELEM = {"bf16": 2, "fp16": 2, "fp32": 4, "u8": 1, "clean_fp32": 4, "clean_fp16": 2,
        "delta_bf16": 2, "delta_fp32": 4}
INT = {1: torch.uint8, 2: torch.int16, 4: torch.int32}


def _delta_numel() -> int:
    return sum(s.numel for s in W.delta_specs())


def listed() -> list[dict]:
    one = dict(form="one", chunk=CHUNK)
    return [
        # the smallest tensors of a model, one at a time: a norm vector, a
        # bias, a low-rank adapter (48 KiB and a ragged tail)
        dict(one, name="small_bf16_compress", op="compress", kind="bf16", numel=24_579),
        dict(one, name="small_bf16_decompress", op="decompress", kind="bf16", numel=24_579),
        # an ordinary tensor, 8 MiB: the one-line compression, and decoding
        # into a buffer that the program keeps
        dict(one, name="tensor_bf16_compress_call", op="compress", form="call", kind="bf16",
             numel=4_194_304),
        dict(one, name="tensor_bf16_decompress", op="decompress", kind="bf16", numel=4_194_304),
        # one large FP32 matrix, 256 MiB (a master weight)
        dict(one, name="matrix_fp32_compress", op="compress", kind="fp32", numel=8192 * 8192),
        dict(one, name="matrix_fp32_decompress", op="decompress", kind="fp32", numel=8192 * 8192),
        # FP16 weights of an odd size: the last chunk is ragged
        dict(one, name="odd_fp16_decompress", op="decompress", kind="fp16", numel=40_000_003),
        # a BF16 model as a whole (six layers, embedding and head of the 8B
        # shapes, 4.7 GB): saving and loading through plans
        dict(name="model_bf16_compress", op="compress", form="plan", kind="model", chunk=CHUNK,
             layers=6, hidden=4096, kv=1024, ffn=14336, vocab=128256),
        dict(name="model_bf16_decompress", op="decompress", form="plan", kind="model", chunk=CHUNK,
             layers=6, hidden=4096, kv=1024, ffn=14336, vocab=128256),
        # a training checkpoint against the one before it (3.43 GB)
        dict(one, name="delta_bf16_compress", op="compress", kind="delta_bf16",
             numel=_delta_numel()),
        dict(one, name="delta_bf16_decompress", op="decompress", kind="delta_bf16",
             numel=_delta_numel()),
        # a model whose tensors have several types, decoded in one call
        dict(name="mixed_model_decompress", op="decompress", form="batch", kind="mixed",
             chunk=CHUNK, layers=12, hidden=2048, kv=512, ffn=8192, vocab=50_000),
    ]


def draw(rng) -> dict:
    op = rng.choice(["compress", "decompress"])
    chunk = rng.choice([CHUNK, CHUNK, CHUNK, 64 << 10, 1 << 20])
    if rng.random() < 0.3:  # a whole model
        hidden = 16 * rng.randint(16, 256)
        kv = hidden // rng.choice([1, 2, 4, 8])
        return dict(op=op, form=rng.choice(["plan", "batch"]), kind=rng.choice(["model", "mixed"]),
                    chunk=chunk, layers=rng.randint(1, 6), hidden=hidden, kv=kv,
                    ffn=hidden * 7 // 2, vocab=rng.randint(1000, 128256))
    kind = rng.choice(list(ELEM))
    nbytes = math.exp(rng.uniform(math.log(32 << 10), math.log(1 << 30)))
    form = "call" if op == "compress" and rng.random() < 0.25 else "one"
    return dict(op=op, form=form, kind=kind, chunk=chunk, numel=int(nbytes) // ELEM[kind])


# ---------------------------------------------------------------------------
# inputs


def _tensor(kind: str, n: int, seed: int):
    """(tensor, delta base or None) of n elements on the GPU."""
    if kind.startswith("delta"):
        nxt, base = W.delta_pair(n, seed=seed, device="cuda")
        return (nxt, base) if kind == "delta_bf16" else (nxt.float(), base.float())
    if kind == "fp32":
        cols = min(n, 8192)
        return W.rowscaled_fp32(-(-n // cols), cols, seed=seed, device="cuda")[:n], None
    if kind == "clean_fp32":
        return W.clean_fp32_from_bf16(n, seed=seed, device="cuda"), None
    if kind == "clean_fp16":
        return W.clean_fp16_from_bf16(n, seed=seed, device="cuda"), None
    if kind == "u8":  # symmetric int8 quantisation of normal weights, three deviations at 60
        q = W.gaussian(n, 20.0, seed=seed, dtype=torch.float32, device="cuda")
        return q.round_().clamp_(-127, 127).to(torch.int8), None
    return W.gaussian(n, 0.02, seed=seed, dtype=W.TORCH_DTYPE[kind], device="cuda"), None


def _mixed_sizes(case: dict) -> list[tuple[str, int]]:
    h, kv, ffn = case["hidden"], case["kv"], case["ffn"]
    sizes = [("bf16", case["vocab"] * h)]
    for _ in range(case["layers"]):
        sizes += [("bf16", h * (h + 2 * kv)),  # fused attention projections
                  ("u8", h * ffn),             # quantised MLP weight
                  ("fp16", 64 * h),            # low-rank adapter
                  ("fp32", 2 * h + 1)]         # norms and a scale
    return sizes


def _model_specs(case: dict):
    return W.llama8b_specs(case["layers"], case["hidden"], case["kv"], case["ffn"], case["vocab"])


def _inputs(case: dict, seed: int):
    """(tensors, bases or None) of a case."""
    if case["kind"] == "model":
        return W.checkpoint_bf16(_model_specs(case), seed=seed, device="cuda"), None
    if case["kind"] == "mixed":
        return [_tensor(k, n, 1000 * seed + i)[0]
                for i, (k, n) in enumerate(_mixed_sizes(case))], None
    x, base = _tensor(case["kind"], case["numel"], seed)
    return [x], None if base is None else [base]


def _bits(t: torch.Tensor) -> torch.Tensor:
    return t.view(INT[t.element_size()])


def prepare(case: dict, seed: int) -> dict:
    chunk, form = case["chunk"], case["form"]
    xs, bases = _inputs(case, seed)
    base = bases[0] if bases else None
    s = {"op": case["op"], "form": form, "chunk": chunk, "base": base}
    if case["op"] == "compress":
        if form == "call":
            # the program appends the container to an archive buffer
            n, code = xs[0].numel() * xs[0].element_size(), Z.dtype_code(xs[0], None)
            s["x"] = xs[0]
            s["archive"] = torch.zeros(Z.compress_bound(n, code, chunk), dtype=torch.uint8,
                                       device="cuda")
        elif form == "one":
            n, code = xs[0].numel() * xs[0].element_size(), Z.dtype_code(xs[0], None)
            s["x"] = xs[0]
            # zeros: the bytes after the container are never written
            s["out"] = torch.zeros(Z.compress_bound(n, code, chunk), dtype=torch.uint8,
                                   device="cuda")
            s["ws"] = torch.empty(Z.workspace_size(n, code, chunk), dtype=torch.uint8,
                                  device="cuda")
            s["nbytes"] = torch.zeros(1, dtype=torch.int64, device="cuda")
        else:
            bc = Z.BatchCompressor(xs, chunk_bytes=chunk, bases=bases)
            for o in bc.outs:
                o.zero_()
            s["bc"] = bc
            if form == "plan":
                s["plan"] = Z.plan_compress(bc)
        return s
    # decompression: the program holds containers and the buffers to fill
    if form == "one":
        s["c"] = Z.compress(xs[0], chunk_bytes=chunk, base=base)
        s["y"] = torch.empty_like(xs[0])
        s["bits"] = _bits(s["y"])
    else:
        bc = Z.BatchCompressor(xs, chunk_bytes=chunk, bases=bases)
        bc()
        s["cs"] = bc.containers()
        s["ys"] = [torch.empty_like(x) for x in xs]
        s["bits"] = [_bits(y) for y in s["ys"]]
        if form == "plan":
            s["plan"] = Z.plan_decompress(s["cs"], s["ys"])
    return s


def run(s: dict):
    if s["form"] == "plan":
        s["plan"].launch()
        return s["bc"].outs + [s["bc"].out_nbytes] if s["op"] == "compress" else s["bits"]
    if s["op"] == "compress":
        if s["form"] == "call":
            c = Z.compress(s["x"], chunk_bytes=s["chunk"], base=s["base"])
            s["archive"][:c.nbytes] = c.device_tensor()
            return s["archive"], c.nbytes
        if s["form"] == "one":
            Z.compress_into(s["x"], s["out"], s["ws"], s["nbytes"], base=s["base"],
                            chunk_bytes=s["chunk"])
            return s["out"], s["nbytes"]
        s["bc"]()
        return s["bc"].outs + [s["bc"].out_nbytes]
    if s["form"] == "one":
        Z.decompress(s["c"], s["y"], base=s["base"])
    else:
        Z.batch_decompress(s["cs"], s["ys"])
    return s["bits"]


def work(case: dict) -> dict:
    if case["kind"] == "model":
        orig = 2 * sum(sp.numel for sp in _model_specs(case))
    elif case["kind"] == "mixed":
        orig = sum(ELEM[k] * n for k, n in _mixed_sizes(case))
    else:
        orig = ELEM[case["kind"]] * case["numel"]
    base = orig if case["kind"].startswith("delta") else 0
    return {"bytes": orig + base + RATIO[case["kind"]] * orig, "flops": 0}
