"""Decoder layouts against the oracle's containers (needs a GB300).

The decoder keeps a chunk's coded payloads in shared memory, whole or slice by
slice of its sub-streams, or reads them through per-thread rings (U8, large
chunks, few long sub-streams); any chunk may be ragged and any item a part of
the sub-streams.  Every byte must come back (lossless, ZipNN Sec. 2.3) whatever
the sizes, lanes and launch shape."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import oracle as O
from paper_2411_05239_gb300 import workloads as W
from paper_2411_05239_gb300 import zipnn as Z

pytestmark = pytest.mark.gpu


def u8(t: torch.Tensor) -> np.ndarray:
    return t.contiguous().view(-1).view(torch.uint8).cpu().numpy()


def quantised(n: int, seed: int) -> torch.Tensor:
    return W.gaussian(n, 20.0, seed, torch.float32).round().clamp(-127, 127).to(torch.int8)


def long_codes(n: int, seed: int) -> torch.Tensor:
    """Bytes with P(k) ~ 2^-k: 12-bit codes beside one-bit ones."""
    g = np.random.default_rng(seed)
    return torch.from_numpy((g.geometric(0.5, size=n) - 1).clip(0, 39).astype(np.uint8))


MAKE = {"bf16": lambda n, s: W.gaussian(n, 0.02, s),
        "fp16": lambda n, s: W.gaussian(n, 0.02, s, torch.float16),
        "clean_fp16": W.clean_fp16_from_bf16,        # two coded groups: slices
        "fp32": lambda n, s: W.gaussian(n, 0.05, s, torch.float32),
        "u8": quantised, "long_u8": long_codes}       # rings


def round_trip(x: torch.Tensor, chunk: int, lanes: int = 0, parts=(0, 1, 8)) -> None:
    dt = Z.dtype_code(x, None)
    c = Z.compress(x.cuda(), chunk_bytes=chunk, lanes=lanes)
    assert c.to_bytes() == O.compress(u8(x), dt, chunk, lanes or Z.default_lanes(dt, chunk))
    out = torch.empty_like(x, device="cuda")
    for p in parts:
        out.zero_()
        Z.batch_decompress([c], [out], tune=Z.tuning(parts=p))
        Z.sync_status()
        assert np.array_equal(u8(out), u8(x)), p
    out.zero_()
    Z.decompress(c, out)
    Z.sync_status()
    assert np.array_equal(u8(out), u8(x))


@pytest.mark.parametrize("kind", list(MAKE))
@pytest.mark.parametrize("tail", [1, 7, 8, 9, 8 * 511 + 3, 8 * 512, 8 * 512 + 1, 8 * 1025])
def test_ragged_chunks(kind, tail):
    """One whole 256 KiB chunk and a ragged one, around whole vectors and whole
    rounds of the sub-streams."""
    es = {"fp32": 4, "u8": 1, "long_u8": 1}.get(kind, 2)
    round_trip(MAKE[kind](262144 // es + tail, 200 + tail), 262144)


@pytest.mark.parametrize("kind", list(MAKE))
@pytest.mark.parametrize("chunk,lanes", [(65536, 0), (1 << 20, 0), (1 << 20, 96), (262144, 1),
                                         (262144, 300), (4096, 256)])
def test_chunk_sizes_and_lanes(kind, chunk, lanes):
    es = {"fp32": 4, "u8": 1, "long_u8": 1}.get(kind, 2)
    round_trip(MAKE[kind](2 * chunk // es + 1003, 300), chunk, lanes, parts=(0, 4))


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("n", [131072 * 2 + 5, 24579, 131072 * 400 + 17])
def test_deltas(dtype, n):
    nxt, base = W.delta_pair(n, seed=310, device="cuda")
    nxt, base = nxt.to(dtype), base.to(dtype)
    c = Z.delta(nxt, base)
    out = torch.empty_like(nxt)
    for tune in (None, Z.tuning(parts=4), Z.tuning(threads=128)):
        out.zero_()
        Z.batch_decompress([c], [out], bases=[base], tune=tune)
        Z.sync_status()
        assert torch.equal(out.view(torch.uint8), nxt.view(torch.uint8))


def test_batch_of_every_family_and_empty_tensors():
    """A batch takes one launch per dtype family; empty tensors and tensors of
    one family between those of others keep their places."""
    xs = [W.gaussian(70_001, 0.02, 320), quantised(300_007, 321), W.gaussian(0, 0.02, 322),
          W.gaussian(40_003, 0.05, 323, torch.float32), W.gaussian(150_000, 0.02, 324, torch.float16),
          quantised(0, 325), long_codes(262_144, 326), W.gaussian(131_072, 0.02, 327)]
    cs = [Z.compress(x.cuda(), chunk_bytes=65536) for x in xs]
    outs = [torch.zeros_like(x, device="cuda") for x in xs]
    Z.batch_decompress(cs, outs)
    Z.sync_status()
    for x, o in zip(xs, outs):
        assert np.array_equal(u8(o), u8(x))
    for o in outs:
        o.zero_()
    p = Z.plan_decompress(cs, outs)
    for _ in range(2):
        p.launch()
    Z.sync_status()
    p.close()
    for x, o in zip(xs, outs):
        assert np.array_equal(u8(o), u8(x))
