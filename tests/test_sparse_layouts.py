"""SPARSE groups beside raw and other coded ones, at every density of live
vectors (ZipNN Sec. 4.2 with this container's bitmap of live vectors): the
containers must equal the oracle's byte for byte, decode in the oracle, and
decode on the GPU to the input.

The CPU tests pin the oracle by the specification decoder and the GPU tests the
kernels by the oracle."""
from __future__ import annotations

import struct

import numpy as np
import pytest
import torch

import oracle as O
from tests import spec_decoder

SPARSE = 4
CODE = {"bf16": O.BF16, "fp16": O.FP16, "fp32": O.FP32, "u8": O.U8}


def pruned(kind: str, vectors: int, live: float, seed: int) -> np.ndarray:
    """The bytes of weights in which only a share `live` of the 16-byte vectors
    is not zero: N(0, 0.02) values, for "u8" uniform bytes."""
    g = np.random.default_rng(seed)
    keep = g.random(vectors) < live
    if kind == "u8":
        x = g.integers(0, 256, size=(vectors, 16), dtype=np.uint8)
    else:
        w = torch.from_numpy((g.standard_normal(vectors * (4 if kind == "fp32" else 8)) * 0.02)
                             .astype(np.float32))
        t = w.to({"bf16": torch.bfloat16, "fp16": torch.float16, "fp32": torch.float32}[kind])
        x = t.view(torch.uint8).numpy().reshape(vectors, 16)
    return np.where(keep[:, None], x, 0).astype(np.uint8).reshape(-1)


def modes(s: bytes) -> list[tuple[int, ...]]:
    G, nch = struct.unpack_from("<II", s, 24)
    m = [struct.unpack_from("<QIBB", s, 64 + 16 * i)[2] for i in range(nch * G)]
    return [tuple(m[c * G:c * G + G]) for c in range(nch)]


# -- one coded group, SPARSE, and the others raw: 2 to 4% zero vectors

BESIDE_RAW = [("bf16", 0.96), ("bf16", 0.97), ("bf16", 0.98), ("fp16", 0.97)]


@pytest.mark.gpu
@pytest.mark.parametrize("kind,live", BESIDE_RAW)
@pytest.mark.parametrize("lanes", [0, 256, 512, 1024])
def test_sparse_beside_raw(kind, live, lanes):
    from paper_2411_05239_gb300 import zipnn as Z
    dt = CODE[kind]
    x = pruned(kind, 4 * 16384 + 777, live, 600)
    want = O.compress(x, dt, 262144, lanes or Z.default_lanes(dt, 262144))
    assert modes(want)[0] == (SPARSE, 0)
    t = torch.from_numpy(x).cuda().view(Z.CODE_TO_TORCH[dt])
    assert Z.compress(t, lanes=lanes).to_bytes() == want
    for encoder in (0, 1):
        bc = Z.BatchCompressor([t], chunk_bytes=262144, lanes=lanes, encoder=encoder)
        bc()
        Z.sync_status()
        c = bc.containers()[0]
        assert c.to_bytes() == want, encoder
    out = torch.zeros_like(t)
    Z.decompress(c, out)
    Z.sync_status()
    assert torch.equal(out.view(torch.uint8), t.view(torch.uint8))


# -- FP32 with several SPARSE groups, whose bitmaps and tables leave little stage


def fp32_delta(vectors: int, live: float, seed: int) -> tuple[np.ndarray, np.ndarray]:
    """(next, base) bytes of FP32 weights of which a share of the 16-byte vectors
    changed, in every byte."""
    g = np.random.default_rng(seed)
    base = (g.standard_normal(vectors * 4) * 0.02).astype(np.float32).view(np.uint8)
    return base ^ pruned("fp32", vectors, live, seed + 1), base


def decode_every_way(c, want: torch.Tensor, base: torch.Tensor | None = None) -> None:
    from paper_2411_05239_gb300 import zipnn as Z
    out = torch.zeros_like(want)

    def check(what):
        Z.sync_status()
        assert torch.equal(out.view(torch.uint8), want.view(torch.uint8)), what
        out.zero_()

    Z.decompress(c, out, base=base)
    check("alone")
    bases = None if base is None else [base]
    for tune in (None, Z.tuning(threads=128), Z.tuning(threads=256), Z.tuning(parts=4)):
        Z.batch_decompress([c], [out], bases=bases, tune=tune)
        check("batch")
        p = Z.plan_decompress([c], [out], bases=bases, tune=tune)
        p.launch()
        check("plan")
        p.close()


@pytest.mark.gpu
@pytest.mark.parametrize("chunk", [65536, 131072, 262144, 524288])
@pytest.mark.parametrize("live", [0.02, 0.05])
@pytest.mark.parametrize("delta", [False, True])
def test_fp32_with_four_sparse_groups(chunk, live, delta):
    from paper_2411_05239_gb300 import zipnn as Z
    v = 5 * chunk // 16 + 333
    x, b = fp32_delta(v, live, 700) if delta else (pruned("fp32", v, live, 700), None)
    lanes = O.default_lanes(O.FP32, chunk, delta)
    want = O.delta(x, b, O.FP32, chunk, lanes) if delta else O.compress(x, O.FP32, chunk, lanes)
    assert modes(want)[0] == (SPARSE,) * 4
    t = torch.from_numpy(x).cuda().view(torch.float32)
    base = None if b is None else torch.from_numpy(b).cuda().view(torch.float32)
    c = Z.compress(t, chunk_bytes=chunk, base=base)
    assert c.to_bytes() == want
    decode_every_way(c, t, base)


@pytest.mark.gpu
def test_sparse_chunks_among_weights():
    """One tensor whose chunks are weights but for one in 200 (a plan then keeps the
    kernel and the stage for weights), and one with every mix of groups."""
    from paper_2411_05239_gb300 import zipnn as Z
    g = np.random.default_rng(701)
    n = 65536 // 4
    x = (g.standard_normal(200 * n) * 0.02).astype(np.float32)
    x[77 * n:78 * n] = pruned("fp32", n // 4, 0.05, 702).view(np.float32)
    t = torch.from_numpy(x).cuda()
    c = Z.compress(t, chunk_bytes=65536)
    assert [m for m in modes(c.to_bytes()) if m != (1, 0, 0, 0)] == [(SPARSE,) * 4]
    decode_every_way(c, t)
    v = np.zeros((16, n, 4), np.uint8)
    for k in range(16):                      # group sets coded and raw
        for byte in range(4):
            v[k, :, byte] = (g.integers(0, 4, n) if k >> byte & 1 else g.integers(0, 256, n))
    t = torch.from_numpy(v.reshape(-1)).cuda().view(torch.float32)
    c = Z.compress(t, chunk_bytes=65536)
    assert c.to_bytes() == O.compress(v.reshape(-1), O.FP32, 65536, Z.default_lanes(O.FP32, 65536))
    decode_every_way(c, t)


@pytest.mark.gpu
@pytest.mark.parametrize("chunk", [1 << 20, 8 << 20, 16 << 20])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
def test_deltas_in_large_chunks(chunk, dtype):
    """Bitmaps of more than a stage, of two and of four groups."""
    from paper_2411_05239_gb300 import zipnn as Z
    g = np.random.default_rng(703)
    v = chunk // 16 + 1251
    low = [127, 3] if dtype == torch.bfloat16 else [63, 63, 63, 3]    # bits that change, by byte
    x = g.integers(0, 256, (v, 16), dtype=np.uint8) & np.resize(np.array(low, np.uint8), 16)
    x[g.random(v) >= 0.3] = 0
    base = torch.from_numpy(pruned("bf16", v, 1.0, 704)).cuda()
    t = (base ^ torch.from_numpy(x.reshape(-1)).cuda()).view(dtype)
    base = base.view(dtype)
    c = Z.delta(t, base, chunk_bytes=chunk)
    m = modes(c.to_bytes())[0]
    assert m == (SPARSE,) * len(m)
    decode_every_way(c, t, base)


# -- 256 codes of 8 bits: uniform bytes in the live vectors


def flat_groups(s: bytes) -> list[int]:
    """Payload offsets of the coded groups whose twelve counts are stored as 0."""
    G, nch = struct.unpack_from("<II", s, 24)
    P = struct.unpack_from("<Q", s, 32)[0]
    ent = [struct.unpack_from("<QIBB", s, 64 + 16 * i) for i in range(nch * G)]
    return [P + e[0] for e in ent if e[2] in (1, SPARSE) and s[P + e[0]:P + e[0] + 12] == bytes(12)]


FLAT = [("u8", 0.1), ("u8", 0.3), ("u8", 0.6), ("u8", 0.9), ("fp16", 0.3), ("fp16", 0.6),
        ("fp32", 0.3), ("fp32", 0.6), ("fp32", 0.9)]


@pytest.mark.parametrize("kind,live", FLAT)
def test_oracle_codes_uniform_live_bytes(kind, live):
    x = pruned(kind, 3 * 16384 + 55, live, 800)
    s = O.compress(x, CODE[kind], 262144)
    at = flat_groups(s)
    assert at and all(s[a + 12:a + 268] == bytes(range(256)) for a in at)
    assert np.array_equal(O.decompress(s), x)
    for k in (12, 77, 267):                  # any other symbols under zero counts: refused
        bad = bytearray(s)
        bad[at[0] + k] ^= 1
        with pytest.raises(O.OracleError):
            O.decompress(bytes(bad))


@pytest.mark.gpu
@pytest.mark.parametrize("kind,live", FLAT)
def test_uniform_live_bytes(kind, live):
    from paper_2411_05239_gb300 import zipnn as Z
    dt = CODE[kind]
    x = pruned(kind, 3 * 16384 + 55, live, 800)
    t = torch.from_numpy(x).cuda().view(Z.CODE_TO_TORCH[dt])
    want = O.compress(x, dt, 262144, Z.default_lanes(dt, 262144))
    c = Z.compress(t)
    assert c.to_bytes() == want
    decode_every_way(c, t)
    for k in (12, 77, 267):
        bad = torch.frombuffer(bytearray(want), dtype=torch.uint8).cuda()
        bad[flat_groups(want)[0] + k] ^= 1
        out = torch.empty_like(t)
        Z.decompress(Z.wrap(bad, bad.numel()), out)
        with pytest.raises(Z.ZipnnError) as e:
            Z.sync_status()
        assert e.value.status == -3
