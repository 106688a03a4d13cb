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
