"""Units of the packer that do not fit its fast passes, against the oracle's
containers (needs a GB300).

A chunk's bits are staged unit by unit (a unit: a part of one sub-stream) in
shared-memory slots of 1248 bits, and written out by the pass that the units'
sizes allow.  Every container must equal the oracle's byte for byte (ZipNN
Sec. 3.1, 3.2) wherever a unit is too long or too short for its chunk's pass."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import oracle as O
from paper_2411_05239_gb300 import zipnn as Z

pytestmark = pytest.mark.gpu


def fp32_units(lanes: int, chunks: int, seed: int) -> np.ndarray:
    """FP32 chunks of 256 KiB whose exponents take codes of two bits on average,
    but for one unit of some chunks, whose elements take rare exponents (codes
    of 11 bits, more than a slot holds); a ragged end with units under 32 bits."""
    g = np.random.default_rng(seed)
    n, T = 65536, lanes
    R, nvt = 512 // T, 16384 // T
    per = nvt // R
    x = g.integers(0, 1 << 32, size=chunks * n + 12 * T, dtype=np.uint32) & 0x807FFFFF
    e = (120 + g.geometric(0.5, size=x.size).clip(1, 8)).astype(np.uint32)
    for c in range(chunks):
        if c % 3 == 2:
            continue
        t, k = int(g.integers(T)), int(g.integers(R))
        v = t + (k * per + np.arange(per)) * T
        at = c * n + (v[:, None] * 4 + np.arange(4)).reshape(-1)
        e[at] = 100 + np.arange(at.size) % 20
    return x | e << 23


@pytest.mark.parametrize("lanes", [64, 128, 256])
def test_fp32_units_past_their_slots(lanes):
    x = fp32_units(lanes, 40, 500 + lanes)
    want = O.compress(x.view(np.uint8), O.FP32, 262144, lanes)
    t = torch.from_numpy(x.view(np.float32)).cuda()
    for _ in range(3):
        assert Z.compress(t, lanes=lanes).to_bytes() == want


def units16(lanes: int, chunks: int, seed: int) -> np.ndarray:
    """The same with 16-bit elements of eight to a vector (BF16's exponent bytes)."""
    g = np.random.default_rng(seed)
    n, T = 131072, lanes
    R, nvt = 512 // T, 16384 // T
    per = nvt // R
    x = g.integers(0, 1 << 16, size=chunks * n + 24 * T + 8, dtype=np.uint16) & 0x807F
    e = (120 + g.geometric(0.5, size=x.size).clip(1, 8)).astype(np.uint16)
    for c in range(chunks):
        if c % 3 == 2:
            continue
        t, k = int(g.integers(T)), int(g.integers(R))
        v = t + (k * per + np.arange(per)) * T
        e[c * n + (v[:, None] * 8 + np.arange(8)).reshape(-1)] = 100 + np.arange(8 * per) % 20
    return x | e << 7


@pytest.mark.parametrize("dtype", [O.BF16, O.FP16])
@pytest.mark.parametrize("lanes", [64, 128, 256, 512])
def test_units16_past_their_slots(lanes, dtype):
    x = units16(lanes, 40, 520 + lanes)
    want = O.compress(x.view(np.uint8), dtype, 262144, lanes)
    t = torch.from_numpy(x.view(np.int16)).cuda().view(Z.CODE_TO_TORCH[dtype])
    for encoder in (0, 0, 1):
        bc = Z.BatchCompressor([t], chunk_bytes=262144, lanes=lanes, encoder=encoder)
        bc()
        Z.sync_status()
        assert bc.containers()[0].to_bytes() == want
