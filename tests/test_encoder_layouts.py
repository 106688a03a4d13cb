"""Encoder variants against the oracle's containers (needs a GB300).

The code builder keeps its lists in one, two, four or eight registers a lane by
the number of symbols; the packer has passes of its own for ragged chunks and
for delta chunks with two coded groups.  Every container must equal the oracle's
byte for byte (ZipNN Sec. 3.1, 3.2, 4.2) around those limits."""
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


def weights(shape: str, k: int) -> np.ndarray:
    i = np.arange(k, dtype=np.float64)
    if shape == "equal":                 # ties everywhere
        p = np.ones(k)
    elif shape == "steep":               # lengths at the 12-bit limit
        p = 0.6 ** np.minimum(i, 40)
    else:                                # a broad bell, as in quantised weights
        p = np.exp(-0.5 * ((i - k / 2) / (k / 7 + 1)) ** 2)
    return p / p.sum()


@pytest.mark.parametrize("k", [2, 3, 31, 32, 33, 34, 63, 64, 65, 66, 127, 128, 129, 130, 255, 256])
@pytest.mark.parametrize("shape", ["equal", "steep", "bell"])
def test_code_builds(k, shape):
    """Exactly k symbols, spread over the byte range, in three chunks."""
    g = np.random.default_rng(400 + k)
    syms = g.permutation(256)[:k].astype(np.uint8)
    x = syms[g.choice(k, size=2 * 65536 + 4099, p=weights(shape, k))]
    for c in range(0, x.size, 65536):
        x[c:c + k] = syms
    if shape == "equal":                 # equal counts, not only close ones
        x[:65536] = np.resize(syms, 65536)
    c = Z.compress(torch.from_numpy(x).cuda(), chunk_bytes=65536)
    assert c.to_bytes() == O.compress(x, Z.U8, 65536, Z.default_lanes(Z.U8, 65536))


def delta_of(kind: str, n: int) -> tuple[torch.Tensor, torch.Tensor]:
    """(next, base) BF16 whose XOR groups take HUFF or SPARSE: a share of
    changed 16-byte vectors (SPARSE) or of changed elements (HUFF)."""
    g = np.random.default_rng(n)
    hi_sparse, lo_sparse = kind[0] == "s", kind[1] == "s"
    changed = np.repeat(g.random((n + 7) // 8) < 0.05, 8)[:n]
    lo = np.where(changed if lo_sparse else g.random(n) < 0.3, g.integers(1, 9, n), 0)
    hi = np.where(changed if hi_sparse else g.random(n) < 0.3, g.integers(1, 5, n), 0)
    base = W.gaussian(n, 0.02, 410).view(torch.int16).numpy()
    nxt = base ^ (hi << 8 | lo).astype(np.int16)
    return torch.from_numpy(nxt).view(torch.bfloat16), torch.from_numpy(base).view(torch.bfloat16)


@pytest.mark.parametrize("kind", ["hh", "hs", "sh", "ss"])
@pytest.mark.parametrize("tail", [1, 8 * 33 + 5, 8 * 256, 70_001])
@pytest.mark.parametrize("chunk,lanes", [(262144, 0), (65536, 100), (262144, 512), (16384, 8)])
def test_delta_groups(kind, tail, chunk, lanes):
    nxt, base = delta_of(kind, chunk // 2 + tail)
    c = Z.delta(nxt.cuda(), base.cuda(), chunk_bytes=chunk, lanes=lanes)
    ln = lanes or O.default_lanes(Z.BF16, chunk, True)
    assert c.to_bytes() == O.delta(u8(nxt), u8(base), Z.BF16, chunk, ln)


def test_call_forms():
    """compress() on the current and on a given stream, of views, with and without
    the exact copy; decompress() into a contiguous view; refusals."""
    x = W.gaussian(300_000, 0.02, 420).cuda()
    want = O.compress(u8(x), Z.BF16, Z.DEFAULT_CHUNK, Z.default_lanes(Z.BF16, Z.DEFAULT_CHUNK))
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    strided = torch.stack([x, x], 1)[:, 0]
    got = [Z.compress(x), Z.compress(x, exact=False), Z.compress(x, stream=side),
           Z.compress(strided), Z.compress(x.view(3, 100_000)), Z.compress(x.requires_grad_())]
    with torch.cuda.stream(side):
        got.append(Z.compress(x))
    for c in got:
        assert c.to_bytes() == want
        assert (c.orig_nbytes, c.zs.lanes, c.is_delta) == (
            600_000, Z.default_lanes(Z.BF16, Z.DEFAULT_CHUNK), False)
    y = torch.zeros(16 + 300_000, dtype=torch.bfloat16, device="cuda")
    Z.decompress(got[0], y[16:])
    Z.sync_status()
    assert torch.equal(y[16:], x.detach())
    with pytest.raises(Z.ZipnnError):
        Z.decompress(got[0], y[1:300_001])      # two bytes off a 16-byte boundary
    with pytest.raises(ValueError):
        Z.compress(x.detach(), base=x.detach()[:5])
    with pytest.raises(ValueError):
        Z.compress(x.detach().cpu())
    with pytest.raises(RuntimeError):
        Z.compress(torch._neg_view(x.detach()))
