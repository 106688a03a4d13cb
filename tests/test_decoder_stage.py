"""The decoder's shared-memory stage at the limits of its sizing rule (needs a
GB300): every launch must get a stage that the device has, and every chunk must
come back (ZipNN Sec. 2.3), however long its sub-streams are."""
from __future__ import annotations

import struct

import pytest
import torch

from paper_2411_05239_gb300 import workloads as W
from paper_2411_05239_gb300 import zipnn as Z

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("lanes", [1, 2, 3])
@pytest.mark.parametrize("chunk", [140_000, 262_144, 280_000, 420_000])
def test_sub_streams_about_as_long_as_the_stage(chunk, lanes, dtype):
    t = W.gaussian(2 * chunk // dtype.itemsize - 1001, 0.02, 705, dtype).cuda()
    c = Z.compress(t, chunk_bytes=chunk, lanes=lanes)
    out = torch.zeros_like(t)
    for tune in (None, Z.tuning(threads=128), Z.tuning(parts=4)):
        Z.batch_decompress([c], [out], tune=tune)
        Z.sync_status()
        assert torch.equal(out.view(torch.uint8), t.view(torch.uint8))
        out.zero_()


@pytest.mark.parametrize("groups", [1, 2])
def test_starts_before_a_slice_are_corrupt(groups):
    """Chunks decoded in slices of their sub-streams (a plan stages 1 MiB chunks so:
    BF16 values of widely spread scales, one coded group, and FP16 holding BF16
    values, two): sub-streams that claim to start before their slice are reported, not
    read from whatever lies there."""
    if groups == 2:
        x = W.clean_fp16_from_bf16(600_000, seed=710, device="cuda")
    else:
        x = W.gaussian(600_000, 1.0, 711, torch.float32)
        x = (x * torch.exp2(torch.arange(600_000) % 40 - 20.0)).to(torch.bfloat16).cuda()
    c = Z.compress(x, chunk_bytes=1 << 20, lanes=1000)
    s = bytearray(c.to_bytes())
    P = struct.unpack_from("<Q", s, 32)[0]
    off, size, mode = struct.unpack_from("<QIB", s, 64)           # chunk 0, group 0
    assert mode == 1
    h = (12 + sum(s[P + off:P + off + 12]) + 3) // 4 * 4
    for t in range(990, 1000):
        struct.pack_into("<I", s, P + off + h + 4 * (t - 1), 5)
    out = torch.empty_like(x)
    for data, want in ((bytes(s), -3), (c.to_bytes(), 0)):
        buf = torch.frombuffer(bytearray(data), dtype=torch.uint8).cuda()
        p = Z.plan_decompress([Z.wrap(buf)], [out], tune=Z.tuning(parts=1))
        p.launch()
        if want:
            with pytest.raises(Z.ZipnnError) as e:
                Z.sync_status()
            assert e.value.status == want
        else:
            Z.sync_status()
            assert torch.equal(out.view(torch.uint8), x.view(torch.uint8))
        p.close()
