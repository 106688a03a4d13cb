"""The decoder's shared-memory stage at the limits of its sizing rule (needs a
GB300): every launch must get a stage that the device has, and every chunk must
come back (ZipNN Sec. 2.3), however long its sub-streams are."""
from __future__ import annotations

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
