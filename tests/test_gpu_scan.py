"""The mutual check and compaction scan where its work split can go wrong.

An image's rows are split over a cluster of 1, 2, 4 or 8 blocks of 1024
threads with up to 4 rows per thread, in rounds.  The reference is the
oracle's pairing and left-to-right compaction of the library's own nearest
neighbours, so only the scan is under test and everything is exact.
"""

from __future__ import annotations

import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu

DEV = "cuda"


@pytest.fixture(scope="module")
def mpm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2604_05718_gb300 as pkg
    from paper_2604_05718_gb300 import build

    build.build()
    pkg.library()
    return pkg


@pytest.mark.parametrize("counts,chunk", [
    ([1], 0),
    ([1023, 1024, 1025], 0),          # one and two blocks, the last block with one row
    ([2048, 0, 2049], 0),
    ([4096], 0),
    ([8191], 256),                    # a cluster of 8, one row per thread
    ([8193], 256),                    # two rows per thread
    ([32768], 256),                   # a whole round
    ([32769 + 2048], 256),            # a second round with few rows
    ([12000] + [5] * 40, 512),        # one long image among short ones: rounds of one block
    ([3, 1, 2] * 400, 0),             # more images than a block has threads
    ([2] * 1024, 0),                  # the pair average adds up to 1024 counts itself
    ([2, 1, 0] * 341 + [3, 3], 0),    # 1025 images: the scan does
    ([2300] * 80, 256),               # too many images for two blocks each, four rows a thread
    ([2300] * 70, 256),               # few enough
    ([700], 1 << 40),                 # a chunk longer than any image
])
def test_scan_equals_the_oracles_compaction(mpm, counts, chunk):
    gen = torch.Generator(device=DEV).manual_seed(11)
    x = torch.randn(sum(counts), 16, generator=gen, device=DEV).to(torch.bfloat16)
    off_h = np.concatenate([[0], np.cumsum(counts)])
    off = torch.from_numpy(off_h).to(DEV)
    ws = mpm.new_workspace(x.shape[0], len(counts), 16, x.dtype, DEV)
    nn, _ = mpm.nearest_neighbors(x, off, workspace=ws, chunk=chunk)
    out, out_off, rmap = mpm.merge(x, off, workspace=ws, chunk=chunk)
    torch.cuda.synchronize()
    assert mpm.device_status(ws) == 0
    nn, rmap, xs = nn.cpu().numpy(), rmap.cpu().numpy(), x.float().cpu().numpy()
    kept = [0]
    rows = []
    for b in range(len(counts)):
        a0, a1 = off_h[b], off_h[b + 1]
        r, rep, partner = oracle.compact_map(oracle.mutual_partners(nn[a0:a1]))
        assert np.array_equal(rmap[a0:a1], r), b
        kept.append(kept[-1] + len(rep))
        img = xs[a0:a1]
        rows.append(np.where((partner >= 0)[:, None], (img[rep] + img[partner]) * np.float32(0.5), img[rep]))
    assert out_off.cpu().tolist() == kept
    want = torch.from_numpy(np.concatenate(rows)).to(torch.bfloat16)
    assert torch.equal(out[:kept[-1]].cpu(), want)
