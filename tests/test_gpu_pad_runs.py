"""Pad and unpad where their split into rows or runs of rows can go wrong:
padded lengths below, at and just past a run, the shortest and longest rows,
odd vector counts, empty images, many images, and images longer than the
padded length.  Both are copies, so everything is bit-exact."""

from __future__ import annotations

import pytest
import torch

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


@pytest.mark.parametrize("dtype,dim,counts,max_len", [
    (torch.bfloat16, 8, [1], 1),                        # one vector
    (torch.float32, 4, [7, 0, 3], 7),
    (torch.bfloat16, 24, [8, 1, 0, 8], 8),
    (torch.bfloat16, 200, [9, 2], 9),
    (torch.float32, 16384, [3, 5], 6),                  # the longest rows
    (torch.bfloat16, 64, [3] * 5000, 3),                # many short images
    (torch.bfloat16, 16, [2000, 1500, 0, 1999] * 40, 2001),   # several rounds of the whole GPU
    (torch.bfloat16, 72, [30, 90, 10], 41),             # one image is cut
    (torch.bfloat16, 64, [900] * 200, 900),             # runs of 24 rows
    (torch.bfloat16, 1024, [65, 700, 0] * 30, 701),     # 128 vectors, the most with four in flight
    (torch.float32, 516, [300, 299] * 40, 300),         # 129 vectors
    # Either side of the rule that chooses between runs and a row a warp.
    (torch.bfloat16, 384, [300, 290] * 10, 301),        # 48 vectors, more rows than warps: runs
    (torch.bfloat16, 384, [50, 0, 49], 50),             # fewer: a row a warp
    (torch.bfloat16, 392, [300, 290] * 10, 301),        # 49 vectors, few rows a warp: a row a warp
    (torch.bfloat16, 768, [150, 120] * 85, 151),        # 96 vectors, many: runs
    (torch.bfloat16, 776, [150, 120] * 85, 151),        # 97: a row a warp, four vectors in flight
    (torch.bfloat16, 1032, [40] + [0, 33] * 20, 36),     # 129: six in flight; one image is cut
])
def test_runs(mpm, dtype, dim, counts, max_len):
    gen = torch.Generator(device=DEV).manual_seed(8)
    off = torch.tensor([0] + counts, device=DEV).cumsum(0)
    x = torch.randn(sum(counts), dim, generator=gen, device=DEV).to(dtype)
    status = torch.zeros(2, dtype=torch.int32, device=DEV)
    out = torch.full((len(counts), max_len, dim), 9.0, dtype=dtype, device=DEV)
    mask = torch.full((len(counts), max_len), 7, dtype=torch.uint8, device=DEV)
    padded, mask, stats = mpm.pad_batch(x, off, max_len, out=out, mask=mask, device_status=status)
    t = torch.arange(max_len, device=DEV)
    live = t[None, :] < torch.tensor(counts, device=DEV)[:, None]
    at = (off[:-1, None] + t[None, :])[live]
    want = torch.zeros_like(padded)
    want[live] = x[at]
    assert torch.equal(padded, want)
    assert torch.equal(mask, live.to(torch.uint8))
    assert stats.tolist() == [min(counts), max(counts), sum(counts)]
    cut = [b for b, n in enumerate(counts) if n > max_len]
    assert status.tolist() == ([6, cut[0]] if cut else [0, 0])

    back = torch.full_like(x, 5.0)
    mpm.unpad_batch(padded, off, out=back, device_status=status)
    expect = torch.full_like(x, 5.0)   # rows of an image past max_len stay as they are
    expect[at] = x[at]
    assert torch.equal(back, expect)
