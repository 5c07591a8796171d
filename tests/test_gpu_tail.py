"""A small merge's one-launch tail (mutual check, compaction and pair average
of at most 1024 rows and 256 images) against the two-launch path.  The same
images in a buffer of more than 1024 rows take the two launches, so both
paths must give the same bits, whatever the images, offsets and chunks."""

from __future__ import annotations

import pytest
import torch

from workloads import make_custom

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


def both_paths(mpm, x, off, chunk=0):
    """(out, out_offsets, map, status) of the one-launch and of the two-launch tail."""
    results = []
    used = x.shape[0]
    for rows in (used, 1200):
        xs = torch.zeros(rows, x.shape[1], dtype=x.dtype, device=DEV)
        xs[:used] = x
        ws = mpm.new_workspace(rows, off.numel() - 1, x.shape[1], x.dtype, DEV)
        ws.fill_(0x5A)
        out = torch.full_like(xs, 7.0)
        out_off = torch.full((off.numel(),), -5, dtype=torch.int64, device=DEV)
        rmap = torch.full((rows,), -5, dtype=torch.int32, device=DEV)
        mpm.merge(xs, off, workspace=ws, out_tokens=out, out_offsets=out_off, out_map=rmap, chunk=chunk)
        results.append((out[:used], out_off, rmap[:used], mpm.device_status(ws)))
    return results


def assert_same(one, two):
    assert torch.equal(one[1], two[1])
    assert torch.equal(one[2], two[2])
    # Bit for bit (tokens may hold NaN); rows past the last merged token stay untouched in both.
    assert torch.equal(one[0].view(torch.uint8), two[0].view(torch.uint8))
    assert one[3] == two[3]


@pytest.mark.parametrize("dtype,dim,counts,chunk", [
    ("bf16", 64, [1], 0),
    ("bf16", 8, [2, 1], 0),
    ("bf16", 200, [255, 1, 256], 0),
    ("f32", 192, [1024], 0),                     # the largest
    ("bf16", 768, [1023, 1], 0),
    ("f32", 68, [0, 0, 33, 0, 700, 0], 0),       # empty images everywhere
    ("bf16", 16, [4] * 256, 0),                  # the most images
    ("bf16", 16, [3] * 257, 0),                  # one more: two launches either way
    ("bf16", 64, [1000], 256),
    ("bf16", 64, [257, 513, 1], 256),            # tokens alone in their chunk
    ("f32", 36, [300, 300], 1 << 33),            # a chunk longer than 32 bits
])
def test_one_launch_equals_two(mpm, dtype, dim, counts, chunk):
    batch = make_custom(counts, dim, dtype, seed=17 + dim)
    off = torch.from_numpy(batch.offsets).to(DEV)
    assert_same(*both_paths(mpm, batch.tokens.to(DEV), off, chunk))


def test_identical_and_special_tokens(mpm):
    """Exact ties, zero rows and non-finite rows (which have no neighbour and are reported)."""
    x = torch.ones(600, 32, device=DEV)
    x[100:200] = 0
    off = torch.tensor([0, 350, 600], device=DEV)
    assert_same(*both_paths(mpm, x.to(torch.bfloat16), off))
    x[7, 3] = float("nan")
    x[400, 0] = float("inf")
    one, two = both_paths(mpm, x, off)
    assert_same(one, two)
    assert one[3] == 6


@pytest.mark.parametrize("bad", [[0, 100, 50, 150], [5, 60, 150], [0, -7, 150], [3, 3, 3]])
def test_bad_offsets(mpm, bad):
    gen = torch.Generator(device=DEV).manual_seed(2)
    x = torch.randn(150, 64, generator=gen, device=DEV).to(torch.bfloat16)
    one, two = both_paths(mpm, x, torch.tensor(bad, dtype=torch.int64, device=DEV))
    assert_same(one, two)
    assert one[3] == 6


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("bad", [[0, 150, 100], [0, 150, 40, 100], [0, 100, -3], [0, 1 << 40, 149]])
def test_results_do_not_depend_on_the_workspace_when_the_last_offset_is_not_the_largest(mpm, bad, dtype):
    """Rows from the last offset on belong to no image: nothing is computed from what the workspace held for them."""
    gen = torch.Generator(device=DEV).manual_seed(4)
    off = torch.tensor(bad, dtype=torch.int64, device=DEV)
    for rows in (150, 1200):
        x = torch.randn(rows, 64, generator=gen, device=DEV).to(dtype)
        results = []
        for fill in (0x00, 0x5A, 0xFF):
            ws = mpm.new_workspace(rows, len(bad) - 1, 64, dtype, DEV)
            ws.fill_(fill)
            out = torch.full_like(x, 7.0)
            rmap = torch.full((rows,), -5, dtype=torch.int32, device=DEV)
            _, out_off, _ = mpm.merge(x, off, workspace=ws, out_tokens=out, out_map=rmap)
            results.append((out, out_off, rmap, mpm.device_status(ws)))
            assert torch.all(rmap[max(bad[-1], 0):] == -5)
            assert results[-1][3] == 6
        for one in results[1:]:
            assert_same(results[0], one)
