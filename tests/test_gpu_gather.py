"""Gather and fused compose + gather where their work split can go wrong.

A warp copies a run of up to 32 grid rows as one sequence of 16-byte vectors,
so the edges are: the shortest row (one vector), odd vector counts, the
longest row, fewer rows than a run, runs that end within a warp's last load,
and row counts around a whole round of warps.  The gather is a copy, so the
result must equal plain indexing bit for bit.
"""

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


def offsets(counts):
    return torch.tensor([0] + counts, dtype=torch.int64, device=DEV).cumsum(0)


@pytest.mark.parametrize("dtype,dim,counts", [
    (torch.float32, 4, [1]),                       # one vector per row, one row
    (torch.bfloat16, 8, [7, 0, 1, 9]),
    (torch.bfloat16, 24, [300, 41]),               # 3 vectors per row
    (torch.bfloat16, 200, [1000, 1, 33]),          # 25
    (torch.float32, 772, [511, 2]),                # 193
    (torch.float32, 16384, [19]),                  # 4096, the longest row
    (torch.bfloat16, 64, [152 * 3 * 8 * 8 + 1]),   # about one round of runs
    (torch.bfloat16, 16, [40000, 39999]),          # several rounds
    (torch.bfloat16, 40, [9, 0, 70, 1, 0, 0, 33, 2]),            # 8 images: offsets searched in place
    (torch.float32, 40, [0, 9, 0, 70, 1, 0, 33, 2, 500]),        # 9: from shared memory
    (torch.bfloat16, 8, [3] * 256),
    (torch.bfloat16, 8, [3, 1, 0] * 85 + [4, 5]),                # 257: in place again
    (torch.bfloat16, 8, [200000, 77777]),          # several rounds of runs of 32 rows
    (torch.bfloat16, 248, [700, 3, 29000]),        # 31 vectors: 24 rows, on the near side of the rule
    (torch.bfloat16, 256, [700, 3, 29000]),        # 32: 8 rows
    (torch.bfloat16, 512, [70000, 1, 50001]),      # more than 120 MB: runs of 3 rows
    (torch.float32, 1540, [9000, 10600]),          # of one row
])
def test_gather_equals_indexing(mpm, dtype, dim, counts):
    gen = torch.Generator(device=DEV).manual_seed(5)
    goff = offsets(counts)
    kept = [(n + 1) // 2 for n in counts]          # merged rows per image
    mid = [(3 * n + 3) // 4 for n in counts]       # rows between two insertions
    moff, off1 = offsets(kept), offsets(mid)
    z = torch.randn(sum(kept) + 3, dim, generator=gen, device=DEV).to(dtype)

    def local_map(rows, span):
        return torch.cat([torch.randint(0, max(s, 1), (n,), generator=gen, device=DEV) for n, s in zip(rows, span)]).int()

    image = torch.repeat_interleave(torch.arange(len(counts), device=DEV), torch.tensor(counts, device=DEV))
    r = local_map(counts, kept)
    status = torch.zeros(2, dtype=torch.int32, device=DEV)
    out = mpm.unmerge_gather(z, moff, r, goff, device_status=status)
    assert torch.equal(out, z[moff[image] + r])

    m1, m2 = local_map(counts, mid), local_map(mid, kept)
    composed = m2[off1[image] + m1]
    got_map = torch.full_like(m1, -9)
    out = mpm.compose_gather(z, moff, m1, goff, m2, off1, out_map=got_map, device_status=status)
    assert torch.equal(got_map, composed)
    assert torch.equal(out, z[moff[image] + composed])
    assert int(status[0]) == 0

    # A bad entry in the middle of a run: its row is zero, its neighbours are whole.
    bad = len(r) // 2
    r[bad] = 1 << 30
    out = mpm.unmerge_gather(z, moff, r, goff, device_status=status)
    want = z[moff[image] + torch.where(r < (1 << 30), r, torch.zeros_like(r))]
    want[bad] = 0
    assert torch.equal(out, want)
    assert status.tolist() == [6, bad]
