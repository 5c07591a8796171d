"""The binding's device and stream handling: a device without an index, and
calls on a side stream while the default stream is busy."""

from __future__ import annotations

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mpm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2604_05718_gb300 as pkg
    from paper_2604_05718_gb300 import build

    build.build()
    pkg.library()
    return pkg


def test_device_without_an_index(mpm):
    from paper_2604_05718_gb300 import mpm as binding

    status = binding.selftest_wait_timeout(1000, device="cuda")
    torch.cuda.synchronize()
    assert status.tolist() == [7, 99]
    assert binding.no_alloc_device_status("cuda") == 0


def test_calls_run_on_the_current_stream(mpm):
    x = torch.zeros(512, 64, device="cuda", dtype=torch.bfloat16)
    off = torch.tensor([0, 512], device="cuda")
    src = torch.randn(512, 64, device="cuda").to(torch.bfloat16)
    want = mpm.merge(src, off)
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        torch.cuda._sleep(20_000_000)  # the merge below reads x only after the copy that follows this
        x.copy_(src)
        got = mpm.merge(x, off)
        grid = mpm.unmerge_gather(got[0], got[1], got[2], off)
    side.synchronize()
    assert torch.equal(got[1], want[1]) and torch.equal(got[2], want[2])
    assert torch.equal(grid, want[0][want[2].long()])
