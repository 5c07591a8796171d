"""Prep and pair average where their work split can go wrong: rows of every
length class of prep (one pass and several, full and partial load slots), row
counts around a block's and a wave's share, more images than the plan's one
pass takes, empty images at either end, and capacity beyond the used rows.
Checked against the oracle (bit-exact on decided rows)."""

from __future__ import annotations

import numpy as np
import pytest
import torch

from parity import check_merge_batch, to_f64
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


@pytest.mark.parametrize("dtype,dim,counts,spare", [
    ("bf16", 8, [1], 0),                      # 1 vector per row
    ("bf16", 256, [33, 0], 5),                # 32: the last of its class
    ("bf16", 264, [0, 40, 0, 7], 0),          # 33
    ("bf16", 512, [64, 1], 300),              # 64
    ("bf16", 520, [100], 0),                  # 65
    ("bf16", 768, [2, 3, 90], 1),             # 96
    ("bf16", 776, [130], 0),                  # 97
    ("bf16", 1024, [31, 31], 0),              # 128
    ("bf16", 1032, [50], 2),                  # 129: two passes
    ("bf16", 1536, [41], 0),                  # 192: two full passes of three vectors
    ("bf16", 1544, [41], 0),                  # 193: two passes of four
    ("bf16", 2056, [33], 1),                  # 257: three of three
    ("f32", 2052, [45, 1], 0),                # 513
    ("bf16", 16, [5] * 255, 0),               # as many images as the plan's block has threads, and one more
    ("bf16", 16, [5] * 256, 0),
    ("bf16", 16, [4, 0, 3] * 90, 17),
    ("bf16", 64, [300] * 20, 9000),           # more than a wave of rows, a third of them used
    # Capacity past 1024 rows: the pair average in its own launch, 4, 2 or 1 rows at a time.
    ("bf16", 8, [1], 1100),
    ("bf16", 256, [66, 1], 1100),
    ("bf16", 264, [35, 0, 1], 1100),
    ("bf16", 512, [64, 1], 1100),
    ("bf16", 768, [45], 1100),
    ("bf16", 776, [45], 1100),
    ("f32", 64, [700, 333, 2, 1], 40),
    ("bf16", 520, [101], 1000),
    ("f32", 256, [33, 0, 2], 1200),
    ("f32", 260, [34], 1200),
    ("bf16", 1024, [31, 31], 1000),
])
def test_merge_row_classes(mpm, dtype, dim, counts, spare):
    batch = make_custom(counts, dim, dtype, seed=91 + dim)
    x = torch.cat([batch.tokens, torch.full((spare, dim), 3.0, dtype=batch.tokens.dtype)]).to(DEV)
    off = torch.from_numpy(batch.offsets).to(DEV)
    ws = mpm.new_workspace(x.shape[0], batch.batch, dim, x.dtype, DEV)
    ws.fill_(0xA5)  # nothing may depend on what the workspace held
    nn, _ = mpm.nearest_neighbors(x, off, workspace=ws)
    ws.fill_(0x5A)
    out, out_off, rmap = mpm.merge(x, off, workspace=ws)
    assert mpm.device_status(ws) == 0
    rows = batch.rows
    st = check_merge_batch(batch.tokens.double().numpy(), batch.offsets, nn.cpu().numpy()[:rows],
                           rmap.cpu().numpy()[:rows], to_f64(out[:int(out_off[-1])]), out_off.cpu().numpy(), dtype,
                           f"{dtype} d={dim}")
    assert st.images == int(np.sum(np.asarray(counts) >= 0))
