"""fp32 tokens through scaled fp16 high and low parts: row lengths at the
edges of the kernels (rows that are no whole 16 bytes in fp16, no multiple of
the MMA's 16 features or of a 64-feature stage, longer than a warp keeps in
registers) and rows far out of the usual range.

Bound on a cosine's error, from the arithmetic: the tensor cores add 16
products at a time, 3 ceil(D / 16) additions that each lose less than one
unit 2^-23 of the running sum (at most about 1); the split loses 2^-22 of
each factor, and the norms, the scaling and the final product a few units.
"""

from __future__ import annotations

import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu

DEV = "cuda"


def bound(dim: int) -> float:
    return (3 * -(-dim // 16) + 8) * 2.0 ** -23


@pytest.fixture(scope="module")
def mpm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2604_05718_gb300 as pkg
    from paper_2604_05718_gb300 import build

    build.build()
    pkg.library()
    return pkg


def check(mpm, x: np.ndarray, rows=None):
    """Neighbours and cosines of one image against the fp64 oracle, on `rows` (all by default)."""
    xd = torch.from_numpy(x).to(DEV)
    off = torch.tensor([0, len(x)], dtype=torch.int64, device=DEV)
    nn, score = mpm.nearest_neighbors(xd, off)
    nn, score = nn.cpu().numpy(), score.cpu().numpy()
    s = oracle.cosine_affinity(x.astype(np.float64))
    tol = bound(x.shape[1])
    rows = np.arange(len(x)) if rows is None else rows
    chosen = s[rows, nn[rows]]
    np.testing.assert_allclose(score[rows], chosen, rtol=0, atol=tol)
    assert np.all(s[rows].max(axis=1) - chosen <= 2 * tol)


@pytest.mark.parametrize("dim", [4, 8, 12, 60, 68, 196, 1024, 1028, 4100])
def test_row_lengths(mpm, dim):
    rng = np.random.default_rng(dim)
    means = rng.standard_normal((9, dim))
    x = means[rng.integers(0, 9, 300)] + 0.3 * rng.standard_normal((300, dim))
    check(mpm, x.astype(np.float32))


def test_rows_of_any_magnitude(mpm):
    """Rows scaled from 1e-9 to 1e30 (their squares overflow from 1e19 on): cosines do not change."""
    rng = np.random.default_rng(3)
    means = rng.standard_normal((5, 96))
    x = means[rng.integers(0, 5, 256)] + 0.3 * rng.standard_normal((256, 96))
    x *= 10.0 ** rng.integers(-9, 31, (256, 1))
    check(mpm, x.astype(np.float32))


@pytest.mark.parametrize("scale", [1.0, 1e25, 1e-18])
def test_small_features_of_rows_of_any_magnitude(mpm, scale):
    """Rows with a feature of their own 2^18 times the others: their cosines come from the small
    features alone.  The bound is relative: the split adds at most 2^-39 of a row's norm to each
    feature's error, 2^-21 of a small one."""
    rng = np.random.default_rng(7)
    x = np.abs(rng.standard_normal((128, 96))) + 0.5
    x[:, :4] = 0.0
    for r in range(4):
        x[r, r] = 2.0 ** 18
    x = (x * scale).astype(np.float32)
    xd = torch.from_numpy(x).to(DEV)
    nn, score = (t.cpu().numpy()[:4] for t in mpm.nearest_neighbors(xd, torch.tensor([0, 128], device=DEV)))
    s = oracle.cosine_affinity(x.astype(np.float64))[:4]
    np.testing.assert_allclose(score, s[np.arange(4), nn], rtol=bound(96) + 2.0 ** -21, atol=0)


def test_tiny_zero_and_non_finite_rows(mpm):
    """Rows below the norm's floor and zero rows score 0; a row with an infinity or NaN is nobody's neighbour."""
    rng = np.random.default_rng(4)
    x = (rng.standard_normal((200, 96)) + 1.0).astype(np.float32)
    x[7] = 0.0
    x[30] *= np.float32(1e-40)
    x[31] *= np.float32(1e-30)
    check(mpm, x)
    bad = [50, 51, 199]
    x[50, 3] = np.inf
    x[51, 0] = np.nan
    x[199, 95] = -np.inf
    xd = torch.from_numpy(x).to(DEV)
    off = torch.tensor([0, len(x)], dtype=torch.int64, device=DEV)
    nn, score = (t.cpu().numpy() for t in mpm.nearest_neighbors(xd, off))
    assert np.all(nn[bad] == -1)
    good = np.setdiff1d(np.arange(len(x)), bad)
    assert not np.isin(nn[good], bad).any()
    s = oracle.cosine_affinity(x[good].astype(np.float64))
    chosen = s[np.arange(len(good)), np.searchsorted(good, nn[good])]
    np.testing.assert_allclose(score[good], chosen, rtol=0, atol=bound(96))
