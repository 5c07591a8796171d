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


@pytest.mark.parametrize("dim", [4, 8, 12, 60, 68, 128, 132, 196, 256, 260, 512, 516, 1024, 1028, 4100])
def test_row_lengths(mpm, dim):
    rng = np.random.default_rng(dim)
    means = rng.standard_normal((9, dim))
    x = means[rng.integers(0, 9, 300)] + 0.3 * rng.standard_normal((300, dim))
    check(mpm, x.astype(np.float32))


@pytest.mark.parametrize("dim", [8, 100, 132])
def test_non_finite_rows_that_are_padded(mpm, dim):
    """Rows whose fp16 parts end in padding: a row with a NaN or an infinity spoils no other row's cosines."""
    rng = np.random.default_rng(dim)
    x = (rng.standard_normal((77, dim)) + 1.0).astype(np.float32)
    x[20, dim - 1] = np.nan
    x[76, 0] = np.inf
    nn, score = (t.cpu().numpy() for t in mpm.nearest_neighbors(torch.from_numpy(x).to(DEV),
                                                                torch.tensor([0, 77], device=DEV)))
    good = np.setdiff1d(np.arange(77), [20, 76])
    assert nn[20] == nn[76] == -1 and not np.isin(nn[good], [20, 76]).any()
    s = oracle.cosine_affinity(x[good].astype(np.float64))
    chosen = s[np.arange(75), np.searchsorted(good, nn[good])]
    np.testing.assert_allclose(score[good], chosen, rtol=0, atol=bound(dim))
    assert np.all(s.max(axis=1) - chosen <= 2 * bound(dim))


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


def lone_features(counts, dim, power, seed):
    """Images of normal tokens whose first two rows (where they have them) hold a feature of their own, 2^power."""
    rng = np.random.default_rng(seed)
    x = rng.standard_normal((sum(counts), dim))
    x[:, :2] = 0.0
    for a, n in zip(np.cumsum([0] + counts), counts):
        for r in range(min(n, 2)):
            x[a + r, r] = 2.0 ** power
    return x.astype(np.float32), np.cumsum([0] + counts)


@pytest.mark.parametrize("power", [12, 24, 44, 90])
@pytest.mark.parametrize("dim,counts,chunk", [
    (8, [40, 1, 0, 33], 0),
    (12, [2, 2, 3], 0),
    (196, [300, 2], 0),
    (768, [129], 0),
    (68, [700], 256),
])
def test_rows_with_a_huge_feature_of_their_own(mpm, dim, counts, chunk, power):
    """Their cosines come from the small features alone, down to 2^-90 of the row's norm: the errors stay
    relative to the terms that are added, as fp32's, and every row's neighbour is as good as the best.
    (Cosines below fp32's range come back as 0.)"""
    x, off = lone_features(counts, dim, power, seed=dim + power)
    nn, score = mpm.nearest_neighbors(torch.from_numpy(x).to(DEV), torch.from_numpy(off).to(DEV), chunk=chunk)
    nn, score = nn.cpu().numpy(), score.cpu().numpy()
    for a, n in zip(off, counts):
        run = chunk or max(n, 1)
        for c0 in range(0, n, run):
            img = x[a + c0:a + min(n, c0 + run)].astype(np.float64)
            if len(img) == 1:
                assert nn[a + c0] == -1
                continue
            s = oracle.cosine_affinity(img)
            got = nn[a + c0:a + c0 + len(img)] - c0
            chosen = s[np.arange(len(img)), got]
            unit = img / np.linalg.norm(img, axis=1, keepdims=True)
            terms = np.abs(unit) @ np.abs(unit).T      # what rounding errors are relative to
            tol = bound(dim) * terms
            error = np.abs(score[a + c0:a + c0 + len(img)] - chosen)
            assert np.all(error <= tol[np.arange(len(img)), got] + 2.0 ** -148)
            assert np.all(s - chosen[:, None] <= tol + tol[np.arange(len(img)), got][:, None])


@pytest.mark.parametrize("dim,images,spare,chunk", [
    (12, 1, 0, 0),         # one launch for the merge's tail
    (196, 256, 0, 0),
    (12, 300, 400, 0),     # its own launch before the scan
    (100, 257, 300, 0),
    (96, 3, 0, 256),       # the triples are the images' last chunks
    (96, 5, 0, 256),
])
def test_merge_pairs_decided_by_small_features(mpm, dim, images, spare, chunk):
    """Triples (-v, v, v + a feature of its own 2^44): the cosine of the last two is tiny, yet each is the other's
    neighbour, so they are a pair in every image."""
    rng = np.random.default_rng(dim + images)
    head = chunk and 2 * rng.standard_normal((chunk, dim))
    parts, counts = [], []
    for _ in range(images):
        v = rng.standard_normal(dim)
        v[0] = 0.0
        own = v.copy()
        own[0] = 2.0 ** 44
        img = np.stack([-v, v, own])
        parts.append(np.concatenate([head, img]) if chunk else img)
        counts.append(len(parts[-1]))
    x = np.concatenate(parts).astype(np.float32)
    off = torch.from_numpy(np.cumsum([0] + counts)).to(DEV)
    xd = torch.cat([torch.from_numpy(x), torch.zeros(spare, dim)]).to(DEV)
    ws = mpm.new_workspace(xd.shape[0], images, dim, xd.dtype, DEV)
    for stage_events in ([None, True] if not chunk else [None]):
        events = [torch.cuda.Event(enable_timing=True) for _ in range(8)] if stage_events else None
        for e in events or []:
            e.record()
        out, out_off, rmap = mpm.merge(xd, off, workspace=ws, chunk=chunk, stage_events=events)
        assert mpm.device_status(ws) == 0
        rmap, out, out_off = rmap.cpu().numpy(), out.cpu().numpy(), out_off.cpu().numpy()
        for b, (n, a) in enumerate(zip(counts, np.cumsum([0] + counts))):
            local = rmap[a + n - 3:a + n]
            assert local[2] == local[1] == local[0] + 1, b
            assert out_off[b + 1] - out_off[b] == local[1] + 1
            want = (x[a + n - 2] + x[a + n - 1]) * np.float32(0.5)
            assert np.array_equal(out[out_off[b] + local[1]], want)


def test_images_of_rows_with_huge_features_of_their_own(mpm):
    """Every cosine lies below fp32's range (2^-200); the order of the small features' products still decides."""
    rng = np.random.default_rng(12)
    x = np.abs(rng.standard_normal((20, 32))) + 0.1
    x[:, :20] = np.eye(20) * 2.0 ** 100
    x = x.astype(np.float32)
    nn, _ = mpm.nearest_neighbors(torch.from_numpy(x).to(DEV), torch.tensor([0, 20], device=DEV))
    s = oracle.cosine_affinity(x.astype(np.float64))
    best = np.sort(s, axis=1)
    assert np.all(best[:, -1] > best[:, -2] * (1 + 2 * bound(32)))
    assert np.array_equal(nn.cpu().numpy(), s.argmax(axis=1))


@pytest.mark.parametrize("dim,rms", [(16, 1.88e-7), (20, 2.70e-7), (64, 5.57e-7)])
def test_error_is_no_larger_than_that_of_three_tf32_products(mpm, dim, rms):
    """Clustered rows with one feature 300 times the others, where fp16 products lost most: the rms error of the
    best cosines against fp64.  `rms` is what the products of two tf32 parts per value gave on such rows, over
    8000 of them (the mean over fewer moves by 2%)."""
    rng = np.random.default_rng(dim)
    errors = []
    for _ in range(8):
        x = rng.standard_normal((12, dim))[rng.integers(0, 12, 1000)] + 0.3 * rng.standard_normal((1000, dim))
        x[:, dim // 2] *= 300.0
        x = x.astype(np.float32)
        nn, score = mpm.nearest_neighbors(torch.from_numpy(x).to(DEV), torch.tensor([0, 1000], device=DEV))
        unit = x.astype(np.float64)
        unit /= np.linalg.norm(unit, axis=1, keepdims=True)
        errors.append(score.cpu().numpy() - (unit * unit[nn.cpu().numpy()]).sum(axis=1))
    assert np.sqrt(np.mean(np.square(errors))) <= rms


@pytest.mark.parametrize("n", [64, 1500])
def test_orthogonal_rows(mpm, n):
    """Cosines of exactly 0 everywhere: every row's neighbour is the lowest other index, so only rows 0 and 1 pair up."""
    x = torch.zeros(n, 1536, device=DEV)
    x[torch.arange(n), torch.arange(n)] = 3.0
    off = torch.tensor([0, n], device=DEV)
    nn, score = mpm.nearest_neighbors(x, off)
    assert nn.tolist() == [1] + [0] * (n - 1) and not score.any()
    out, out_off, rmap = mpm.merge(x, off)
    assert out_off.tolist() == [0, n - 1]
    assert rmap.tolist() == [0, 0] + list(range(1, n - 1))


def test_capacity_past_the_last_image_changes_nothing(mpm):
    """Small merges with spare rows: what the workspace holds for those is nobody's key, whatever it looks like."""
    rng = np.random.default_rng(2)
    x = torch.zeros(300, 64)
    x[:100] = torch.from_numpy(rng.standard_normal((100, 64)).astype(np.float32))
    xd, off = x.to(DEV), torch.tensor([0, 60, 100], device=DEV)
    results = []
    for fill in (0, 0x7F, 0x80, 0xFF):
        ws = mpm.new_workspace(300, 2, 64, xd.dtype, DEV)
        ws.fill_(fill)
        out, rmap = torch.full_like(xd, 7.0), torch.full((300,), -5, dtype=torch.int32, device=DEV)
        _, out_off, _ = mpm.merge(xd, off, workspace=ws, out_tokens=out, out_map=rmap)
        assert mpm.device_status(ws) == 0
        results.append((out, out_off, rmap))
    for r in results[1:]:
        assert all(torch.equal(a, b) for a, b in zip(results[0], r))


def test_bad_rows_after_an_undecided_one_are_reported(mpm):
    """A long image among short ones is scanned in rounds; one undecided row in the first must not hide a row without
    a neighbour (here a NaN) in a later one."""
    rng = np.random.default_rng(9)
    counts = [5000] + [4] * 200
    x = rng.standard_normal((sum(counts), 16)).astype(np.float32)
    x[:, 0] = 0.0
    x[3, 0] = 2.0 ** 60
    off = torch.from_numpy(np.cumsum([0] + counts)).to(DEV)
    ws = mpm.new_workspace(len(x), len(counts), 16, torch.float32, DEV)
    for bad in (None, 4000, 3500):
        xd = torch.from_numpy(x).to(DEV)
        if bad is not None:
            xd[bad, 2] = float("nan")
        nn, _ = mpm.nearest_neighbors(xd, off, chunk=256)
        out, out_off, rmap = mpm.merge(xd, off, workspace=ws, chunk=256)
        assert mpm.device_status(ws) == (0 if bad is None else 6)
        part, nn = rmap[:5000].cpu().numpy(), nn[:5000].cpu().numpy()
        assert np.array_equal(part, oracle.compact_map(oracle.mutual_partners(nn))[0])


def test_images_of_tiny_rows(mpm):
    """Norms far below the floor of 1e-12: cosines scale with the neighbour's norm, in the oracle as here."""
    rng = np.random.default_rng(6)
    x = (rng.standard_normal((12, 48))[rng.integers(0, 12, 400)] + 0.3 * rng.standard_normal((400, 48))) * 1e-20
    x = x.astype(np.float32)
    nn, score = (t.cpu().numpy() for t in mpm.nearest_neighbors(torch.from_numpy(x).to(DEV),
                                                                torch.tensor([0, 400], device=DEV)))
    s = oracle.cosine_affinity(x.astype(np.float64))
    chosen = s[np.arange(400), nn]
    np.testing.assert_allclose(score, chosen, rtol=bound(48), atol=0)
    assert np.all(s.max(axis=1) <= chosen * (1 + 2 * bound(48)))
