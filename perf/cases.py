"""Timed cases: what programs that use this library have it do.

A case is one or more images' worth of tokens and the calls a program makes
on them.  ``kind`` is
  "merge"  1 to 3 insertions and the way back to the token grid: merge for
           each insertion (in chunks if ``chunk`` > 0, on the library's own
           scratch if ``no_alloc``), then unmerge_gather, or compose_gather
           over the last two maps with the earlier ones composed before;
  "pad"    the padded batch that dense attention takes, and back to packed;
  "nn"     nearest neighbours with their cosines.
``counts`` lists the images' token counts ("64x1024" is 64 images of 1024).

Inputs.  Tokens are Voronoi images: K sites on the patch grid, each with an
N(0, I) mean, tokens = their site's mean + sigma * N(0, I), stored as bf16 or
fp32.  The input of a later insertion is the merged tokens plus
N(0, 0.05^2), in the place of the encoder blocks between two insertions.
A token whose two best cosines lie within GAP of each other is drawn again:
two correct implementations, whose cosines differ by a few 1e-6, may pair
such a token differently, and every row after it would shift.  With decided
inputs, maps and offsets are whole numbers that have to be the same, and a
merged token is one correctly rounded mean, so those cases are compared
exactly.
"""

from __future__ import annotations

import math

import torch

import paper_2604_05718_gb300 as mpm

GAP = 2e-5
STAGE_NOISE = 0.05
DTYPES = {"bf16": torch.bfloat16, "f32": torch.float32}
# Merged tokens per input token on these inputs (0.84 to 0.87); work() only.
KEPT = 0.86
# Largest drawn case: tokens x features, and flops of one pass (fp32 passes cost several times a bf16 one's).
MAX_ELEMS = {"bf16": 64 * 1024 * 768, "f32": 32 * 1024 * 768}
MAX_FLOPS = {"bf16": 1.2e11, "f32": 3e10}
NO_ALLOC_BYTES = 8 << 20


def _case(name, counts, dim, dtype, kind="merge", insertions=2, sites=32, sigma=0.3, chunk=0, no_alloc=False):
    return {"name": name, "kind": kind, "counts": counts, "dim": dim, "dtype": dtype, "insertions": insertions,
            "sites": sites, "sigma": sigma, "chunk": chunk, "no_alloc": no_alloc}


def listed():
    return [
        # A handful of small crops, one of them a single token: launches and host time count.
        _case("tiny_ragged", "300,1,129", 128, "bf16", sites=8),
        # One 512 x 512 image through a tiny encoder in fp32, one insertion.
        _case("vit_t_single", "1024", 192, "f32", insertions=1),
        # One image at a time on a server that must not allocate.
        _case("single_no_alloc", "1024", 768, "bf16", sites=64, no_alloc=True),
        # One high-resolution image (56 x 56 patches, not a multiple of any tile).
        _case("hires_single", "3136", 1024, "bf16", sites=96, sigma=0.25),
        # Batched inference at 512 x 512, small and base encoder.
        _case("vit_s", "32x1024", 384, "bf16"),
        _case("vit_b", "64x1024", 768, "bf16", sites=64),
        # 768 x 768 images through a large encoder.
        _case("vit_l", "16x2304", 1024, "bf16", sites=96, sigma=0.25),
        # A ragged batch of images of mixed resolution, 32 x 32 to 64 x 64 patches.
        _case("mixed", "1600,4096,2x1600,1024,1600,1024,2304,2x4096,1024,3x1600,3x4096,5x1024,2x2304", 768, "bf16",
              sites=64),
        # fp32 tokens, batched, one insertion.
        _case("vit_b_f32", "64x1024", 768, "f32", insertions=1, sites=64),
        # Similarity statistics of a ragged fp32 batch of odd sizes.
        _case("nn_f32_ragged", "1369,577,1025,197,2209,784,1", 196, "f32", kind="nn"),
        # One very large image (128 x 128 patches): similarity in chunks.
        _case("large_chunked", "16384", 768, "bf16", sites=128, chunk=1024),
        # Merged images padded to the longest for dense attention, and back.
        _case("pad_unpad", ",".join(str(820 + (37 * b) % 58) for b in range(64)), 768, "bf16", kind="pad"),
    ]


def draw(rng):
    kind = rng.choices(["merge", "pad", "nn"], [8, 1, 1])[0]
    dtype = rng.choices(["bf16", "f32"], [7, 3])[0]
    step = 8 if dtype == "bf16" else 4
    dim = step * max(1, round(2 ** rng.uniform(6, 10.2) / step))
    top = round(2 ** rng.uniform(6, 12.3))
    batch = round(2 ** rng.uniform(0, 6))
    low = rng.choice([1.0, 0.8, 0.4])
    counts = [max(1, round(top * rng.uniform(low, 1.0))) for _ in range(batch)]
    chunk = 256 * rng.randint(1, 6) if kind == "merge" and top > 512 and rng.random() < 0.2 else 0
    insertions = rng.choices([1, 2, 3], [3, 6, 1])[0]
    case = _case("", "", dim, dtype, kind, insertions, rng.randint(8, 128), round(rng.uniform(0.15, 0.5), 3), chunk)
    while len(counts) > 1:
        case["counts"] = ",".join(map(str, counts))
        if sum(counts) * dim <= MAX_ELEMS[dtype] and work(case)["flops"] <= MAX_FLOPS[dtype]:
            break
        counts.pop()
    case["counts"] = ",".join(map(str, counts))
    # Small latency-critical calls: half of them without any allocation.
    per_row = 20 + (8 * dim if dtype == "f32" else 0)
    if kind == "merge" and not chunk and sum(counts) * per_row + 20 * batch + 4096 < NO_ALLOC_BYTES and \
            sum(counts) <= 2048:
        case["no_alloc"] = rng.random() < 0.5
    del case["name"]
    return case


def _counts(case):
    out = []
    for part in case["counts"].split(","):
        k, _, n = part.rpartition("x")
        out += [int(n)] * int(k or 1)
    return out


def _runs(counts, chunk):
    """Lengths of the runs of tokens that are compared with one another."""
    out = []
    for n in counts:
        while chunk and n > chunk:
            out.append(chunk)
            n -= chunk
        out.append(n)
    return out


# ---------------------------------------------------------------------------
# Inputs (plain torch, on the GPU)
# ---------------------------------------------------------------------------
def _offsets(counts, dev):
    return torch.tensor([0] + counts, dtype=torch.int64, device=dev).cumsum(0)


def _voronoi(counts, dim, sites, sigma, gen, dev):
    """fp32 means of every token's site, and the function that adds fresh noise."""
    means = []
    for n in counts:
        side = max(1, math.ceil(math.sqrt(n)))
        k = max(1, min(sites, n // 4))
        pos = torch.rand(k, 2, generator=gen, device=dev) * side
        idx = torch.arange(n, device=dev)
        at = torch.stack([idx // side, idx % side], 1).float() + 0.5
        site = torch.cdist(at, pos, compute_mode="donot_use_mm_for_euclid_dist").argmin(1)
        means.append(torch.randn(k, dim, generator=gen, device=dev)[site])
    return torch.cat(means)


def _neighbours(x, runs, dtype):
    """(neighbour's packed row or -1, best cosine, gap to the second best) of every row, within its run."""
    rows = x.shape[0]
    nbr = torch.full((rows,), -1, dtype=torch.int64, device=x.device)
    best = torch.full((rows,), -math.inf, dtype=dtype, device=x.device)
    gap = torch.full((rows,), math.inf, dtype=dtype, device=x.device)
    k, a = 0, 0
    while k < len(runs):
        n, m = runs[k], 1
        while k + m < len(runs) and runs[k + m] == n and (m + 1) * n * n <= 1 << 27:
            m += 1
        if n > 1:
            xs = x[a:a + m * n].view(m, n, -1).to(dtype)
            xs = xs / xs.norm(dim=2, keepdim=True).clamp_min(1e-12)
            s = xs @ xs.transpose(1, 2)
            s.diagonal(dim1=1, dim2=2).fill_(-math.inf)
            v, j = s.topk(2, dim=2)
            base = a + n * torch.arange(m, device=x.device)[:, None]
            nbr[a:a + m * n] = (j[:, :, 0] + base).reshape(-1)
            best[a:a + m * n] = v[:, :, 0].reshape(-1)
            gap[a:a + m * n] = (v[:, :, 0] - v[:, :, 1]).reshape(-1)
        k, a = k + m, a + m * n
    return nbr, best, gap


def _decided(fresh, runs):
    """Tokens from ``fresh()``, with every row drawn again whose two best cosines lie within GAP."""
    x = fresh()
    for _ in range(40):
        near = _neighbours(x, runs, torch.float32)[2] < GAP
        if not bool(near.any()):
            break
        x = torch.where(near[:, None], fresh(), x)
    return x


def _merged(x, nbr, off, acc):
    """One insertion on packed tokens, given the neighbours: tokens (in ``acc``), counts per image, local map."""
    rows = torch.arange(x.shape[0], device=x.device)
    has = nbr >= 0
    pair = has & (nbr[nbr.clamp_min(0)] == rows)
    rep = ~pair | (rows < nbr)
    ids = rep.cumsum(0) - 1
    image = torch.searchsorted(off[1:], rows, right=True)
    kept = torch.zeros(off.numel() - 1, dtype=torch.int64, device=x.device).index_add_(0, image, rep.long())
    start = kept.cumsum(0) - kept
    local = torch.where(rep, ids, ids[nbr.clamp_min(0)]) - start[image]
    first = rows[rep]
    partner = torch.where(pair, nbr, rows)[rep]
    return (x[first].to(acc) + x[partner].to(acc)) * 0.5, kept, local


def _inputs(case, seed):
    """Each insertion's input tokens and counts, and the counts after the last."""
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev).manual_seed(int(seed))
    dtype, counts = DTYPES[case["dtype"]], _counts(case)
    means = _voronoi(counts, case["dim"], case["sites"], case["sigma"], gen, dev)

    def fresh(center, sigma):
        return (center + sigma * torch.randn(center.shape, generator=gen, device=dev)).to(dtype)

    if case["kind"] == "pad":
        return [(fresh(means, case["sigma"]), counts)], counts
    stages = []
    center, sigma = means, case["sigma"]
    for _ in range(case["insertions"] if case["kind"] == "merge" else 1):
        runs = _runs(counts, case["chunk"])
        x = _decided(lambda: fresh(center, sigma), runs)
        stages.append((x, counts))
        x_out, kept, _ = _merged(x, _neighbours(x, runs, torch.float32)[0], _offsets(counts, dev), torch.float32)
        center, sigma, counts = x_out.to(dtype).float(), STAGE_NOISE, kept.tolist()
    return stages, counts


def _room(x, rows):
    """x with zero rows after it, ``rows`` in all."""
    return torch.cat([x, x.new_zeros(rows - x.shape[0], *x.shape[1:])])


# ---------------------------------------------------------------------------
# The measured pass
# ---------------------------------------------------------------------------
def prepare(case, seed):
    stages, counts = _inputs(case, seed)
    x0 = stages[0][0]
    dev, rows, dim, batch = x0.device, x0.shape[0], x0.shape[1], len(counts)
    # A later insertion's tokens lie in a buffer of the first one's rows: the host does not know how many there are.
    st = {"kind": case["kind"], "x": [_room(x, rows) for x, _ in stages], "off": _offsets(stages[0][1], dev),
          "chunk": case["chunk"]}
    if case["kind"] == "pad":
        st["max_len"] = max(counts)
        return st
    st["ws"] = None if case["no_alloc"] else mpm.new_workspace(rows, batch, dim, x0.dtype, dev)
    # Buffers for every insertion's results, at the first insertion's rows; what a pass leaves unwritten stays zero.
    st["out"] = [(torch.zeros_like(x0), torch.zeros(batch + 1, dtype=torch.int64, device=dev),
                  torch.zeros(rows, dtype=torch.int32, device=dev)) for _ in stages]
    st["grid"] = torch.empty_like(x0)
    return st


def run(st):
    if st["kind"] == "pad":
        padded, mask, stats = mpm.pad_batch(st["x"][0], st["off"], st["max_len"])
        return padded, mask, stats, mpm.unpad_batch(padded, st["off"], rows=st["x"][0].shape[0])
    if st["kind"] == "nn":
        return mpm.nearest_neighbors(st["x"][0], st["off"], workspace=st["ws"])
    offs, maps = [st["off"]], []
    for x, (out, off, m) in zip(st["x"], st["out"]):
        if st["ws"] is None:
            mpm.merge_no_alloc(x, offs[-1], out, off, m)
        else:
            mpm.merge(x, offs[-1], workspace=st["ws"], out_tokens=out, out_offsets=off, out_map=m, chunk=st["chunk"])
        offs.append(off)
        maps.append(m)
    if len(maps) == 1:
        mpm.unmerge_gather(out, offs[1], maps[0], offs[0], out=st["grid"])
    else:
        m = maps[0]
        for k in range(1, len(maps) - 1):
            m = mpm.compose_maps(m, offs[0], maps[k], offs[k])
        mpm.compose_gather(out, offs[-1], m, offs[0], maps[-1], offs[-2], out=st["grid"])
    return st["out"], st["grid"]


def exact(case, seed):
    stages, _ = _inputs(case, seed)
    if case["kind"] == "pad":
        x, counts = stages[0]
        length = max(counts)
        padded = torch.zeros(len(counts), length, x.shape[1], dtype=torch.float64, device=x.device)
        mask = torch.zeros(len(counts), length, dtype=torch.uint8, device=x.device)
        for b, (n, part) in enumerate(zip(counts, x.double().split(counts))):
            padded[b, :n] = part
            mask[b, :n] = 1
        return padded, mask, torch.tensor([min(counts), length, sum(counts)]), x.double()
    done, to_merged, rows = [], None, stages[0][0].shape[0]
    for x, counts in stages:
        off = _offsets(counts, x.device)
        nbr, best, _ = _neighbours(x, _runs(counts, case["chunk"]), torch.float64)
        image = torch.searchsorted(off[1:], torch.arange(x.shape[0], device=x.device), right=True)
        if case["kind"] == "nn":
            return torch.where(nbr >= 0, nbr - off[image], nbr).int(), best
        x_out, kept, local = _merged(x, nbr, off, torch.float64)
        off_out = _offsets(kept.tolist(), x.device)
        to_here = local + off_out[image]
        to_merged = to_here if to_merged is None else to_here[to_merged]
        done.append((_room(x_out, rows), off_out, _room(local.int(), rows)))
    return done, done[-1][0][to_merged]


def work(case):
    counts, dim, e = _counts(case), case["dim"], 2 if case["dtype"] == "bf16" else 4
    rows = sum(counts)
    if case["kind"] == "pad":
        padded = len(counts) * max(counts)
        return {"bytes": (rows + padded) * dim * e + padded + (padded + rows) * dim * e, "flops": 0}
    total_bytes, flops, n, grid = 0, 0, float(rows), rows
    share = 1.0
    for _ in range(case["insertions"] if case["kind"] == "merge" else 1):
        # The off-diagonal half of the cosine matrix, within runs.
        runs = _runs([max(1, round(c * share)) for c in counts], case["chunk"])
        flops += sum(r * (r - 1) for r in runs) * dim
        if case["kind"] == "nn":
            return {"bytes": n * (dim * e + 8), "flops": flops}
        # Tokens in, merged tokens out, the map out.
        total_bytes += n * dim * e + KEPT * n * dim * e + 4 * n
        n, share = KEPT * n, KEPT * share
    # The merged tokens in, every map in, the grid out.
    total_bytes += n * dim * e + grid * dim * e + 4 * grid * case["insertions"]
    return {"bytes": total_bytes, "flops": flops}


def tolerance(case):
    if case["kind"] == "nn":
        return {"rel": 1.5e-5, "max": 1e-4}  # fp32 sums, 4e-6 off fp64 at 1000 features
    return "exact"
