"""GPU parity of LSH banding at the edges of its forms: object counts around
the one-CTA-per-band sort and the tiles of the large one, key rows that are
the signature rows themselves and packed ones (1-, 2- and 4-byte lanes, up to
128 bytes), buckets shorter and longer than the staged rows and batches, with
the full keep record, a partial one and none.  The candidate set is the
oracle's; cosine pairs come in order of (band, key, x, y)."""
import numpy as np
import pytest
import torch

import oracle as O

pytestmark = pytest.mark.gpu
dev = torch.device("cuda")


def candidates(B, ctx, sig, kind, rows, bands, rec_bytes):
    N = sig.shape[0]
    t = torch.from_numpy(np.ascontiguousarray(sig).view(np.int32)).to(dev)
    full = B.blsh_lsh_candidates_workspace(N, kind, rows, bands)
    base = full - 64 * N * bands
    ws = torch.full((base + min(rec_bytes, 64 * N * bands),), 0xA5, dtype=torch.uint8, device=dev)
    n = torch.zeros(1, dtype=torch.int64, device=dev)
    B.blsh_lsh_candidates(ctx, t, kind, rows, bands, None, n, ws)
    assert B.blsh_status(ctx) == (B.ETRUNC if int(n.item()) else 0)
    pairs = torch.full((max(1, int(n.item())), 2), -1, dtype=torch.int32, device=dev)
    B.blsh_lsh_candidates(ctx, t, kind, rows, bands, pairs, n, ws)
    assert B.blsh_status(ctx) == 0
    return pairs[: int(n.item())].cpu().numpy().view(np.uint32)


def packed(p):
    return (p[:, 0].astype(np.uint64) << np.uint64(32)) | p[:, 1]


def cosine_keys(sig, rows, bands):
    bits = np.unpackbits(np.ascontiguousarray(sig).view(np.uint8), axis=1, bitorder="little")
    w = (1 << np.arange(rows, dtype=np.uint64))
    return np.stack([(bits[:, b * rows:(b + 1) * rows].astype(np.uint64) * w).sum(1) for b in range(bands)], 1)


def near_duplicates(rng, N, words, flip):
    """Rows drawn around N / 20 centres, every bit flipped with probability flip."""
    centres = rng.integers(0, 1 << 32, (max(1, N // 20), words), dtype=np.uint64).astype(np.uint32)
    noise = np.packbits(rng.random((N, 32 * words)) < flip, axis=1).view(np.uint32)
    return centres[rng.integers(0, len(centres), N)] ^ noise


@pytest.mark.parametrize("N", [2, 31, 33, 300, 4096, 4097, 6001])
@pytest.mark.parametrize("rows,bands", [(8, 5), (8, 64), (16, 3), (16, 62), (32, 2), (5, 13), (12, 33), (20, 17), (6, 1)])
def test_cosine(B, ctx, N, rows, bands):
    rng = np.random.default_rng(N + rows)
    sig = near_duplicates(rng, N, 32, 0.02)
    want = O.lsh_candidates(sig, O.COSINE, rows, bands)
    got = candidates(B, ctx, sig, 1, rows, bands, 1 << 40)
    assert len(got) == len(want) and np.array_equal(np.sort(packed(got)), np.sort(packed(want)))
    if len(got):
        key = cosine_keys(sig, rows, bands)
        same = key[got[:, 0]] == key[got[:, 1]]
        band = same.argmax(1)
        k = key[got[:, 0], band]
        assert same.any(1).all() and (got[:, 0] < got[:, 1]).all()
        order = np.lexsort((got[:, 1], got[:, 0], k, band))
        assert np.array_equal(order, np.arange(len(got)))
    for rec in (0, 8 * N):
        assert np.array_equal(candidates(B, ctx, sig, 1, rows, bands, rec), got)


@pytest.mark.parametrize("N", [2, 40, 4096, 4097, 6001])
@pytest.mark.parametrize("rows,bands", [(1, 1), (1, 3), (2, 16), (3, 32), (2, 40)])
def test_jaccard(B, ctx, N, rows, bands):
    rng = np.random.default_rng(N + bands)
    # values with a power law: a few long buckets and many short ones
    sig = np.minimum(rng.zipf(1.3, (N, 96)), N).astype(np.uint32)
    if rows == 1:
        sig = (sig + rng.integers(0, max(1, N // 50), (N, 96))).astype(np.uint32)
    want = O.lsh_candidates(sig, O.JACCARD, rows, bands)
    got = candidates(B, ctx, sig, 0, rows, bands, 1 << 40)
    assert len(got) == len(want) and np.array_equal(np.sort(packed(got)), np.sort(packed(want)))
    for rec in (0, 8 * N):
        assert np.array_equal(candidates(B, ctx, sig, 0, rows, bands, rec), got)


@pytest.mark.parametrize("kind,rows,bands", [(1, 8, 5), (1, 16, 62), (1, 12, 20), (0, 2, 4), (0, 2, 32)])
def test_long_buckets(B, ctx, kind, rows, bands):
    """Buckets of thousands of objects, cut into segments: 4,500 of 5,200
    objects agree on the last band, a third of those on band 1 as well."""
    rng = np.random.default_rng(rows + bands)
    N = 5200
    sig = rng.integers(0, 1 << 32, (N, 64), dtype=np.uint64).astype(np.uint32)
    chosen = rng.permutation(N)[:4500]
    for band, who in ((bands - 1, chosen), (1, chosen[::3])):
        if kind == 0:
            sig[np.ix_(who, np.arange(band * rows, (band + 1) * rows))] = 7
        else:
            bits = np.unpackbits(sig.view(np.uint8), axis=1, bitorder="little")
            bits[np.ix_(who, np.arange(band * rows, (band + 1) * rows))] = 1
            sig = np.packbits(bits, axis=1, bitorder="little").view(np.uint32)
    want = O.lsh_candidates(sig, O.COSINE if kind else O.JACCARD, rows, bands)
    assert len(want) > 10_000_000
    got = candidates(B, ctx, sig, kind, rows, bands, 1 << 40)
    assert len(got) == len(want) and np.array_equal(np.sort(packed(got)), np.sort(packed(want)))
    for rec in (0, 64 * N):   # no record: every chunk by its own warp, in the same order
        assert np.array_equal(candidates(B, ctx, sig, kind, rows, bands, rec), got)


@pytest.mark.parametrize("N", [2019, 2028, 2035, 2040, 2047, 2049, 2050])
@pytest.mark.parametrize("kind,rows,band", [(1, 16, 1), (1, 16, 2), (0, 2, 1), (0, 2, 2)])
def test_long_bucket_past_a_band_edge(B, ctx, N, kind, rows, band):
    """About as many objects as a chunk may have partners before it is cut into
    segments, nearly all of them in one bucket of a band whose first position
    lies inside a chunk of 32: the bucket's end is N + (N * band) % 32
    positions from the chunk's start."""
    rng = np.random.default_rng(N)
    sig = rng.permutation(1 << 16)[: N * 8].reshape(N, 8).astype(np.uint32) if kind == 0 else \
        np.stack([rng.permutation(1 << 16)[:N] for _ in range(8)], 1).astype(np.uint16).view(np.uint32)
    if kind == 0:
        sig[3:, band * rows:(band + 1) * rows] = 7
    else:
        sig.view(np.uint16)[3:, band] = 7
    want = O.lsh_candidates(sig, O.COSINE if kind else O.JACCARD, rows, 3)
    assert len(want) >= (N - 3) * (N - 4) // 2
    got = candidates(B, ctx, sig, kind, rows, 3, 1 << 40)
    assert len(got) == len(want) and np.array_equal(np.sort(packed(got)), np.sort(packed(want)))
    for rec in (0, 8 * N):
        assert np.array_equal(candidates(B, ctx, sig, kind, rows, 3, rec), got)


def test_scan_in_one_launch_up_to_8192_entries(B, ctx):
    """The pairs' offsets are a scan of one entry per 32 positions: one launch up
    to 8,192 of them, three from 8,193 on (all else is the same)."""
    launches = []
    for N in (32_768, 32_769):
        sig = torch.from_numpy(np.random.default_rng(N).integers(0, 1 << 31, (N, 4)).astype(np.int32)).to(dev)
        ws = torch.empty(B.blsh_lsh_candidates_workspace(N, 1, 16, 8), dtype=torch.uint8, device=dev)
        n = torch.zeros(1, dtype=torch.int64, device=dev)
        before = B.blsh_launch_count(ctx)
        B.blsh_lsh_candidates(ctx, sig, 1, 16, 8, None, n, ws)
        launches.append(B.blsh_launch_count(ctx) - before)
        assert B.blsh_status(ctx) == B.ETRUNC and int(n) > 0
    assert launches[1] - launches[0] == 2
