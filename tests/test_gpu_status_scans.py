"""The passes that scan statuses, on both sides of their rules: compaction by
one CTA and by many, Lite's collection with four and sixteen tiles a group,
and the resumed pairs with their words read ahead or not, against the oracle
or the unlimited call."""
import numpy as np
import pytest
import torch

import oracle as O

pytestmark = pytest.mark.gpu
dev = torch.device("cuda")


@pytest.mark.parametrize("P", [15, 16, 16_384, 16_385, 131_071, 131_072, 131_073, 700_001])
@pytest.mark.parametrize("offset, used", [(0, None), (3, None), (0, 0.4)])
def test_compaction(B, ctx, P, offset, used):
    rng = np.random.default_rng(P + offset)
    st = rng.choice([0, 1, 2, 3, 31, 32, 252, 254, 255], P).astype(np.uint8)
    n = P if used is None else int(P * used)
    keep = 1 << 1 | 1 << 3 | 1 << 31
    want = O.compact(st[:n], keep)
    store = torch.zeros(P + offset, dtype=torch.uint8, device=dev)
    store[offset:] = torch.from_numpy(st).to(dev)
    count = None if used is None else torch.tensor([n], dtype=torch.int64, device=dev)
    for cap in (P, max(1, len(want) // 2)):
        out = torch.full((cap,), -1, dtype=torch.int64, device=dev)
        n_out = torch.zeros(1, dtype=torch.int64, device=dev)
        B.blsh_compact(ctx, store[offset:], keep, out, n_out, P_dev=count)
        assert B.blsh_status(ctx) == (B.ETRUNC if len(want) > cap else 0)
        assert int(n_out) == len(want)
        m = min(cap, len(want))
        assert np.array_equal(out[:m].cpu().numpy(), want[:m]) and bool((out[m:] == -1).all())


def test_lite_collection_groups(B, ctx):
    """9e7 pairs in one call, and in two calls that each take the shorter
    groups: the same statuses and similarities."""
    torch.manual_seed(5)
    P, N = 90_000_001, 4000
    base = torch.randint(-2**31, 2**31, (50, 16), dtype=torch.int32, device=dev)
    sig = base[torch.randint(0, 50, (N,), device=dev)].contiguous()
    noise = torch.rand(N, 16, device=dev) < 0.3
    sig[noise] = torch.randint(-2**31, 2**31, (int(noise.sum()),), dtype=torch.int32, device=dev)
    pairs = torch.randint(0, N, (P, 2), dtype=torch.int32, device=dev)
    indptr = torch.arange(0, 5 * N + 1, 5, dtype=torch.int64, device=dev)
    indices = (torch.arange(5 * N, device=dev, dtype=torch.int32) % 5) * 7
    values = torch.rand(5 * N, device=dev)
    tab = B.blsh_tables_build(ctx, B.make_params(kind=1, t=0.8, k=32, n_max=512, h=128))
    res = []
    for cut in ([0, P], [0, P // 2 // 16 * 16, P]):
        st = torch.full((P,), 77, dtype=torch.uint8, device=dev)
        sim = torch.full((P,), -1.0, dtype=torch.float64, device=dev)
        for a, b in zip(cut, cut[1:]):
            B.blsh_verify_lite(ctx, tab, pairs[a:b], sig, indptr, indices, values, st[a:b], sim[a:b])
            assert B.blsh_status(ctx) == 0
        res.append((st, sim))
    assert torch.equal(res[0][0], res[1][0]) and torch.equal(res[0][1], res[1][1])
    assert int((res[0][1] >= 0).sum()) > 1000


@pytest.mark.parametrize("kind, k", [(0, 32), (0, 64), (1, 32), (1, 64), (1, 128)])
@pytest.mark.parametrize("P", [1, 511, 30_001])
def test_resumed_pairs(B, ctx, kind, k, P):
    rng = np.random.default_rng(P + k)
    N, n_max, limit = 700, 2048 if kind else 512, 128
    W = n_max if kind == 0 else n_max // 32
    # pairs that agree in about the threshold's share of the hashes stay open past the limit
    sig = rng.integers(0, 2**32, (8, W), dtype=np.uint32)[rng.integers(0, 8, N)]
    if kind == 0:
        sig = np.where(rng.random((N, W)) < 0.2, rng.integers(0, 2**32, (N, W), dtype=np.uint32), sig)
    else:
        flips = np.packbits(rng.random((N, W * 32)) < 0.13, axis=1).view(np.uint32)
        sig = sig ^ flips
    t32 = lambda x: torch.from_numpy(np.ascontiguousarray(x).view(np.int32)).to(dev)
    pt, st32 = t32(rng.integers(0, N, (P, 2)).astype(np.uint32)), t32(sig)
    tab = B.blsh_tables_build(ctx, B.make_params(kind=kind, t=0.65, k=k, n_max=n_max, h=limit))
    ip = torch.arange(N + 1, dtype=torch.int64, device=dev)
    ix = torch.arange(N, dtype=torch.int32, device=dev)
    val = torch.ones(N, device=dev) if kind else None
    z = lambda t, v=0: torch.full((P,), v, dtype=t, device=dev)
    fresh = lambda: [z(torch.uint8, 77), z(torch.int16), z(torch.int16), z(torch.float32, -1.0),
                     torch.zeros(tab.levels, dtype=torch.int64, device=dev)]
    want, got = fresh(), fresh()
    B.blsh_verify(ctx, tab, pt, st32, *want)
    B.blsh_verify_both_capped(ctx, tab, limit, pt, st32, *got, ip, ix, val, z(torch.uint8, 77), z(torch.float64),
                              torch.zeros(N, dtype=torch.uint8, device=dev))
    opened = int((got[0] == B.NEEDS_HASHES).sum())
    B.blsh_verify_resume(ctx, tab, pt, st32, *got)
    assert B.blsh_status(ctx) == 0
    for a, b in zip(got, want):
        assert torch.equal(a, b)
    assert opened > P // 50 or P == 1


@pytest.mark.parametrize("P", [0, 1, 4095, 4096, 4097, 8193, 126_977, 131_072])
@pytest.mark.parametrize("keep", [0, 1 << 4, 0xffffffff])
@pytest.mark.parametrize("offset", [0, 1, 15])
def test_compaction_in_one_launch(B, ctx, P, keep, offset):
    """Tiles of 4,096 statuses from a 16-byte boundary on, all kept, some and
    none, and a device count at and past the end of a tile."""
    st = (np.arange(P) * 7 % 37).astype(np.uint8)   # 32 .. 36 are never kept
    store = torch.full((P + offset + 16,), 4, dtype=torch.uint8, device=dev)   # kept, but outside
    dst = store[offset:offset + P]
    dst.copy_(torch.from_numpy(st))
    for used in sorted({0, min(P, 5), max(0, 4096 - offset) if P >= 4096 else 0, P // 2 // 4096 * 4096, P // 2, P}):
        want = O.compact(st[:used], keep)
        out = torch.full((P,), -1, dtype=torch.int64, device=dev)
        n_out = torch.full((1,), 5, dtype=torch.int64, device=dev)
        B.blsh_compact(ctx, dst, keep, out, n_out, P_dev=torch.tensor([used], dtype=torch.int64, device=dev))
        assert B.blsh_status(ctx) == 0 and int(n_out) == len(want)
        assert np.array_equal(out[: len(want)].cpu().numpy(), want) and bool((out[len(want):] == -1).all())


@pytest.mark.parametrize("P", [60_000, 131_072])
def test_compaction_of_kept_statuses_takes_no_single_block(B, ctx, P):
    """Everything kept: 8 bytes a status written by all the blocks (a single one
    takes 40 to 80 us, two launches 12)."""
    st = torch.full((P,), 3, dtype=torch.uint8, device=dev)
    out, n_out = torch.zeros(P, dtype=torch.int64, device=dev), torch.zeros(1, dtype=torch.int64, device=dev)
    times = []
    for _ in range(4):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(20):
            B.blsh_compact(ctx, st, 1 << 3, out, n_out)
        b.record()
        b.synchronize()
        times.append(a.elapsed_time(b) / 20)
    assert int(n_out) == P and torch.equal(out, torch.arange(P, device=dev))
    assert min(times) < 0.025, times


@pytest.mark.parametrize("offset", [0, 1, 15])
@pytest.mark.parametrize("P", [131_073, 2_500_000])
def test_compaction_from_any_address(B, ctx, P, offset):
    st = (np.arange(P) * 11 % 41).astype(np.uint8)
    store = torch.full((P + offset + 16,), 4, dtype=torch.uint8, device=dev)
    dst = store[offset:offset + P]
    dst.copy_(torch.from_numpy(st))
    for used in (0, 3, 700, P - 1, P):
        want = O.compact(st[:used], 0x80000015)
        out = torch.full((P,), -1, dtype=torch.int64, device=dev)
        n_out = torch.full((1,), 5, dtype=torch.int64, device=dev)
        B.blsh_compact(ctx, dst, 0x80000015, out, n_out, P_dev=torch.tensor([used], dtype=torch.int64, device=dev))
        assert B.blsh_status(ctx) == 0 and int(n_out) == len(want)
        assert np.array_equal(out[: len(want)].cpu().numpy(), want) and bool((out[len(want):] == -1).all())


@pytest.mark.parametrize("offset", [0, 7])
@pytest.mark.parametrize("P", [131_073, 1_300_000])
@pytest.mark.parametrize("share", [0.2, 0.25, 0.3, 1.0])
def test_compaction_of_full_and_empty_ranges(B, ctx, P, share, offset):
    """Shares of kept statuses on both sides of the line between the two write
    forms, next to ranges that keep few, and a buffer that ends inside a full
    range."""
    rng = np.random.default_rng(P + offset)
    p = np.where(np.arange(P) // 50_000 % 2 == 0, share, 0.001)
    st = np.where(rng.random(P) < p, 2, 1).astype(np.uint8)
    store = torch.full((P + offset + 16,), 2, dtype=torch.uint8, device=dev)
    dst = store[offset:offset + P]
    dst.copy_(torch.from_numpy(st))
    want = O.compact(st, 1 << 2)
    for cap in (P, len(want), 6_007):
        out = torch.full((cap,), -1, dtype=torch.int64, device=dev)
        n_out = torch.full((1,), 5, dtype=torch.int64, device=dev)
        B.blsh_compact(ctx, dst, 1 << 2, out, n_out)
        assert int(n_out) == len(want)
        assert (B.blsh_status(ctx) == 0) == (cap >= len(want))
        got = out.cpu().numpy()
        assert np.array_equal(got[: len(want)], want[:cap]) and (got[len(want):] == -1).all()
