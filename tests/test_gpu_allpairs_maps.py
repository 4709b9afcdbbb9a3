"""GPU parity of the prefix-filter candidates on both sides of their dispatch:
bit maps where the keys are many for the number of rows, sorted keys where
they are few, at map sizes around a word and a block, rows around the lengths
where the prefix computation changes, and truncated outputs.  Pair for pair
against the CPU oracle."""
import numpy as np
import pytest
import torch

import oracle as O
import synth

pytestmark = pytest.mark.gpu
dev = torch.device("cuda")


def rows_csr(lens, dim, seed, values):
    rng = np.random.default_rng(seed)
    rows = [np.sort(rng.choice(dim, n, replace=False)).astype(np.uint32) for n in lens]
    indptr = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    vals = None
    if values:
        v = [rng.uniform(0.1, 1.0, n) for n in lens]
        vals = np.concatenate([x / max(np.linalg.norm(x), 1e-9) for x in v]).astype(np.float32)
    return synth.CSR(indptr, np.concatenate(rows) if rows else np.zeros(0, np.uint32), vals, dim)


def candidates(B, ctx, csr, t, kind, cap_less=0):
    ip = torch.from_numpy(csr.indptr).to(dev)
    ix = torch.from_numpy(csr.indices.view(np.int32)).to(dev)
    val = None if kind == O.JACCARD else torch.from_numpy(csr.values).to(dev)
    N, nnz = csr.n, int(csr.indptr[-1])
    n_pairs, n_dups = (torch.zeros(1, dtype=torch.int64, device=dev) for _ in range(2))
    ws = torch.full((B.blsh_allpairs_workspace(N, nnz, csr.dim, 0),), 0xEE, dtype=torch.uint8, device=dev)
    B.blsh_allpairs_candidates(ctx, ip, ix, val, csr.dim, t, kind, None, n_pairs, ws, 0, n_dups)
    assert B.blsh_status(ctx) == 0
    dups = int(n_dups.item())
    if dups == 0:
        return np.zeros((0, 2), np.uint32), 0, []
    ws = torch.full((B.blsh_allpairs_workspace(N, nnz, csr.dim, dups),), 0xEE, dtype=torch.uint8, device=dev)
    pairs = torch.full((max(1, dups - cap_less), 2), -1, dtype=torch.int32, device=dev)
    B.blsh_timing_begin(ctx)
    B.blsh_allpairs_candidates(ctx, ip, ix, val, csr.dim, t, kind, pairs, n_pairs, ws, dups, n_dups)
    names = [n for n, _ in B.blsh_timing_end(ctx)]
    assert B.blsh_status(ctx) == (B.ETRUNC if int(n_pairs.item()) > pairs.shape[0] else 0)
    assert int(n_dups.item()) == dups
    return pairs.cpu().numpy().view(np.uint32), int(n_pairs.item()), names


@pytest.mark.parametrize("n", [2, 31, 32, 33, 257, 8200])
@pytest.mark.parametrize("kind", [O.JACCARD, O.COSINE])
def test_maps(B, ctx, n, kind):
    rng = np.random.default_rng(n)
    csr = rows_csr(rng.integers(0 if n > 2 else 20, 30, n), 300, n, kind == O.COSINE)
    want = O.allpairs_candidates(csr, 0.4, kind)
    got, k, names = candidates(B, ctx, csr, 0.4, kind)
    assert k == len(want) and np.array_equal(got[:k], want)
    assert (n == 2 and not names) or "ap_map_kernel (write pass)" in names   # (two rows may share no feature)


@pytest.mark.parametrize("kind", [O.JACCARD, O.COSINE])
def test_sorted_keys(B, ctx, kind):
    csr = rows_csr(np.full(3000, 6), 200000, 4, kind == O.COSINE)
    want = O.allpairs_candidates(csr, 0.3, kind)
    assert len(want) > 0
    got, k, names = candidates(B, ctx, csr, 0.3, kind)
    assert k == len(want) and np.array_equal(got[:k], want)
    assert "digit_scatter_kernel" in names


@pytest.mark.parametrize("kind", [O.JACCARD, O.COSINE])
def test_row_lengths_of_the_prefix(B, ctx, kind):
    csr = rows_csr([1, 31, 32, 33, 64, 96, 97, 127, 128, 129, 200, 4096, 4097, 0, 128, 128], 6000, 5, kind == O.COSINE)
    for t in (0.2, 0.7):
        want = O.allpairs_candidates(csr, t, kind)
        got, k, _ = candidates(B, ctx, csr, t, kind)
        assert k == len(want) and np.array_equal(got[:k], want)


def test_truncated_map_output(B, ctx):
    csr = rows_csr(np.full(300, 20), 200, 6, False)
    want = O.allpairs_candidates(csr, 0.5, O.JACCARD)
    dups = len(candidates(B, ctx, csr, 0.5, O.JACCARD)[0])
    less = dups - len(want) + 11
    got, k, _ = candidates(B, ctx, csr, 0.5, O.JACCARD, cap_less=less)
    assert k == len(want) and np.array_equal(got, want[:-11])


@pytest.mark.parametrize("dim, kept", [(700, True), (4500, False)])
@pytest.mark.parametrize("kind", [O.JACCARD, O.COSINE])
@pytest.mark.parametrize("cap_less", [0, 1000])
def test_maps_kept_or_formed_again(B, ctx, dim, kept, kind, cap_less):
    """The write pass from the maps the count pass kept, and where they do not
    fit the place of the key buffers (32 bytes a key)."""
    n = 6001
    csr = rows_csr(np.full(n, 3), dim, dim, kind == O.COSINE)
    want = O.allpairs_candidates(csr, 0.01, kind)   # every feature indexed: 4.5 n^2 / dim keys
    got, k, names = candidates(B, ctx, csr, 0.01, kind, cap_less)
    assert k == len(want) and "ap_map_kernel (write pass)" in names
    m = min(k, len(got))
    assert np.array_equal(got[:m], want[:m]) and np.all(got[m:] == 2**32 - 1)
    assert (n * n <= 256 * (len(got) + cap_less)) == kept


@pytest.mark.parametrize("n", [392_200, 393_200])
@pytest.mark.parametrize("kept", [True, False])
def test_maps_at_the_default_shared_memory(B, n, kept):
    """Maps of just under 48 KB, which with the kernels' own shared memory pass
    the launch default: kept for the write pass, and formed again."""
    i = np.arange(n)
    feats = np.sort(np.stack([i // 2, n // 2 + (i * 7919) % 190_000], 1), 1)
    csr = synth.CSR(np.arange(n + 1, dtype=np.int64) * 2, feats.ravel().astype(np.uint32), None, n // 2 + 190_000)
    want = O.allpairs_candidates(csr, 0.4, O.JACCARD)
    assert len(want) > n // 2
    max_dups = n * n // (256 if kept else 400) + 1
    ip, ix = torch.from_numpy(csr.indptr).to(dev), torch.from_numpy(csr.indices.view(np.int32)).to(dev)
    ws = torch.empty(B.blsh_allpairs_workspace(n, 2 * n, csr.dim, max_dups), dtype=torch.uint8, device=dev)
    pairs = torch.full((len(want) + 5, 2), -1, dtype=torch.int32, device=dev)
    n_pairs = torch.zeros(1, dtype=torch.int64, device=dev)
    ctx = B.Context(0)
    B.blsh_allpairs_candidates(ctx, ip, ix, None, csr.dim, 0.4, O.JACCARD, pairs, n_pairs, ws, max_dups)
    assert B.blsh_status(ctx) == 0 and int(n_pairs.item()) == len(want)
    assert np.array_equal(pairs[: len(want)].cpu().numpy().view(np.uint32), want)


@pytest.mark.parametrize("first,last", [(300, 1200), (0, 1000), (250, 1100), (1199, 1200)])
@pytest.mark.parametrize("kind", [O.JACCARD, O.COSINE])
@pytest.mark.parametrize("sparse", [False, True])
def test_some_rows_of_a_larger_csr(B, ctx, first, last, kind, sparse):
    """indptr a part of a larger one over the whole index array: the elements of
    the other rows, before indptr[0] and past indptr[N], count for nothing, in
    the bit maps as in the sorted keys."""
    csr = rows_csr(np.full(1200, 6), 60_000, 8, kind == O.COSINE) if sparse else \
        rows_csr(np.random.default_rng(9).integers(0, 30, 1200), 300, 9, kind == O.COSINE)
    part = csr.indptr[first:last + 1]
    s, e = part[0], part[-1]
    sub = synth.CSR(part - s, csr.indices[s:e], None if csr.values is None else csr.values[s:e], csr.dim)
    want = O.allpairs_candidates(sub, 0.3, kind)
    ip, ix = torch.from_numpy(part.copy()).to(dev), torch.from_numpy(csr.indices.view(np.int32)).to(dev)
    val = None if csr.values is None else torch.from_numpy(csr.values).to(dev)
    n_pairs, n_dups = (torch.zeros(1, dtype=torch.int64, device=dev) for _ in range(2))
    dups, names = 0, []
    for counted in (False, True):
        ws = torch.full((B.blsh_allpairs_workspace(last - first, ix.numel(), csr.dim, dups),), 0xEE, dtype=torch.uint8,
                        device=dev)
        pairs = torch.full((max(1, dups), 2), -1, dtype=torch.int32, device=dev) if counted else None
        B.blsh_timing_begin(ctx)
        B.blsh_allpairs_candidates(ctx, ip, ix, val, csr.dim, 0.3, kind, pairs, n_pairs, ws, dups, n_dups)
        names = [n for n, _ in B.blsh_timing_end(ctx)]
        assert B.blsh_status(ctx) == 0
        if not counted:
            dups = int(n_dups.item())
        if dups == 0:
            assert len(want) == 0
            return
    assert int(n_dups.item()) == dups and int(n_pairs.item()) == len(want)
    assert np.array_equal(pairs[: len(want)].cpu().numpy().view(np.uint32), want)
    assert ("digit_scatter_kernel" in names) == sparse


@pytest.mark.parametrize("n,length,by_lists", [(2000, 65, True), (2000, 69, False), (6000, 7, True), (6000, 8, False)])
@pytest.mark.parametrize("kind", [O.JACCARD, O.COSINE])
def test_count_only_by_lists_or_by_sorting(B, ctx, n, length, by_lists, kind):
    """The number of keys from either form of a count-only call, which walks
    lists only where n rows' every list is short enough in the worst case."""
    csr = rows_csr(np.full(n, length), 400, n + length, kind == O.COSINE)
    nnz = csr.indices.size
    assert (nnz * n <= 2**28) == by_lists
    indexed = O.allpairs_indexed(csr, 0.4, kind).astype(bool)
    # the keys: (row x, indexed feature f of x, row y > x with f)
    row = np.repeat(np.arange(n), length)
    has = np.zeros((n, csr.dim), bool)
    has[row, csr.indices] = True
    later = has[::-1].cumsum(0)[::-1] - has
    want = int(later[row[indexed], csr.indices[indexed]].sum())
    ip, ix = torch.from_numpy(csr.indptr).to(dev), torch.from_numpy(csr.indices.view(np.int32)).to(dev)
    val = None if kind == O.JACCARD else torch.from_numpy(csr.values).to(dev)
    n_pairs, n_dups = (torch.full((1,), 7, dtype=torch.int64, device=dev) for _ in range(2))
    ws = torch.full((B.blsh_allpairs_workspace(n, nnz, csr.dim, 0),), 0xEE, dtype=torch.uint8, device=dev)
    B.blsh_timing_begin(ctx)
    B.blsh_allpairs_candidates(ctx, ip, ix, val, csr.dim, 0.4, kind, None, n_pairs, ws, 0, n_dups)
    names = [k for k, _ in B.blsh_timing_end(ctx)]
    assert B.blsh_status(ctx) == 0 and int(n_pairs.item()) == 0 and int(n_dups.item()) == want > 0
    assert ("ap_map_kernel (keys)" in names) == by_lists and ("digit_scatter_kernel" in names) != by_lists


@pytest.mark.parametrize("n,maps", [(46_000, True), (60_000, False)])
def test_many_rows_of_few_keys(B, ctx, n, maps):
    """Around the number of rows from which maps that the key buffers' place
    cannot hold cost more than sorting the few keys there are."""
    length, dim = 10, 190_000
    rng = np.random.default_rng(n)
    feats = rng.integers(0, dim // length, (n, length)) + np.arange(length) * (dim // length)
    csr = synth.CSR(np.arange(n + 1, dtype=np.int64) * length, feats.ravel().astype(np.uint32), None, dim)
    want = O.allpairs_candidates(csr, 0.05, O.JACCARD)
    got, k, names = candidates(B, ctx, csr, 0.05, O.JACCARD)
    assert n * n <= 4096 * len(got) and n * n > 256 * len(got)
    assert k == len(want) and np.array_equal(got[:k], want)
    assert ("ap_map_kernel (write pass)" in names) == maps and ("digit_scatter_kernel" in names) != maps
