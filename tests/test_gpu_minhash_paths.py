"""GPU parity of minhash on both sides of its dispatch: a CTA per set where
the sets are few, a warp per set otherwise, and the chunks of long sets around
the lengths where they begin.  Bit-exact against the CPU oracle."""
import numpy as np
import pytest
import torch

import oracle as O
import synth

pytestmark = pytest.mark.gpu
dev = torch.device("cuda")


def t32(a):
    return torch.from_numpy(np.ascontiguousarray(a).view(np.int32)).to(dev)


@pytest.mark.parametrize("n_sets", [1, 40, 6000])
@pytest.mark.parametrize("n_hashes", [32, 96, 256])
def test_minhash_paths(B, ctx, n_sets, n_hashes):
    rng = np.random.default_rng(n_sets + n_hashes)
    sizes = rng.integers(1, 12, n_sets)
    edges = [0, 4, 31, 32, 33, 255, 256, 257, 512, 513, 2048, 2049, 6001]
    sizes[: len(edges)] = edges[:n_sets]
    if n_sets == 1:
        sizes[0] = 2049
    indptr = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    indices = rng.integers(0, (1 << 31) - 1, indptr[-1]).astype(np.uint32)
    if n_sets > 9:   # the residues' ends: 0, p - 1, p, 2p, 2p + 1
        indices[indptr[3]:indptr[3] + 5] = [0, 2**31 - 2, 2**31 - 1, 2**32 - 2, 2**32 - 1]
    a, b = synth.minhash_coeffs(n_hashes, seed=3)
    a[:2], b[:2] = [1, 2**31 - 2], [0, 2**31 - 2]
    csr = synth.CSR(indptr, indices, None, 1 << 32)
    want = O.minhash(csr, a, b)
    sig = torch.zeros((n_sets, n_hashes), dtype=torch.int32, device=dev)
    B.blsh_minhash(ctx, torch.from_numpy(indptr).to(dev), t32(indices), n_hashes, t32(a), t32(b), sig)
    assert B.blsh_status(ctx) == 0
    assert np.array_equal(sig.cpu().numpy().view(np.uint32), want)


def lists(n, kinds, length, seed):
    """n sets on the GPU, set i a copy of row i % kinds of `length` elements:
    indptr, indices, and the distinct rows as a CSR."""
    rows = np.random.default_rng(seed).integers(0, (1 << 31) - 1, (kinds, length)).astype(np.uint32)
    indptr = torch.arange(n + 1, dtype=torch.int64, device=dev) * length
    indices = t32(rows)[torch.arange(n, device=dev) % kinds].reshape(-1)
    return indptr, indices, synth.CSR(np.arange(kinds + 1, dtype=np.int64) * length, rows.ravel(), None, 1 << 31)


@pytest.mark.parametrize("n,length", [((1 << 20) + 333, 2049), ((1 << 23) + 333, 257)])
def test_more_long_sets_than_their_list_holds(B, ctx, n, length):
    """Sets past the list of hubs (2^20) and past that of other long sets
    (2^23), which their own warps hash."""
    n_hashes, kinds = 64, 37
    indptr, indices, csr = lists(n, kinds, length, length)
    a, b = synth.minhash_coeffs(n_hashes, seed=4)
    sig = torch.zeros((n, n_hashes), dtype=torch.int32, device=dev)
    B.blsh_minhash(ctx, indptr, indices, n_hashes, t32(a), t32(b), sig)
    assert B.blsh_status(ctx) == 0
    want = t32(O.minhash(csr, a, b))
    for first in range(0, n, 1 << 20):
        at = torch.arange(first, min(n, first + (1 << 20)), device=dev)
        assert torch.equal(sig[at], want[at % kinds])


@pytest.mark.parametrize("lens", [[3, 257, 40], [5, 2049]])
def test_more_tiles_than_a_grid_has_rows(B, ctx, lens):
    n_hashes = 32 * 65537   # an odd number of words: tiles of 32 hashes, past the 65,535 of a grid's second axis
    rng = np.random.default_rng(1)
    indptr = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    indices = rng.integers(0, (1 << 31) - 1, indptr[-1]).astype(np.uint32)
    a, b = synth.minhash_coeffs(n_hashes, seed=5)
    sig = torch.zeros((len(lens), n_hashes), dtype=torch.int32, device=dev)
    B.blsh_minhash(ctx, torch.from_numpy(indptr).to(dev), t32(indices), n_hashes, t32(a), t32(b), sig)
    assert B.blsh_status(ctx) == 0
    want = O.minhash(synth.CSR(indptr, indices, None, 1 << 31), a, b)
    assert np.array_equal(sig.cpu().numpy().view(np.uint32), want)


def test_a_late_hub_is_not_one_warps_work(B, ctx):
    """A hub of 2e6 elements after 600,000 sets of 300: a warp alone takes 92 ms
    for it, the whole GPU 10 ms for all sets."""
    n, hub = 600_000, 2_000_000
    indptr, indices, _ = lists(n, 50, 300, 6)
    g = torch.Generator(device=dev).manual_seed(7)
    indices = torch.cat([indices, torch.randint(0, (1 << 31) - 1, (hub,), generator=g, device=dev, dtype=torch.int32)])
    indptr = torch.cat([indptr, indptr[-1:] + hub])
    a, b = synth.minhash_coeffs(256, seed=6)
    ta, tb = t32(a), t32(b)
    sig = torch.zeros((n + 1, 256), dtype=torch.int32, device=dev)
    times = []
    for _ in range(3):
        t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        t0.record()
        B.blsh_minhash(ctx, indptr, indices, 256, ta, tb, sig)
        t1.record()
        t1.synchronize()
        times.append(t0.elapsed_time(t1))
    assert B.blsh_status(ctx) == 0
    want = O.minhash(synth.CSR(np.array([0, hub], np.int64), indices[-hub:].cpu().numpy().view(np.uint32), None, 1 << 31), a, b)
    assert np.array_equal(sig[-1].cpu().numpy().view(np.uint32), want[0])
    assert min(times) < 40.0, times
