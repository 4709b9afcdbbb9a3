"""GPU parity of the sparse projection on both sides of its rules: rows around
the lengths at which a block of 32 and the long rows' kernel begin, few rows
(handed out singly, piece by piece) and many (several a grab, all pieces of a
row together), four and eight columns a lane, and malformed indices, which
contribute nothing and are reported.  Bit-exact against the CPU oracle."""
import numpy as np
import pytest
import torch

import oracle as O
import synth

pytestmark = pytest.mark.gpu
dev = torch.device("cuda")
EDGES = [0, 1, 7, 8, 9, 31, 32, 33, 64, 65, 255, 256, 257, 287, 511, 512, 513, 2049, 9000]


def rows(n, dim, seed):
    rng = np.random.default_rng(seed)
    lens = rng.integers(0, 6, n)
    lens[rng.choice(n, len(EDGES), replace=False)] = EDGES
    indptr = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    ix = rng.integers(0, dim, indptr[-1]).astype(np.uint32)
    return synth.CSR(indptr, ix, rng.standard_normal(indptr[-1]).astype(np.float32), dim)


@pytest.mark.parametrize("n", [60, 40_000, 90_000])
@pytest.mark.parametrize("form, bits", [("float", 256), ("codes", 384), ("codes", 512), ("codes on 8 bytes", 512)])
def test_srp_rows(B, ctx, n, form, bits):
    dim = 3000
    csr = rows(n, dim, n + bits)
    bad = csr.indices.copy()
    drop = np.zeros(len(bad), bool)
    drop[::97] = True
    drop[int(csr.indptr[np.argmax(np.diff(csr.indptr))]) + 300] = True   # past a long row's first round of blocks
    bad[drop] = np.where(np.arange(drop.sum()) % 2, dim, 2**32 - 1).astype(np.uint32)
    kept = np.concatenate([[0], np.cumsum(~drop)])[csr.indptr].astype(np.int64)
    clean = synth.CSR(kept, csr.indices[~drop], csr.values[~drop], dim)
    ip, val = torch.from_numpy(csr.indptr).to(dev), torch.from_numpy(csr.values).to(dev)
    sig = torch.zeros((n, bits // 32), dtype=torch.int32, device=dev)
    if form == "float":
        R = synth.gaussian_matrix(dim, bits, seed=5)
        Rd, oracle, call = torch.from_numpy(R).to(dev), O.srp_sparse, B.blsh_srp_sparse
    else:
        R = O.gaussian_codes(5, dim, bits)
        off = 4 if form.endswith("8 bytes") else 0
        store = torch.zeros(R.size + off, dtype=torch.int16, device=dev)
        Rd = store[off:].view(dim, bits)
        Rd.copy_(torch.from_numpy(R.view(np.int16)))
        oracle, call = O.srp_sparse_q16, B.blsh_srp_sparse_q16
    for indices, want, rc in ((csr.indices, oracle(csr, R), 0), (bad, oracle(clean, R), B.ERANGE)):
        call(ctx, ip, torch.from_numpy(indices.view(np.int32)).to(dev), val, Rd, sig)
        assert B.blsh_status(ctx) == rc
        assert np.array_equal(sig.cpu().numpy().view(np.uint32), want)


@pytest.mark.parametrize("form", ["float", "codes"])
def test_rechecked_long_rows(B, ctx, form):
    """Rows whose every sum is zero, or cancels to its last entry, at the
    lengths where a recheck takes more entries at a time."""
    dim, bits = 4000, 256
    half = dim // 2
    if form == "float":
        R = synth.gaussian_matrix(dim, bits, seed=9)
        R[half:] = -R[:half]
        Rd, oracle, call = torch.from_numpy(R).to(dev), O.srp_sparse, B.blsh_srp_sparse
    else:
        R = np.maximum(O.gaussian_codes(9, dim, bits), 1)
        R[half:] = (65536 - R[:half].astype(np.int64)).astype(np.uint16)   # decoded: the negatives
        Rd, oracle, call = torch.from_numpy(R.view(np.int16)).to(dev), O.srp_sparse_q16, B.blsh_srp_sparse_q16
    rng = np.random.default_rng(4)
    rows, vals = [], []
    for n in (1, 15, 63, 64, 65, 255, 256, 257, 512, 1000):   # pairs of entries that cancel
        f = np.sort(rng.choice(half, n, replace=False))
        v = rng.standard_normal(n).astype(np.float32)
        rows += [np.concatenate([f, f + half])] * 2
        vals += [np.concatenate([v, v]), np.concatenate([v, v[:-1], np.nextafter(v[-1:], np.float32(9))])]
    csr = synth.CSR(np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int64),
                    np.concatenate(rows).astype(np.uint32), np.concatenate(vals).astype(np.float32), dim)
    sig = torch.zeros((csr.n, bits // 32), dtype=torch.int32, device=dev)
    call(ctx, torch.from_numpy(csr.indptr).to(dev), torch.from_numpy(csr.indices.view(np.int32)).to(dev),
         torch.from_numpy(csr.values).to(dev), Rd, sig)
    rc, c = B.blsh_status(ctx, counters=True)
    assert rc == 0 and c[2] >= csr.n * bits // 2
    assert np.array_equal(sig.cpu().numpy().view(np.uint32), oracle(csr, R))


@pytest.mark.parametrize("n", [1, 700, 20_000, 160_000])
@pytest.mark.parametrize("share", [0.0, 0.03, 1.0])
@pytest.mark.parametrize("form", ["float", "codes"])
def test_masked_rows(B, ctx, n, share, form):
    """Some rows' columns 128 .. 383: a warp's first rows all it takes, and more
    rows than that; the others stay as they are."""
    dim, bits = 500, 512
    csr = rows(n, dim, n) if n > 100 else synth.CSR(np.array([0, 40], np.int64), np.arange(40, dtype=np.uint32) * 3,
                                                    np.linspace(-1, 1, 40).astype(np.float32), dim)
    mask = np.random.default_rng(n).random(n) < share
    ip, val = torch.from_numpy(csr.indptr).to(dev), torch.from_numpy(csr.values).to(dev)
    ix = torch.from_numpy(csr.indices.view(np.int32)).to(dev)
    if form == "float":
        R = synth.gaussian_matrix(dim, bits, seed=5)
        want, Rd, call = O.srp_sparse(csr, R), torch.from_numpy(R).to(dev), B.blsh_srp_sparse_cols
    else:
        R = O.gaussian_codes(5, dim, bits)
        want, Rd, call = O.srp_sparse_q16(csr, R), torch.from_numpy(R.view(np.int16)).to(dev), B.blsh_srp_sparse_q16_cols
    for first, count in ((128, 256), (256, 128)):
        sig = torch.full((n, bits // 32), 0x5A5A5A5A, dtype=torch.int32, device=dev)
        call(ctx, ip, ix, val, Rd, sig, first, count, row_mask=torch.from_numpy(mask.astype(np.uint8)).to(dev))
        assert B.blsh_status(ctx) == 0
        got = sig.cpu().numpy().view(np.uint32)
        there = np.zeros_like(got, bool)
        there[mask, first // 32:(first + count) // 32] = True
        assert np.array_equal(got, np.where(there, want, 0x5A5A5A5A))


def test_an_empty_mask_costs_no_grabs(B, ctx):
    """100,000 rows, none of them left: one look at the mask (a grab of a few rows
    at a time takes 47 us for the counter alone)."""
    n, dim, bits = 100_000, 300, 256
    csr = rows(n, dim, 4)
    ip, val = torch.from_numpy(csr.indptr).to(dev), torch.from_numpy(csr.values).to(dev)
    ix = torch.from_numpy(csr.indices.view(np.int32)).to(dev)
    R = torch.from_numpy(synth.gaussian_matrix(dim, bits, seed=5)).to(dev)
    sig, mask = torch.zeros((n, bits // 32), dtype=torch.int32, device=dev), torch.zeros(n, dtype=torch.uint8, device=dev)
    times = []
    for _ in range(4):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(20):
            B.blsh_srp_sparse_cols(ctx, ip, ix, val, R, sig, 128, 128, row_mask=mask)
        b.record()
        b.synchronize()
        times.append(a.elapsed_time(b) / 20)
    assert min(times) < 0.03, times


@pytest.mark.parametrize("form", ["float", "codes"])
@pytest.mark.parametrize("mean", [20, 150, 400])
def test_long_rows_by_the_average(B, ctx, form, mean):
    """20,000 rows, enough for every warp: a CTA's rows begin at four times the
    average, at least 256 and at most 1,024."""
    n, dim = 20_000, 4000
    bits = 128 if form == "float" else 256
    rng = np.random.default_rng(mean)
    lens = np.full(n, mean)
    edge = [255, 256, 257, 4 * mean - 2, 4 * mean - 1, 4 * mean, 4 * mean + 1, 4 * mean + 2, 1023, 1024, 1025, 3000, 0, 1]
    lens[rng.choice(n, len(edge), replace=False)] = edge
    indptr = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    csr = synth.CSR(indptr, rng.integers(0, dim, indptr[-1]).astype(np.uint32),
                    rng.standard_normal(indptr[-1]).astype(np.float32), dim)
    ip, val = torch.from_numpy(csr.indptr).to(dev), torch.from_numpy(csr.values).to(dev)
    ix = torch.from_numpy(csr.indices.view(np.int32)).to(dev)
    sig = torch.zeros((n, bits // 32), dtype=torch.int32, device=dev)
    if form == "float":
        R = synth.gaussian_matrix(dim, bits, seed=6)
        B.blsh_srp_sparse(ctx, ip, ix, val, torch.from_numpy(R).to(dev), sig)
        want = O.srp_sparse(csr, R)
    else:
        R = O.gaussian_codes(6, dim, bits)
        B.blsh_srp_sparse_q16(ctx, ip, ix, val, torch.from_numpy(R.view(np.int16)).to(dev), sig)
        want = O.srp_sparse_q16(csr, R)
    assert B.blsh_status(ctx) == 0
    assert np.array_equal(sig.cpu().numpy().view(np.uint32), want)
