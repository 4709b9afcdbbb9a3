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
