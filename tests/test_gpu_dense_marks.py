"""GPU parity of the tensor-core projection's rechecks where many signs are
marked: exact ties (whole-number data), zero rows and columns, rows outside
the range of the norms, infinities and NaN, more marks in a row than are
listed at a time, and items of one, two and four rows.  Bit-exact against the
CPU oracle, with every exact zero counted."""
import numpy as np
import pytest
import torch

import oracle as O

pytestmark = pytest.mark.gpu
dev = torch.device("cuda")


@pytest.mark.parametrize("n, d, bits", [(1, 8, 256), (67, 64, 1024), (301, 256, 2048), (130, 130, 768), (77, 257, 512),
                                        (50, 600, 1024)])
@pytest.mark.parametrize("offset", [0, 1])
def test_marked_signs(B, ctx, n, d, bits, offset):
    rng = np.random.default_rng(n + d)
    X = rng.integers(-2, 3, (n, d)).astype(np.float32)
    R = rng.integers(-1, 2, (d, bits)).astype(np.float32)
    R[:, 5] = 0.0
    X[n // 2] = 0.0
    zeros = int((X.astype(np.float64) @ R.astype(np.float64) == 0).sum())
    if n > 20:   # rows whose sums are never zero, or not finite
        special = {3: rng.standard_normal(d) * 1e-22, 4: rng.standard_normal(d) * 1e25, 6: rng.standard_normal(d) * 1e-41}
        for r, v in special.items():
            zeros -= int((X[r].astype(np.float64) @ R == 0).sum())
            X[r] = v.astype(np.float32)
            zeros += int((X[r].astype(np.float64) @ R.astype(np.float64) == 0).sum())
        for r, v in ((8, np.nan), (9, np.inf), (10, -np.inf)):
            zeros -= int((X[r].astype(np.float64) @ R == 0).sum())
            X[r] = 1.0
            X[r, 0] = v
            with np.errstate(invalid="ignore"):
                s = np.where(R[0] == 0, np.nan, v * R[0])
            zeros += int((s == 0).sum())
    want = O.srp_dense(X, R)
    store = torch.zeros(n * (bits // 32) + offset, dtype=torch.int32, device=dev)
    sig = store[offset:].view(n, bits // 32)
    ws = torch.full((B.blsh_srp_dense_workspace(n, d, bits),), 0xCD, dtype=torch.uint8, device=dev)
    B.blsh_srp_dense(ctx, torch.from_numpy(X).to(dev), torch.from_numpy(R).to(dev), sig, workspace=ws)
    rc, c = B.blsh_status(ctx, counters=True)
    assert rc == 0
    assert np.array_equal(sig.cpu().numpy().view(np.uint32), want)
    assert c[3] == zeros and c[2] >= zeros
