"""GPU parity of the dense sign projections at the shapes where their tiles
end: widths that are no multiple of a K stage, row and bit counts at the edges
of a tile, on the tensor cores (with a workspace) and on the CUDA cores
(without), and rows whose norms lie outside the range the tensor cores
decide.  Bit-exact against the CPU oracle."""
import numpy as np
import pytest
import torch

import oracle as O
import synth

pytestmark = pytest.mark.gpu
dev = torch.device("cuda")


def project(B, ctx, X, R, margin=0.0, workspace=True):
    n, d = X.shape
    bits = R.shape[1]
    sig = torch.full((n, bits // 32), -1, dtype=torch.int32, device=dev)
    ws = None
    if workspace:
        nws = B.blsh_srp_dense_workspace(n, d, bits)
        assert nws > 0
        ws = torch.full((nws,), 0xCD, dtype=torch.uint8, device=dev)
    B.blsh_srp_dense(ctx, torch.from_numpy(X).to(dev), torch.from_numpy(R).to(dev), sig, margin=margin, workspace=ws)
    rc, c = B.blsh_status(ctx, counters=True)
    assert rc == 0
    return sig.cpu().numpy().view(np.uint32), c


@pytest.mark.parametrize("n,d,bits", [(1, 1, 256), (127, 63, 256), (128, 65, 512), (129, 100, 256), (300, 300, 1024),
                                      (257, 301, 256), (64, 1030, 256)])
@pytest.mark.parametrize("margin", [0.0, 1e-2])
def test_ragged_width_on_tensor_cores(B, ctx, n, d, bits, margin):
    X = synth.gaussian_mixture(n_points=n, dim=d, n_centers=20, seed=d)
    if n > 5:
        X[5] = 0.0
    R = synth.gaussian_matrix(d, bits, seed=5)
    want = O.srp_dense(X, R)
    got, _ = project(B, ctx, X, R, margin)
    assert np.array_equal(got, want)
    # too small a workspace for such a width: the CUDA cores, as before
    if d % 64:
        sig = torch.zeros((n, bits // 32), dtype=torch.int32, device=dev)
        B.blsh_srp_dense(ctx, torch.from_numpy(X).to(dev), torch.from_numpy(R).to(dev), sig, margin=margin,
                         workspace=torch.zeros(256, dtype=torch.uint8, device=dev))
        assert B.blsh_status(ctx) == 0
        assert np.array_equal(sig.cpu().numpy().view(np.uint32), want)


@pytest.mark.parametrize("n,d,bits", [(1, 1, 32), (31, 31, 96), (33, 32, 128), (63, 33, 160), (65, 100, 288),
                                      (20000, 65, 128), (20011, 30, 320)])
def test_cuda_core_tiles(B, ctx, n, d, bits):
    X = synth.gaussian_mixture(n_points=n, dim=d, n_centers=20, seed=d + 1)
    X[n // 2] = 0.0
    R = synth.gaussian_matrix(d, bits, seed=6)
    got, c = project(B, ctx, X, R, workspace=False)
    assert np.array_equal(got, O.srp_dense(X, R))
    assert c[3] >= bits


@pytest.mark.parametrize("workspace", [True, False])
@pytest.mark.parametrize("d", [100, 128])
def test_rows_outside_the_decided_range(B, ctx, d, workspace):
    """Norms near the ends of the FP32 range (sums and splits that would
    overflow or underflow), infinities and NaN."""
    X = synth.gaussian_mixture(n_points=160, dim=d, n_centers=20, seed=3)
    R = synth.gaussian_matrix(d, 256, seed=7)
    X[3] *= np.float32(1e30)
    X[4] *= np.float32(1e-30)
    X[5] *= np.float32(1e-38)
    X[6, 7] = np.inf
    X[7, 1] = -np.inf
    X[8, 2] = np.nan
    X[9, :2] = [3e38, -3e38]
    R[:, 17] *= np.float32(1e28)
    R[:, 18] *= np.float32(1e-33)
    R[0, 40] = np.inf
    with np.errstate(invalid="ignore"):
        want = O.srp_dense(X, R)
    got, _ = project(B, ctx, X, R, workspace=workspace)
    assert np.array_equal(got, want)
