"""GPU parity of Lite's exact similarities in each form they are computed in:
batches dealt over the warp (with the rows' norms formed), survivors one by
one, rows around the lengths where the forms change (a stage of 127 and of
1,024 elements, several stages), index arrays that do not start on 16 bytes,
and sums past the carry of their limbs.  Bit-exact against the CPU oracle."""
import numpy as np
import pytest
import torch

import oracle as O
import synth

pytestmark = pytest.mark.gpu
dev = torch.device("cuda")


def csr_of(lens, dim, seed, values):
    rng = np.random.default_rng(seed)
    rows = [np.sort(rng.choice(dim, n, replace=False)).astype(np.uint32) for n in lens]
    vals = None
    if values:
        v = [rng.standard_normal(n) * rng.choice([1e-6, 1.0], n) for n in lens]
        vals = np.concatenate([x / max(np.linalg.norm(x), 1e-30) for x in v]).astype(np.float32)
    return synth.CSR(np.concatenate([[0], np.cumsum(lens)]).astype(np.int64), np.concatenate(rows), vals, dim)


def lite(B, ctx, csr, pairs, kind, shift=0, reserve=False):
    """Every pair survives (identical signatures); shift: words the index array
    starts past a 16-byte boundary."""
    N, P = csr.n, len(pairs)
    W = 64 if kind == 0 else 8
    if reserve:
        ctx = B.Context(0)
        B.blsh_ctx_reserve(ctx, N)
    ix = torch.zeros(csr.indices.size + 4, dtype=torch.int32, device=dev)
    ix[shift:shift + csr.indices.size] = torch.from_numpy(csr.indices.view(np.int32)).to(dev)
    val = None if kind == 0 else torch.from_numpy(csr.values).to(dev)
    tab = B.blsh_tables_build(ctx, B.make_params(kind=kind, t=0.3, n_max=64 if kind == 0 else 256, h=64))
    st = torch.zeros(P, dtype=torch.uint8, device=dev)
    sim = torch.full((P,), float("nan"), dtype=torch.float64, device=dev)
    B.blsh_verify_lite(ctx, tab, torch.from_numpy(pairs.view(np.int32)).to(dev),
                       torch.zeros((N, W), dtype=torch.int32, device=dev), torch.from_numpy(csr.indptr).to(dev),
                       ix[shift:shift + csr.indices.size], val, st, sim)
    assert B.blsh_status(ctx) == 0
    want = O.verify_lite(O.tables(O.Params(kind=kind, t=0.3, n_max=64 if kind == 0 else 256, h=64)), pairs,
                         np.zeros((N, W), np.uint32), csr)
    assert np.array_equal(st.cpu().numpy(), want.status)
    assert np.array_equal(sim.cpu().numpy(), want.sim)


LENS = [0, 1, 2, 7, 8, 9, 16, 17, 31, 32, 33, 100, 126, 127, 128, 129, 300, 1023, 1024, 1025, 2050, 5000]


@pytest.mark.parametrize("kind", [0, 1])
@pytest.mark.parametrize("shift", [0, 1, 3])
@pytest.mark.parametrize("many", [False, True])
def test_forms(B, ctx, kind, shift, many):
    csr = csr_of(LENS, 6000, 3, kind == 1)
    x, y = np.triu_indices(csr.n, 1)
    pairs = np.stack([x, y], 1).astype(np.uint32)
    if many:   # over 8 survivors for every warp of the GPU, in batches of 32
        pairs = np.tile(pairs, (-(-200_000 // len(pairs)), 1))
    else:      # one survivor a warp
        pairs = pairs[::3]
    lite(B, ctx, csr, pairs, kind, shift, reserve=many)


def test_sums_past_the_limbs(B, ctx):
    """Near-identical long rows of equal signs: hundreds of hits per survivor,
    terms near the top of their limbs."""
    n = 3000
    rng = np.random.default_rng(5)
    base = np.sort(rng.choice(8000, n, replace=False)).astype(np.uint32)
    rows, vals = [], []
    for i in range(40):
        keep = np.sort(rng.choice(n, n - 10 * i, replace=False))
        v = np.full(len(keep), 1.0 / np.sqrt(len(keep))) * (1 - 2e-8 * rng.random(len(keep)))
        rows.append(base[keep])
        vals.append((v * (1 if i % 2 else -1)).astype(np.float32))
    lens = [len(r) for r in rows]
    csr = synth.CSR(np.concatenate([[0], np.cumsum(lens)]).astype(np.int64), np.concatenate(rows),
                    np.concatenate(vals), 8000)
    x, y = np.triu_indices(40, 1)
    pairs = np.tile(np.stack([x, y], 1).astype(np.uint32), (200, 1))
    lite(B, ctx, csr, pairs, 1, 2, reserve=True)


@pytest.mark.parametrize("kind", [0, 1])
def test_rows_of_a_small_tile_one_by_one(B, ctx, kind):
    """Survivors formed singly whose longer row is one tile of fewer than 128
    elements and whose shorter one has up to 64, and just past both."""
    csr = csr_of([1, 31, 33, 63, 64, 65, 96, 126, 127, 128, 129, 64, 65, 40], 200, 8, kind == 1)
    x, y = np.triu_indices(csr.n, 1)
    pairs = np.stack([x, y], 1).astype(np.uint32)
    lite(B, ctx, csr, pairs, kind, 1)
    lite(B, ctx, csr, np.tile(pairs, (400, 1)), kind)   # batches of them, no norms formed
