"""Lite's exact similarities of survivors whose two rows are long, which a CTA
forms by eighths of the shorter row, around the length where that begins, with
parts of the longer row left empty, equal indices at a part's edge, with and
without formed norms, among short survivors and alone.  Bit-exact against the
CPU oracle, the repeated index against the sums themselves."""
import numpy as np
import pytest
import torch

import oracle as O
import synth

pytestmark = pytest.mark.gpu
dev = torch.device("cuda")


def run(B, csr, pairs, kind, reserve):
    N, P, W = csr.n, len(pairs), 64 if kind == 0 else 8
    ctx = B.Context(0)
    if reserve:
        B.blsh_ctx_reserve(ctx, N)
    tab = B.blsh_tables_build(ctx, B.make_params(kind=kind, t=0.3, n_max=64 if kind == 0 else 256, h=64))
    st = torch.zeros(P, dtype=torch.uint8, device=dev)
    sim = torch.full((P,), float("nan"), dtype=torch.float64, device=dev)
    B.blsh_verify_lite(ctx, tab, torch.from_numpy(pairs.view(np.int32)).to(dev),
                       torch.zeros((N, W), dtype=torch.int32, device=dev), torch.from_numpy(csr.indptr).to(dev),
                       torch.from_numpy(csr.indices.view(np.int32)).to(dev),
                       None if kind == 0 else torch.from_numpy(csr.values).to(dev), st, sim)
    assert B.blsh_status(ctx) == 0
    return st.cpu().numpy(), sim.cpu().numpy()


@pytest.mark.parametrize("kind", [0, 1])
@pytest.mark.parametrize("reserve", [False, True])
@pytest.mark.parametrize("short", [0, 3000])
def test_long_rows(B, kind, reserve, short):
    rng = np.random.default_rng(kind + short)
    dim = 30_000
    lens = [511, 512, 513, 514, 700, 1025, 4097, 9000, 25_000]
    rows = [np.sort(rng.choice(dim, n, replace=False)) for n in lens]
    rows += [np.arange(600), np.arange(dim - 900, dim), np.arange(0, dim, 40)]   # one below, one above, one between
    nl = len(rows)
    rows += [np.sort(rng.choice(dim, n, replace=False)) for n in rng.integers(0, 40, 60 if short else 1)]
    ln = [len(r) for r in rows]
    vals = np.concatenate([rng.standard_normal(n) / max(np.sqrt(n), 1) for n in ln]).astype(np.float32)
    csr = synth.CSR(np.concatenate([[0], np.cumsum(ln)]).astype(np.int64), np.concatenate(rows).astype(np.uint32),
                    vals if kind else None, dim)
    x, y = np.triu_indices(nl)
    pairs = np.concatenate([np.stack([x, y], 1), np.stack([y, x], 1), rng.integers(0, csr.n, (short, 2))]).astype(np.uint32)
    pairs = pairs[rng.permutation(len(pairs))]
    W = 64 if kind == 0 else 8
    want = O.verify_lite(O.tables(O.Params(kind=kind, t=0.3, n_max=64 if kind == 0 else 256, h=64)), pairs,
                         np.zeros((csr.n, W), np.uint32), csr)
    st, sim = run(B, csr, pairs, kind, reserve)
    assert np.array_equal(st, want.status) and np.array_equal(sim, want.sim)


def test_repeated_indices_stay_together(B):
    """A row in which one index stands 200 times, across the edges of eighths:
    every occurrence meets the other row's entry."""
    a = np.sort(np.concatenate([np.arange(0, 1600, 4), np.full(200, 801)]))
    b = np.arange(1, 2001, 2)
    csr = synth.CSR(np.array([0, len(a), len(a) + len(b)], np.int64), np.concatenate([a, b]).astype(np.uint32),
                    np.full(len(a) + len(b), 0.03125, np.float32), 3000)
    pairs = np.array([[0, 1], [1, 0]], np.uint32)
    st, sim = run(B, csr, pairs, 1, False)
    term = 2.0**50   # 0.03125 squared, times 2^60
    want = (200 * term) / np.sqrt((len(a) * term) * (len(b) * term))
    assert np.array_equal(sim, [want, want])


@pytest.mark.parametrize("kind", [0, 1])
@pytest.mark.parametrize("long_share", [0.01, 0.3])
def test_past_the_queue_and_the_list(B, kind, long_share):
    """More survivors than the queue holds (2^23), and fewer or more pairs of
    long rows among the queued ones than their list holds (2^20)."""
    rng = np.random.default_rng(11 + kind)
    dim = 2000
    ln = np.concatenate([rng.integers(513, 560, 24), rng.integers(3, 30, 400)])
    rows = [np.sort(rng.choice(dim, n, replace=False)) for n in ln]
    vals = np.concatenate([rng.standard_normal(n) / np.sqrt(n) for n in ln]).astype(np.float32)
    csr = synth.CSR(np.concatenate([[0], np.cumsum(ln)]).astype(np.int64), np.concatenate(rows).astype(np.uint32),
                    vals if kind else None, dim)
    some = 4001
    heavy = rng.random(some) < long_share
    few = np.where(heavy[:, None], rng.integers(0, 24, (some, 2)), rng.integers(24, csr.n, (some, 2))).astype(np.uint32)
    reps = (1 << 23) // some + 40
    assert ((1 << 23) * long_share > 1.2 * (1 << 20)) == (long_share > 0.2)
    W = 64 if kind == 0 else 8
    want = O.verify_lite(O.tables(O.Params(kind=kind, t=0.3, n_max=64 if kind == 0 else 256, h=64)), few,
                         np.zeros((csr.n, W), np.uint32), csr)
    st, sim = run(B, csr, np.tile(few, (reps, 1)), kind, True)
    assert np.array_equal(st.reshape(reps, some), np.broadcast_to(want.status, (reps, some)))
    assert np.array_equal(sim.reshape(reps, some), np.broadcast_to(want.sim, (reps, some)))
