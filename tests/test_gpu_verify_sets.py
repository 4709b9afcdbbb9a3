"""Jaccard verification with a lane per pair for the tests (the plain form's
eight lanes a pair, the default from 2^18 pairs) against the general path of
four lanes a pair: every output of both algorithms, with and without a hash
limit, for every chunk size, around a warp's 32 pairs and over many rounds of
a warp, with bad pairs and a device pair count."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
dev = torch.device("cuda")


@pytest.mark.parametrize("k", [32, 64, 128])
@pytest.mark.parametrize("P", [1, 31, 33, 70_001, 400_003])
@pytest.mark.parametrize("limit", [0, 256])
def test_sets_plan_matches_general(B, ctx, k, P, limit):
    rng = np.random.default_rng(P + k)
    N, n_max = 3000, 512
    # rows of 40 groups: a pair within a group agrees in about 30 to 95% of the hashes
    sig = rng.integers(0, 2**32, (40, n_max), dtype=np.uint32)[rng.integers(0, 40, N)]
    noise = rng.random((N, n_max)) < rng.uniform(0.02, 0.5, (N, 1))
    sig = np.where(noise, rng.integers(0, 2**32, (N, n_max), dtype=np.uint32), sig)
    pairs = rng.integers(0, N, (P, 2)).astype(np.uint32)
    close = rng.random(P) < 0.5
    pairs[close, 1] = np.minimum(pairs[close, 0] + 1, N - 1)
    if P > 40:
        pairs[[3, 40], [0, 1]] = [N, 2**32 - 1]
    t32 = lambda x: torch.from_numpy(np.ascontiguousarray(x).view(np.int32)).to(dev)
    pt, st32 = t32(np.concatenate([pairs, np.zeros((9, 2), np.uint32)])), t32(sig)
    count = torch.tensor([P], dtype=torch.int64, device=dev)
    ip = torch.arange(N + 1, dtype=torch.int64, device=dev)
    ix = torch.arange(N, dtype=torch.int32, device=dev)
    tab = B.blsh_tables_build(ctx, B.make_params(kind=0, t=0.6, k=k, n_max=n_max, h=256))

    def run(plan):
        if plan is not None:
            B.blsh_set_plan(ctx, tab, plan)
        z = lambda t, v=0: torch.full((P + 9,), v, dtype=t, device=dev)
        o = dict(status=z(torch.uint8, 77), n_used=z(torch.int16), m=z(torch.int16), est=z(torch.float32, -1.0),
                 hist=torch.zeros(tab.levels, dtype=torch.int64, device=dev), lstatus=z(torch.uint8, 77),
                 lnu=z(torch.int16), sim=z(torch.float64, -1.0), need=torch.zeros(N, dtype=torch.uint8, device=dev))
        head = (ctx, tab) if not limit else (ctx, tab, limit)
        call = B.blsh_verify_both_capped if limit else B.blsh_verify_both
        tail = (o["need"],) if limit else ()
        call(*head, pt, st32, o["status"], o["n_used"], o["m"], o["est"], o["hist"], ip, ix, None, o["lstatus"],
             o["sim"], *tail, lite_n_used=o["lnu"], P_dev=count)
        assert B.blsh_status(ctx) == (B.ERANGE if P > 40 else 0)
        return {name: v.cpu().numpy() for name, v in o.items()}

    first = run(None)   # the plan of the size
    want = run(B.blsh_plan(B.PLAN_PLAIN, 4, 128, 32, 0))
    for got in (first, run(B.blsh_plan(B.PLAN_PLAIN, 8, 128, 32, 0)), run(B.blsh_plan(B.PLAN_PLAIN, 8, 512, 32, 0))):
        for name in want:
            assert np.array_equal(got[name], want[name]), name
    if P > 1000:
        assert len(np.unique(want["n_used"][:P])) > 2 and (want["need"].any() or not limit)
