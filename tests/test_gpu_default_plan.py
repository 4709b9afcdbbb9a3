"""The launch form of cosine calls that have no tuned plan: packed stores where
every output takes them, and where one does not, the persistent form up to
2^22 pairs and the two passes of the plain form above.  The outputs are the
same."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
dev = torch.device("cuda")


@pytest.mark.parametrize("P", [40_000, 70_000, (1 << 22) - 1, (1 << 22) + 5])
@pytest.mark.parametrize("which", ["pairs", "status", "n_used", "m"])
def test_outputs_off_their_boundary(B, ctx, P, which):
    g = torch.Generator(device=dev).manual_seed(P)
    N, W = 3000, 16
    base = torch.randint(-2**31, 2**31, (40, W), generator=g, device=dev).to(torch.int32)
    sig = base[torch.randint(0, 40, (N,), generator=g, device=dev)].contiguous()
    sig ^= torch.where(torch.rand(N, W, generator=g, device=dev) < 0.5,
                       1 << torch.randint(0, 31, (N, W), generator=g, device=dev), 0).to(torch.int32)
    pairs = torch.randint(0, N, (P, 2), generator=g, device=dev).to(torch.int32)
    tab = B.blsh_tables_build(ctx, B.make_params(kind=1, t=0.7, k=32, n_max=512, h=128))
    got = []
    for off in (0, 1):
        at = {"pairs": 0, "status": 0, "n_used": 0, "m": 0, which: off}
        p = torch.zeros((P + 1, 2), dtype=torch.int32, device=dev)[at["pairs"]:at["pairs"] + P]
        p.copy_(pairs)
        out = {name: torch.zeros(P + 1, dtype=t, device=dev)[at[name]:at[name] + P]
               for name, t in (("status", torch.uint8), ("n_used", torch.int16), ("m", torch.int16))}
        est, hist = torch.full((P,), -1.0, device=dev), torch.zeros(tab.levels, dtype=torch.int64, device=dev)
        B.blsh_timing_begin(ctx)
        B.blsh_verify(ctx, tab, p, sig, out["status"], out["n_used"], out["m"], est, hist)
        names = [n for n, _ in B.blsh_timing_end(ctx)]
        assert B.blsh_status(ctx) == 0
        if P < 65_536 or (off and P < 1 << 22):
            assert names == ["verify_kernel"]
        else:
            assert names == (["verify_first_kernel", "verify_kernel"] if off else ["verify_tile_kernel"])
        got.append([out["status"], out["n_used"], out["m"], est, hist])
    assert all(torch.equal(a, b) for a, b in zip(*got))
    assert len(np.unique(got[0][0].cpu().numpy())) > 1 and len(np.unique(got[0][1].cpu().numpy())) > 2
