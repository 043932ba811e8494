"""Drafting with several CTAs per row: every cluster size the launch chooses, at
row lengths whose tiles do not divide evenly, against the float64 draw."""

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,N,V", [(1, 3, 131072), (1, 60, 70001), (2, 60, 40004), (4, 60, 20000),
                                   (3, 3, 8191), (1, 1, 300001), (40, 31, 33000)])
def test_against_float64(B, N, V):
    import paper_2505_12398_gb300 as tv
    g = torch.Generator(device="cuda").manual_seed(V)
    parents = [-1] + [(c - 1) // 3 for c in range(1, N + 1)]
    drafts = torch.softmax(3.0 * torch.randn(B, N + 1, V, generator=g, device="cuda"), dim=-1)
    drafts[:, :, 100:400] = 0.0                # whole tiles without mass
    u = torch.rand(B, N + 1, generator=g, device="cuda")
    u[:, 1] = 0.0
    u[:, 2:3] = 0.99999994
    par = torch.tensor(parents, dtype=torch.int32, device="cuda").expand(B, N + 1).contiguous()
    v = tv.Verifier(V, N, B, "bf16", path="three")
    tok = v.draft_children(par, drafts, u)
    torch.cuda.synchronize()
    assert v.status() == 0
    v.close()
    at = torch.arange(B, device="cuda")
    for i in range(N + 1):
        q = drafts[:, i].double()
        for c in [c for c in range(1, N + 1) if parents[c] == i]:
            cdf = torch.cumsum(q, dim=-1)
            W = cdf[:, -1]
            t = u[:, c].double() * W
            y = tok[:, c].long()
            assert (q[at, y] > 0).all()
            lo = cdf[at, y] - q[at, y]
            # within 1e-6 W of u W: float32 sums of 256-token tiles
            assert (lo - 1e-6 * W <= t).all() and (t < cdf[at, y] + 1e-6 * W).all()
            q[at, y] = 0.0
