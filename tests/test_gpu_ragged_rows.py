"""Vocabularies that are not a multiple of 8 (the three-kernel path): rows that
start anywhere in a 16-byte block, slices split over clusters, the arrays' last
partial block, and high temperatures, where a masked element's weight would
not be negligible; against the oracle."""

import pytest
import torch

from oracle.verify import verify_batch
from tests.parity import assert_rate_budget, compare_batch, to_numpy_inputs
from workloads.synth import Workload, make_inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", ["", "8,8,0", "16,16,0", "4,1,2"])
@pytest.mark.parametrize("V,dtype,T", [(7, torch.float32, 1.0), (1001, torch.bfloat16, 300.0),
                                       (4099, torch.float32, 0.7), (20003, torch.bfloat16, 0.7),
                                       (32005, torch.bfloat16, 1.0)])
def test_against_oracle(V, dtype, T, shape, monkeypatch):
    import paper_2505_12398_gb300 as tv
    monkeypatch.setenv("TV_FUSED_PLAN", shape)
    w = Workload("ragged_rows", 7, V, levels=(2, 4, 3), branching=(2, 2, 1), logit_dtype=dtype,
                 temperature=T, sigma=1.0)
    inp = make_inputs(w, seed=V, device="cuda")
    B, R = inp.parents.shape
    v = tv.Verifier(V, R - 1, B, "bf16" if dtype == torch.bfloat16 else "fp32")
    assert v.launch_shape(B, R - 1)[0] == 0
    out = v.verify(inp.parents, inp.tokens, inp.logits, inp.draft_probs, inp.temperature,
                   inp.uniforms, debug=True)
    torch.cuda.synchronize()
    assert v.status() & ~16 == 0
    v.close()
    path, tau, bonus, node_p, stats = [t.cpu().numpy() for t in out]
    par, tok, lg, dp, un = to_numpy_inputs(inp)
    _, _, _, det = verify_batch(par, tok, lg, dp, inp.temperature, un, keep_cdf=True)
    summ = compare_batch(det, path, tau, bonus, node_p, stats)
    assert not summ["bad"], summ["bad"][:5]
    assert_rate_budget(summ)
    internal = len({int(p) for p in par[0][1:]})
    assert (stats[:, 4] == internal).all()
