"""Vocabularies that are not a multiple of 8 (the path with separate normalisers): rows that
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
    code, C, ncw, stages = v.launch_shape(B, R - 1)
    assert code == 0 and stages >= 2
    if shape:
        want = [int(x) for x in shape.split(",")]
        assert [ncw, C] == want[:2] and want[2] in (0, stages)
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


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("B,V", [(2, 40001), (3, 20001), (20, 4003), (200, 1003)])
def test_rows_without_a_normaliser(B, V, dtype):
    """Every thread count of the normaliser kernel: a row of -inf or with +inf makes
    its tree invalid; single tokens far below or alone in their row do not, and
    other trees are what they were."""
    import paper_2505_12398_gb300 as tv
    w = Workload("nonfinite", B, V, levels=(2, 3), branching=(2, 2), logit_dtype=dtype, sigma=1.0)
    inp = make_inputs(w, seed=V, device="cuda")
    R = inp.parents.shape[1]
    v = tv.Verifier(V, R - 1, B, "bf16" if dtype == torch.bfloat16 else "fp32")

    def run(logits):
        out = v.verify(inp.parents, inp.tokens, logits, inp.draft_probs, inp.temperature,
                       inp.uniforms, debug=True)
        torch.cuda.synchronize()
        return [x.clone() for x in out], v.status() & ~16
    clean, status = run(inp.logits)
    assert status == 0
    for bad in (float("-inf"), float("inf")):
        lg = inp.logits.clone()
        if bad < 0:
            lg[1, 0] = bad
        else:
            lg[1, 0, V - 1] = bad
        out, status = run(lg)
        assert status == 64
        assert int(out[1][1]) == -1 and int(out[2][1]) == -1
        keep = [b for b in range(B) if b != 1]
        for x, y in zip(out[:3], clean[:3]):
            assert torch.equal(x[keep], y[keep])
    lg = inp.logits.clone()
    lg[1, 0, :] = float("-inf")
    lg[1, 0, inp.tokens[1, 1].long()] = -30000.0   # the row's only token: M_b = 1
    out, status = run(lg)
    v.close()
    assert status == 0
    first = int((inp.parents[1] == 0).nonzero()[0])
    assert int(inp.tokens[1, 1]) == int(inp.tokens[1, first])
    inp.logits = lg
    par, tok, lgn, dp, un = to_numpy_inputs(inp, trees=[1])
    _, _, _, det = verify_batch(par, tok, lgn, dp, inp.temperature, un, keep_cdf=True)
    summ = compare_batch(det, *[x[1:2].cpu().numpy() for x in out])
    assert not summ["bad"], summ["bad"]
