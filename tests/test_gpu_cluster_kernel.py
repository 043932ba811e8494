"""The cluster kernel at the sizes where its splits can go wrong, against the
oracle: every launch shape it can choose, chains longer than one normaliser job
takes, slices of a few tokens, resident and streamed row pairs, and given row
normalisers."""

import pytest
import torch

from oracle import lmhead
from oracle.verify import verify_batch
from tests.parity import assert_rate_budget, compare_batch, to_numpy_inputs
from workloads.synth import Workload, make_inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tv():
    import paper_2505_12398_gb300 as tv
    from paper_2505_12398_gb300.build import build
    build()
    return tv


def _check(inp, out):
    path, tau, bonus, node_p, stats = [t.cpu().numpy() for t in out]
    par, tok, lg, dp, un = to_numpy_inputs(inp)
    _, _, _, det = verify_batch(par, tok, lg, dp, inp.temperature, un, keep_cdf=True)
    summ = compare_batch(det, path, tau, bonus, node_p, stats)
    assert not summ["bad"], summ["bad"][:5]
    assert_rate_budget(summ)


def _verify(tv, inp, path):
    B, R = inp.parents.shape
    V = inp.logits.shape[-1]
    dt = "bf16" if inp.logits.dtype == torch.bfloat16 else "fp32"
    v = tv.Verifier(V, R - 1, B, dt, path=path)
    out = v.verify(inp.parents, inp.tokens, inp.logits, inp.draft_probs, inp.temperature,
                   inp.uniforms, debug=True)
    torch.cuda.synchronize()
    assert v.status() & ~16 == 0
    v.close()
    return out


@pytest.mark.parametrize("shape", ["16,16", "16,1", "8,16", "4,1", "16,2"])
@pytest.mark.parametrize("V,dtype", [(8, torch.bfloat16), (4104, torch.float32),
                                     (24584, torch.bfloat16)])
def test_launch_shapes(tv, shape, V, dtype, monkeypatch):
    """Slices of no, one and several 8-token blocks, pairs that stay in the ring
    and pairs that do not."""
    monkeypatch.setenv("TV_FUSED_PLAN", shape + ",0")
    w = Workload("shapes", 6, V, levels=(2, 3, 2), branching=(2, 2, 1), logit_dtype=dtype,
                 sigma=1.0)
    inp = make_inputs(w, seed=V, device="cuda")
    _check(inp, _verify(tv, inp, "cluster"))


@pytest.mark.parametrize("shape", ["8,16,0", "4,1,2", "16,4,0"])
def test_chains_longer_than_a_normaliser_job(tv, shape, monkeypatch):
    """Chains of 19 nodes: three normaliser jobs, rows in several waves of the
    ring."""
    monkeypatch.setenv("TV_FUSED_PLAN", shape)
    w = Workload("chain19", 5, 9000, levels=(1,) * 19, branching=(1,) * 19, sigma=0.5)
    inp = make_inputs(w, seed=19, device="cuda")
    _check(inp, _verify(tv, inp, "cluster"))


@pytest.mark.parametrize("V,B", [(128256, 3), (65536, 9), (32000, 40), (2000, 300)])
def test_given_normalisers(tv, V, B):
    """tv_verify_batch_stats on the cluster kernel (a handle that chooses its path
    itself): no row is normalised, results as the oracle's; a row without a
    finite normaliser makes its tree invalid."""
    w = Workload("given", B, V, levels=(3, 5, 4), branching=(3, 2, 1), sigma=1.0)
    inp = make_inputs(w, seed=B, device="cuda")
    lf = inp.logits.double()
    m = lf.max(dim=-1).values
    s = torch.exp2((lf - m[..., None]) * (lmhead.LOG2E / inp.temperature)).sum(dim=-1)
    row_stats = torch.stack([m, s], dim=-1).float().contiguous()
    del lf
    R = inp.parents.shape[1]
    v = tv.Verifier(V, R - 1, B, "bf16")
    assert v.launch_shape(B, R - 1)[0] == 1
    args = (inp.parents, inp.tokens, inp.logits, inp.draft_probs, inp.temperature, inp.uniforms)
    out = v.verify_stats(*args, row_stats, debug=True)
    torch.cuda.synchronize()
    assert v.status() & ~16 == 0
    assert (out[4][:, 4] == 0).all()
    _check(inp, out)
    row_stats[1, 0, 1] = 0.0
    bad = v.verify_stats(*args, row_stats, debug=True)
    torch.cuda.synchronize()
    assert v.status() & 64
    v.close()
    assert int(bad[1][1]) == -1 and int(bad[2][1]) == -1 and (bad[0][1] == -1).all()
    keep = [b for b in range(B) if b != 1]
    for x, y in zip(bad[:3], out[:3]):
        assert torch.equal(x[keep], y[keep])


@pytest.mark.parametrize("path", ["cluster", "persistent"])
@pytest.mark.parametrize("sigma", [0.05, 0.5, 3.0])
def test_runs_of_siblings(tv, path, sigma):
    """Passes that follow a sibling's rejection or removal at the same node, whose
    sums come in units of D / 2^e: leaves of one root, drafts close to the target (D
    near 0, wherever the rate is near 1) and far from it (rate 0, many removals)."""
    w = Workload("siblings", 24, 8008, levels=(12, 3), branching=(12, 3), sigma=sigma)
    inp = make_inputs(w, seed=int(100 * sigma), device="cuda")
    _check(inp, _verify(tv, inp, path))


@pytest.mark.parametrize("path", ["cluster", "persistent"])
@pytest.mark.parametrize("value", [float("inf"), float("-inf")])
def test_fp32_rows_without_a_normaliser(tv, path, value):
    """The packed exponentials of fp32 logits give such rows the weights of the scalar
    ones: 0, so the tree is invalid and the others are what they were."""
    w = Workload("nonfinite", 5, 8008, levels=(2, 3), branching=(2, 2),
                 logit_dtype=torch.float32, sigma=1.0)
    inp = make_inputs(w, seed=8, device="cuda")
    clean = [x.clone() for x in _verify(tv, inp, path)[:3]]
    if value > 0:
        inp.logits[3, 0, 4001] = value
    else:
        inp.logits[3, 0] = value
    R = inp.parents.shape[1]
    v = tv.Verifier(8008, R - 1, 5, "fp32", path=path)
    out = v.verify(inp.parents, inp.tokens, inp.logits, inp.draft_probs, inp.temperature,
                   inp.uniforms)
    torch.cuda.synchronize()
    assert v.status() & ~16 == 64
    v.close()
    assert int(out[1][3]) == -1 and int(out[2][3]) == -1
    keep = [0, 1, 2, 4]
    for x, y in zip(out[:3], clean):
        assert torch.equal(x[keep], y[keep])
