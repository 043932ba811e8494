"""Target rows with tokens far below the row's maximum -- masked logits (-inf) at
temperatures where the exponent of anything below the maximum leaves float32's
integers -- on every path, in residual and in leaf draws, against the oracle."""

import pytest
import torch

from oracle.verify import verify_batch
from tests.parity import assert_rate_budget, compare_batch, to_numpy_inputs
from workloads.synth import Workload, make_inputs

pytestmark = pytest.mark.gpu

PATH_CODE = {"two": 0, "cluster": 1, "persistent": 2}


def _inputs(B, V, dtype, T, shift=0.0, masked=0.3, seed=0):
    """Logits shift + T l for l of unit temperature, a share of them -inf: of the
    drafted tokens too in odd trees (rate 0, draws from the residual), never in
    even ones (leaves are accepted)."""
    w = Workload("masked", B, V, levels=(3, 5, 4), branching=(3, 2, 1), sigma=0.4)
    inp = make_inputs(w, seed=seed, device="cuda")
    lg = inp.logits.float() * T + shift
    g = torch.Generator(device="cuda").manual_seed(seed + 1)
    out = torch.rand(lg.shape, generator=g, device="cuda") < masked
    for i in range(1, inp.parents.shape[1]):
        rows = torch.arange(0, B, 2, device="cuda")
        out[rows, inp.parents[0, i].long(), inp.tokens[rows, i].long()] = False
    lg[out] = float("-inf")
    inp.logits = lg.to(dtype)
    inp.temperature = T
    return inp


def _run(inp, path):
    import paper_2505_12398_gb300 as tv
    B, R = inp.parents.shape
    V = inp.logits.shape[-1]
    dt = "bf16" if inp.logits.dtype == torch.bfloat16 else "fp32"
    v = tv.Verifier(V, R - 1, B, dt, path="auto" if path == "two" else path)
    assert v.launch_shape(B, R - 1)[0] == PATH_CODE[path]
    out = v.verify(inp.parents, inp.tokens, inp.logits, inp.draft_probs, inp.temperature,
                   inp.uniforms, debug=True)
    torch.cuda.synchronize()
    assert v.status() & ~16 == 0
    v.close()
    return out


def _check(inp, out):
    path, tau, bonus, node_p, stats = [t.cpu().numpy() for t in out]
    par, tok, lg, dp, un = to_numpy_inputs(inp)
    _, _, _, det = verify_batch(par, tok, lg, dp, inp.temperature, un, keep_cdf=True)
    summ = compare_batch(det, path, tau, bonus, node_p, stats)
    assert not summ["bad"], summ["bad"][:5]
    assert_rate_budget(summ)
    leaf = [r["leaf_row_read"] for r in det.values()]
    assert any(leaf) and not all(leaf)       # both kinds of draw


@pytest.mark.parametrize("path,V,dtype", [
    ("cluster", 8008, torch.bfloat16), ("cluster", 65544, torch.bfloat16),
    ("persistent", 8008, torch.bfloat16), ("two", 8005, torch.bfloat16),
    ("cluster", 8008, torch.float32), ("two", 8005, torch.float32)])
@pytest.mark.parametrize("T", [1e-4, 1e-5])
def test_masked_logits_at_low_temperatures(path, V, dtype, T):
    """The weight of a masked token is 0 however large the exponent."""
    inp = _inputs(8, V, dtype, T, seed=V % 1000)
    _check(inp, _run(inp, path))


@pytest.mark.parametrize("path,V,dtype", [
    ("two", 8005, torch.float32), ("two", 40003, torch.float32), ("two", 8005, torch.bfloat16),
    ("cluster", 8008, torch.float32), ("cluster", 8008, torch.bfloat16),
    ("persistent", 8008, torch.float32), ("persistent", 8008, torch.bfloat16)])
@pytest.mark.parametrize("T", [1e-6, 1e-9, 1e-20])
def test_one_token_holds_the_mass(path, V, dtype, T):
    """Ordinary logits at a temperature that leaves each row's largest all of the mass,
    down to where the least exponent times T is lost beside the logit; even trees drafted
    it, so that leaves are accepted."""
    inp = _inputs(6, V, dtype, 1.0, masked=0.1, seed=V % 1000)
    inp.temperature = T
    par = inp.parents[0].tolist()
    for i in range(len(par)):
        kids = [c for c in range(1, len(par)) if par[c] == i]
        if not kids:
            continue
        # (bf16 rows have ties at the top)
        top = inp.logits[:, i].float().argmax(dim=-1).to(torch.int32)
        inp.logits[torch.arange(6), i, top.long()] += 1.0
        for b in range(0, 6, 2):
            for c in kids[1:]:
                if inp.tokens[b, c] == top[b]:
                    inp.tokens[b, c] = inp.tokens[b, kids[0]]
            inp.tokens[b, kids[0]] = top[b]
    _check(inp, _run(inp, path))


def _given(inp):
    """(max, sum of 2^((l - max) log2(e) / T)) of every row, in float64."""
    lf = inp.logits.double()
    m = lf.max(dim=-1).values
    s = torch.exp((lf - m[..., None]) / inp.temperature).sum(dim=-1)
    return torch.stack([m, s], dim=-1).float().contiguous()


@pytest.mark.parametrize("path,V,dtype", [
    ("cluster", 8008, torch.bfloat16), ("cluster", 65544, torch.bfloat16),
    ("persistent", 8008, torch.bfloat16), ("two", 8005, torch.bfloat16),
    ("cluster", 8008, torch.float32), ("persistent", 8008, torch.float32),
    ("two", 8005, torch.float32)])
@pytest.mark.parametrize("shift", [-30000.0, 30000.0])
def test_rows_far_from_zero(path, V, dtype, shift):
    """Weights depend on the distance to the row's maximum alone: rows wholly below (or
    above) what a masked logit might be taken for, with normalisers of the call's own
    and given ones."""
    inp = _inputs(8, V, dtype, 300.0, shift=shift, seed=V % 1000)
    _check(inp, _run(inp, path))
    if path == "two":
        return
    import paper_2505_12398_gb300 as tv
    B, R = inp.parents.shape
    # (a handle of the cluster path does not take normalisers; one that chooses does)
    v = tv.Verifier(V, R - 1, B, "bf16" if dtype == torch.bfloat16 else "fp32",
                    path="auto" if path == "cluster" else path)
    assert v.launch_shape(B, R - 1)[0] == PATH_CODE[path]
    out = v.verify_stats(inp.parents, inp.tokens, inp.logits, inp.draft_probs, inp.temperature,
                         inp.uniforms, _given(inp), debug=True)
    torch.cuda.synchronize()
    assert v.status() & ~16 == 0
    v.close()
    _check(inp, out)


@pytest.mark.parametrize("path,V", [("cluster", 8008), ("persistent", 8008), ("two", 8005)])
@pytest.mark.parametrize("value", [float("-inf"), float("inf")])
def test_bf16_rows_without_a_normaliser(path, V, value):
    """A row the traversal needs without a finite logit, or with +inf, makes its tree
    invalid and no other."""
    import paper_2505_12398_gb300 as tv
    inp = _inputs(6, V, torch.bfloat16, 1.0)
    clean = _run(inp, path)
    if value < 0:
        inp.logits[2, 0] = value
    else:
        inp.logits[2, 0, V - 3] = value
    R = inp.parents.shape[1]
    v = tv.Verifier(V, R - 1, 6, "bf16", path="auto" if path == "two" else path)
    out = v.verify(inp.parents, inp.tokens, inp.logits, inp.draft_probs, 1.0, inp.uniforms)
    torch.cuda.synchronize()
    assert v.status() & ~16 == 64
    v.close()
    assert int(out[1][2]) == -1 and int(out[2][2]) == -1 and (out[0][2] == -1).all()
    keep = [0, 1, 3, 4, 5]
    for x, y in zip(out[:3], clean):
        assert torch.equal(x[keep], y[keep])


@pytest.mark.parametrize("path,V", [("cluster", 8008), ("persistent", 8008), ("two", 8005)])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
def test_masked_logits_at_a_high_temperature(path, V, dtype):
    """Nor does a masked token weigh anything where a bound on the distance to the row's
    maximum, 1e4 say, would leave it e^-5."""
    inp = _inputs(8, V, dtype, 2000.0, seed=V % 1000)
    _check(inp, _run(inp, path))
