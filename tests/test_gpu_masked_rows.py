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
