"""CPU checks of the error bounds the GPU parity tests rely on, by replaying
the kernels' own float32 / float64 operation order with numpy (IEEE
round-to-nearest-even in both, as on the GPU).

Drafting (tv_draft.cu): a lane sums its 8 tokens pairwise in float32 and a warp
adds its 32 lane sums with a 5-step xor butterfly in float32 (a 256-token tile
sum).  One warp adds 32 runs of consecutive tile sums in float64, each run in two
interleaved chains, and scans the run totals across lanes (Hillis-Steele); their
last is the row's total.  A child's run is found from those prefixes less the
earlier siblings' masses; inside it the tiles are scanned 32 at a time on top of
the prefix before the run (siblings' masses taken off their tiles), inside the
crossing tile the lanes' 8-token sums (siblings' tokens as 0), inside the crossing
lane its 8 tokens, every step starting from the prefix before what it scans.  The
GPU drafting tests allow a token to differ from the oracle's only when u W is
within 1e-6 W of a step of the exact CDF; these tests measure how far every
prefix the kernel compares u W with is from the exact one."""

import numpy as np
import pytest

TILE = 256


def scan(v):
    """The warp's inclusive scan (Hillis-Steele) of up to 32 float64 values."""
    x = np.array(v, dtype=np.float64)
    o = 1
    while o < len(x):
        y = np.concatenate([np.zeros(o), x[:-o]])
        x = np.where(np.arange(len(x)) >= o, x + y, x)
        o *= 2
    return x


def tile_sums_f32(q):
    """The kernel's float32 tile sums of a row (zeros past the end)."""
    V = len(q)
    n_tiles = (V + TILE - 1) // TILE
    x = np.zeros(n_tiles * TILE, dtype=np.float32)
    x[:V] = q.astype(np.float32)
    v = x.reshape(n_tiles, 32, 8)
    s = ((v[..., 0] + v[..., 1]) + (v[..., 2] + v[..., 3])) + \
        ((v[..., 4] + v[..., 5]) + (v[..., 6] + v[..., 7]))       # [tiles, 32] lane sums
    lane = np.arange(32)
    for o in (16, 8, 4, 2, 1):                                     # xor butterfly
        s = (s + s[:, lane ^ o]).astype(np.float32)
    return s[:, 0]


def run_prefixes(tsum):
    """(tiles per run, inclusive prefixes of the 32 runs)."""
    n = len(tsum)
    per = (n + 31) // 32
    runs = np.zeros(32)
    for lane in range(32):
        ts = [float(x) for x in tsum[min(n, lane * per):min(n, lane * per + per)]]
        run = odd = 0.0
        for k in range(0, len(ts) - 1, 2):
            run += ts[k]
            odd += ts[k + 1]
        if len(ts) % 2:
            run += ts[-1]
        runs[lane] = run + odd
    return per, scan(runs)


def run_and_tile_prefixes(tsum, removed=()):
    """Every prefix the kernel forms above a tile once the (token, mass) pairs
    `removed` are gone: those of the runs and those of the tiles, and W."""
    n = len(tsum)
    per, upto = run_prefixes(tsum)
    incl = upto.copy()
    rsum = 0.0
    for tok, m in removed:
        for lane in range(32):
            if tok // TILE < min(n, min(n, lane * per) + per):
                incl[lane] -= m
        rsum += m
    tiles = np.zeros(n)
    for f in range(32):
        lo, hi = min(n, f * per), min(n, f * per + per)
        base = incl[f - 1] if f else 0.0
        for t0 in range(lo, hi, 32):
            d = np.zeros(32)
            d[:min(32, hi - t0)] = tsum[t0:min(t0 + 32, hi)].astype(np.float64)
            for tok, m in removed:
                if t0 <= tok // TILE < min(t0 + 32, hi):
                    d[tok // TILE - t0] -= m
            x = base + scan(d)
            tiles[t0:min(t0 + 32, hi)] = x[:min(32, hi - t0)]
            base = x[31]
    return incl, tiles, upto[31] - rsum


def token_prefixes(q, t, base, removed=()):
    """The prefixes of the tokens of tile t, on top of `base` before it."""
    v = np.zeros(TILE)
    part = q[t * TILE:(t + 1) * TILE]
    v[:len(part)] = part
    for tok, _ in removed:
        if tok // TILE == t:
            v[tok - t * TILE] = 0.0
    w = v.reshape(32, 8)
    ls = ((w[:, 0] + w[:, 1]) + (w[:, 2] + w[:, 3])) + ((w[:, 4] + w[:, 5]) + (w[:, 6] + w[:, 7]))
    x = base + scan(ls)
    out = np.zeros((32, 8))
    for lane in range(32):
        out[lane] = (x[lane - 1] if lane else base) + scan(w[lane])
    return out.reshape(-1), x


def test_replay_matches_a_direct_sum_on_exact_rows():
    """On dyadic rows every float32 and float64 sum is exact, so the replay
    must give the exact prefixes (a check of the replay itself)."""
    rng = np.random.default_rng(0)
    q = rng.integers(0, 64, 20000).astype(np.float64) / 1024.0
    removed = [(int(t), float(q[t])) for t in (3, 255, 256, 7000, 19999)]
    left = q.copy()
    left[[t for t, _ in removed]] = 0.0
    tsum = tile_sums_f32(q)
    incl, tiles, W = run_and_tile_prefixes(tsum, removed)
    padded = np.pad(left, (0, (-len(q)) % TILE))
    want = np.cumsum(padded.reshape(-1, TILE).sum(1))
    per, _ = run_prefixes(tsum)
    assert np.array_equal(tiles, want) and W == want[-1]
    assert np.array_equal(incl, want[np.minimum(np.arange(1, 33) * per, len(want)) - 1])
    cdf = np.cumsum(padded)
    for t in (0, 1, 27, len(want) - 1):
        tok, _ = token_prefixes(q, t, want[t - 1] if t else 0.0, removed)
        assert np.array_equal(tok, cdf[t * TILE:(t + 1) * TILE])


@pytest.mark.parametrize("V,scale", [(1000, 3.0), (32003, 3.0), (128256, 3.0), (151936, 1.0)])
def test_drafting_prefix_error_bound(V, scale):
    """Every prefix that the kernel compares u W with is within 5e-7 W of the exact
    cumulative sum (float64 of the float32 row values) on draft rows of the
    workloads' kind (softmax of scaled Gaussian logits), for the first child and
    for one whose seven earlier siblings are gone."""
    rng = np.random.default_rng(V)
    worst = 0.0
    for _ in range(4):
        z = rng.standard_normal(V) * scale
        q = np.exp(z - z.max())
        q = (q / q.sum()).astype(np.float32).astype(np.float64)
        tsum = tile_sums_f32(q)
        per, _ = run_prefixes(tsum)
        gone = rng.choice(V, size=7, replace=False, p=q / q.sum())
        for removed in ([], [(int(t), float(q[t])) for t in gone]):
            left = q.copy()
            left[[t for t, _ in removed]] = 0.0
            incl, tiles, W = run_and_tile_prefixes(tsum, removed)
            padded = np.pad(left, (0, (-V) % TILE))
            cdf = np.cumsum(padded)
            exact = cdf[TILE - 1::TILE]
            at = np.minimum(np.arange(1, 33) * per, len(exact)) - 1
            err = [np.abs(tiles - exact).max(), np.abs(incl - exact[at]).max(),
                   abs(W - exact[-1])]
            for t in rng.choice(len(tiles), size=min(8, len(tiles)), replace=False):
                tok, lanes = token_prefixes(q, t, tiles[t - 1] if t else 0.0, removed)
                err.append(np.abs(tok - cdf[t * TILE:(t + 1) * TILE]).max())
                err.append(np.abs(lanes - cdf[t * TILE:(t + 1) * TILE][7::8]).max())
            worst = max(worst, float(max(err) / exact[-1]))
    print(f"\nV={V}: worst prefix error {worst:.2e} W")
    assert worst < 5e-7
