"""The LM head at the edges of its tiles and of its two forms (single SMs up to
128 rows, SM pairs above): a few rows, one row past a form's or a tile's
boundary, column tiles cut by the vocabulary, and rows too short for 32-byte
stores, on exact operands (bit for bit against the oracle)."""

import numpy as np
import pytest
import torch

from oracle import lmhead

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,K,V", [(1, 64, 8), (1, 4096, 1000), (61, 128, 33000), (128, 192, 520),
                                   (129, 64, 264), (129, 512, 40008), (257, 128, 24),
                                   (511, 64, 5000), (513, 320, 20008)])
def test_exact_operands_at_tile_edges(M, K, V):
    import paper_2505_12398_gb300 as tv
    g = torch.Generator().manual_seed(M + K + V)
    H = (torch.randint(-8, 9, (M, K), generator=g).float() / 16).to(torch.bfloat16)
    W = (torch.randint(-8, 9, (V, K), generator=g).float() / 16).to(torch.bfloat16)
    v = tv.Verifier(V, 0, M, "bf16")
    lg, st = v.lm_head(H.cuda(), W.cuda(), 0.8)
    # a logits array that starts 16 but not 32 bytes into a sector
    buf = torch.empty(M * V + 8, dtype=torch.bfloat16, device="cuda")
    off = buf[8:].view(M, V)
    st2 = torch.empty_like(st)
    v.lm_head(H.cuda(), W.cuda(), 0.8, out=(off, st2))
    torch.cuda.synchronize()
    assert v.status() == 0
    v.close()
    ref = lmhead.to_bf16(lmhead.logits(H.float().numpy(), W.float().numpy()))
    assert np.array_equal(lg.float().cpu().numpy().astype(np.float64), ref)
    assert torch.equal(lg, off) and torch.equal(st, st2)
    m, s = lmhead.row_stats(ref, 0.8)
    st = st.cpu().numpy().astype(np.float64)
    assert np.array_equal(st[:, 0], m)
    assert np.max(np.abs(st[:, 1] - s) / s) < 1e-5   # the parity bar of the normalisers


def test_handle_of_more_rows_than_an_int_counts():
    """2^31 rows of 8 tokens: 16 GiB of row statistics and of scratch on the handle, a call of
    a few rows as on any other."""
    import paper_2505_12398_gb300 as tv
    if torch.cuda.mem_get_info()[0] < 64 << 30:
        pytest.skip("not enough free device memory")
    g = torch.Generator().manual_seed(5)
    H = (torch.randint(-8, 9, (5, 64), generator=g).float() / 16).to(torch.bfloat16)
    W = (torch.randint(-8, 9, (8, 64), generator=g).float() / 16).to(torch.bfloat16)
    v = tv.Verifier(8, 1023, 1 << 21, "bf16", path="three")
    lg, _ = v.lm_head(H.cuda(), W.cuda(), 1.0)
    torch.cuda.synchronize()
    v.close()
    ref = lmhead.to_bf16(lmhead.logits(H.float().numpy(), W.float().numpy()))
    assert np.array_equal(lg.float().cpu().numpy().astype(np.float64), ref)
