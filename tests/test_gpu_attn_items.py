"""Attention: how the query tiles are dealt out to the SMs (single tiles or pairs, one or several
items per CTA, packed sequences of every kind), against the fp64 oracle."""
import numpy as np
import pytest
import torch

import oracle
from workloads import get_attn_config, make_attn_inputs, widen
from gdn_testlib import assert_close, f64

pytestmark = pytest.mark.gpu


def _dev(a):
    return torch.from_numpy(a.view(np.int16)).view(torch.bfloat16).cuda()


def _check(B, T, Hq, Hkv, lens=None):
    import paper_2607_14568_b200 as gdn
    cfg = get_attn_config("attn_small", B=B, T=T, Hq=Hq, Hkv=Hkv)
    q, k, v = make_attn_inputs(cfg)
    if lens is not None:
        q, k, v = q[0], k[0], v[0]
    dq, dk, dv = _dev(q), _dev(k), _dev(v)
    cu = None if lens is None else torch.tensor([0] + lens).cumsum(0).to(device="cuda", dtype=torch.int32)
    out = torch.full_like(dq, float("nan"))
    gdn.gdn_attn_causal_prefill(dq, dk, dv, out, cfg.scale, cu_seqlens=cu)
    torch.cuda.synchronize()
    assert gdn.gdn_query_status() == 0
    q, k, v = widen(q), widen(k), widen(v)
    if lens is None:
        assert_close(f64(out), oracle.attention_causal(q, k, v, cfg.scale), 5e-3, 2e-2, "out")
        return
    tok = 0
    for n in lens:
        s = slice(tok, tok + n)
        tok += n
        if n:
            want = oracle.attention_causal(q[None, s], k[None, s], v[None, s], cfg.scale)[0]
            assert_close(f64(out[s]), want, 5e-3, 2e-2, f"out of {n} tokens at {s.start}")


# 148 SMs: one tile per item below 296 of them, pairs from there on; one item per SM, two, or several taken over
@pytest.mark.parametrize("B,T,Hq", [(1, 129, 74), (1, 257, 98), (1, 257, 99), (37, 129, 4), (5, 385, 30), (1, 1281, 29)])
def test_items(B, T, Hq):
    _check(B, T, Hq, Hq)


@pytest.mark.parametrize("lens", [[1] * 40, [0, 300, 0, 128, 129, 0], [(37 * i) % 290 for i in range(70)], [1, 1300, 255, 256, 257]])
@pytest.mark.parametrize("heads", [(2, 1), (16, 4)])
def test_packed_items(lens, heads):
    _check(1, sum(lens), heads[0], heads[1], lens)
