"""Attention: what stands behind the end of a sequence in memory does not reach it.  The last key tile of a sequence is
completed with the rows that follow, which belong to somebody else; here they are infinite or not numbers."""
import numpy as np
import pytest
import torch

import oracle
import paper_2607_14568_b200 as gdn
from workloads import get_attn_config, make_attn_inputs, widen
from gdn_testlib import assert_close, f64

pytestmark = pytest.mark.gpu


def _dev(a):
    return torch.from_numpy(a.view(np.int16)).view(torch.bfloat16).cuda()


# lengths with the spoiled sequences between the good ones: a tail of one row, of all but one, single tiles and pairs, several
# items per CTA, grouped heads
@pytest.mark.parametrize("lens,spoiled,heads", [((65, 128, 7), (1,), (2, 1)), ((1, 200, 127, 200, 129, 40), (1, 3, 5), (4, 2)),
                                                ((383, 300, 511, 260), (1, 3), (2, 2)), ((700, 64) * 12, tuple(range(1, 24, 2)), (16, 4))])
def test_neighbours_that_are_not_finite(lens, spoiled, heads):
    cfg = get_attn_config("attn_small", B=1, T=sum(lens), Hq=heads[0], Hkv=heads[1])
    q, k, v = (a[0] for a in make_attn_inputs(cfg))
    dq, dk, dv = _dev(q), _dev(k), _dev(v)
    ends = np.cumsum((0,) + lens)
    for n in spoiled:
        for i, bad in enumerate((float("nan"), float("inf"), -float("inf"))):
            dv[ends[n] + i:ends[n + 1]:3] = bad
            dk[ends[n] + i:ends[n + 1]:3] = bad
            dq[ends[n] + i:ends[n + 1]:3] = bad
    out = torch.empty_like(dq)
    gdn.gdn_attn_causal_prefill(dq, dk, dv, out, cfg.scale, cu_seqlens=torch.from_numpy(ends.astype(np.int32)).cuda())
    torch.cuda.synchronize()
    assert gdn.gdn_query_status() == 0
    q, k, v = widen(q), widen(k), widen(v)
    for n in set(range(len(lens))) - set(spoiled):
        s = slice(ends[n], ends[n + 1])
        assert_close(f64(out[s]), oracle.attention_causal(q[None, s], k[None, s], v[None, s], cfg.scale)[0], 5e-3, 2e-2, f"sequence {n}")


def test_batched_neighbours_that_are_not_finite():
    cfg = get_attn_config("attn_small", B=3, T=203, Hq=4, Hkv=2)
    q, k, v = make_attn_inputs(cfg)
    dq, dk, dv = _dev(q), _dev(k), _dev(v)
    dk[1] = float("inf")
    dv[1] = float("nan")
    out = torch.empty_like(dq)
    gdn.gdn_attn_causal_prefill(dq, dk, dv, out, cfg.scale)
    torch.cuda.synchronize()
    want = oracle.attention_causal(widen(q), widen(k), widen(v), cfg.scale)
    for n in (0, 2):
        assert_close(f64(out[n]), want[n], 5e-3, 2e-2, f"sequence {n}")
