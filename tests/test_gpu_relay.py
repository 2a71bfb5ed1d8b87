"""Chains cut into pieces that relay their state through final_state inside one launch (used when more chains than SMs do not
fill a whole number of rounds) against the fp64 oracle, forced on small inputs: ragged last pieces, more pieces than chunks
allow, wide values, an initial state that final_state aliases, the form without W, the output stage, repeated calls."""
import numpy as np
import pytest
import torch

import oracle
import paper_2607_14568_b200 as gdn
from workloads import epilogue_inputs, get_config, make_inputs, widen
from gdn_testlib import BF16_MAX_ABS, BF16_REL_L2, assert_close, f64, to_device

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pieces,kw,alias,compact,gated", [
    (2, dict(B=1, T=64 * 2, H=1, init_std=0.3), False, 0, False),
    (3, dict(B=2, T=64 * 7 + 5, H=3, init_std=0.0), False, 0, False),
    (5, dict(B=1, T=64 * 13, H=2, d_v=256, init_std=0.3), True, 0, False),
    (9, dict(B=1, T=64 * 4 + 63, H=2, init_std=0.3), True, 0, False),
    (4, dict(B=2, T=64 * 9 + 1, H=2, init_std=0.3), False, 1, False),
    (3, dict(B=1, T=64 * 8 + 40, H=2, init_std=0.1), False, 0, True),
    (2, dict(B=4, T=64 * 6, H=50, init_std=0.1), True, 0, False),          # more pieces than SMs
])
def test_relayed_chains_match_oracle(pieces, kw, alias, compact, gated):
    cfg = get_config("short", seed=78, **kw)
    x = make_inputs(cfg)
    d = to_device(x)
    L = gdn.lib()
    ws = torch.empty(gdn.gdn_workspace_bytes(cfg.B, cfg.T, cfg.H, cfg.d_k, cfg.d_v, False), dtype=torch.uint8, device="cuda")
    gdn.gdn_set_workspace(ws)
    L.gdn_debug_set_relay(pieces)
    L.gdn_debug_set_compact(compact)
    e = epilogue_inputs(cfg, x.q.shape[:-2])
    try:
        for _ in range(2):                                       # the second call finds the counters the first one left
            s0 = d["initial_state"]
            fin = d["final_state"]
            if alias:
                fin.copy_(s0)
                s0 = fin
            args = (d["q"], d["k"], d["v"], d["log_alpha"], d["beta"], s0)
            if gated:
                z = torch.from_numpy(e["z"].view(np.int16)).view(torch.bfloat16).cuda()
                gdn.gdn_chunk_prefill_gated(*args, z, torch.from_numpy(e["weight"]).cuda(), 1e-6, d["out"], fin)
            else:
                gdn.gdn_chunk_prefill(*args, d["out"], fin)
        assert gdn.gdn_query_status_stream() == 0
    finally:
        L.gdn_debug_set_compact(-1)
        L.gdn_debug_set_relay(-1)
        gdn.gdn_set_workspace(None)
    o, want = oracle.sequential(widen(x.q), widen(x.k), widen(x.v), x.log_alpha, x.beta, x.initial_state, None)
    bar = BF16_MAX_ABS
    if gated:
        plain, o = o, oracle.epilogue(o, widen(e["z"]), e["weight"], 1e-6)
        bar *= max(1.0, float(np.abs(o).max() / np.abs(plain).max()))
    assert_close(f64(d["out"]), o, BF16_REL_L2, bar, "out")
    assert_close(f64(d["final_state"]), want, BF16_REL_L2, BF16_MAX_ABS, "final_state")
