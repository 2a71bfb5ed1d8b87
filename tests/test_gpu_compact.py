"""The form of the chain that reads no W (scratch items of (T diag beta)^T, P and the gate vectors only; used for grids that
are bound by memory) against the fp64 oracle, forced on small inputs: one chunk and less, ragged tails, more chunks than
any ring has slots, packed neighbours, wide values, raw projections and the fused output stage; a split (four or three segments)
keeps its W whatever is asked for."""
import numpy as np
import pytest
import torch

import oracle
import paper_2607_14568_b200 as gdn
from workloads import epilogue_inputs, get_config, make_inputs, widen
from gdn_testlib import BF16_MAX_ABS, BF16_REL_L2, assert_close, f64, to_device

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("entry,kw,nseg", [
    ("plain", dict(B=1, T=1, H=1, init_std=0.3), 1),
    ("plain", dict(B=1, T=63, H=2, init_std=0.3), 1),
    ("plain", dict(B=2, T=64 * 7 + 1, H=2, init_std=0.0), 1),
    ("plain", dict(B=1, T=64 * 13, H=2, d_v=256, init_std=0.3), 1),
    ("plain", dict(B=4, T=0, H=2, init_std=0.2, lengths=(130, 1, 64, 207)), 1),
    ("plain", dict(B=1, T=64 * 18 + 30, H=2, init_std=0.3), 4),
    ("raw", dict(B=2, T=64 * 5 + 23, H=2, init_std=0.3), 1),
    ("raw", dict(B=1, T=64 * 20, H=2, init_std=0.0), 3),
    ("gated", dict(B=2, T=64 * 5 + 23, H=2, init_std=0.3), 1),
    ("gated", dict(B=1, T=64 * 16 + 9, H=2, init_std=0.1), 4),
])
def test_compact_chain_matches_oracle(entry, kw, nseg):
    cfg = get_config("short", raw=(entry == "raw"), seed=77, **kw)
    x = make_inputs(cfg)
    d = to_device(x)
    L = gdn.lib()
    ws = torch.empty(max(gdn.gdn_workspace_bytes(len(x.lengths), x.T_arg, cfg.H, cfg.d_k, cfg.d_v, cfg.packed), 4096),
                     dtype=torch.uint8, device="cuda")
    gdn.gdn_set_workspace(ws)
    L.gdn_debug_force_segments(nseg)
    L.gdn_debug_set_compact(1)
    args = (d["q"], d["k"], d["v"], d["log_alpha"], d["beta"])
    tail = (d["out"], d["final_state"], d["cu_seqlens"])
    e = epilogue_inputs(cfg, x.q.shape[:-2])
    try:
        if entry == "raw":
            gdn.gdn_chunk_prefill_raw(*args, cfg.gate_scale, 1e-6, d["initial_state"], *tail)
        elif entry == "gated":
            z = torch.from_numpy(e["z"].view(np.int16)).view(torch.bfloat16).cuda()
            gdn.gdn_chunk_prefill_gated(*args, d["initial_state"], z, torch.from_numpy(e["weight"]).cuda(), 1e-6, *tail)
        else:
            gdn.gdn_chunk_prefill(*args, d["initial_state"], *tail)
        assert gdn.gdn_query_status_stream() == 0
    finally:
        L.gdn_debug_set_compact(-1)
        L.gdn_debug_force_segments(0)
        gdn.gdn_set_workspace(None)
    q, k, la, be = widen(x.q), widen(x.k), x.log_alpha, x.beta
    if entry == "raw":
        q, k, la, be = oracle.prologue(q, k, la, be, cfg.gate_scale, 1e-6)
    o, fin = oracle.sequential(q, k, widen(x.v), la, be, x.initial_state, x.cu_seqlens)
    bar = BF16_MAX_ABS
    if entry == "gated":
        plain, o = o, oracle.epilogue(o, widen(e["z"]), e["weight"], 1e-6)
        bar *= max(1.0, float(np.abs(o).max() / np.abs(plain).max()))
    assert_close(f64(d["out"]), o, BF16_REL_L2, bar, "out")
    assert_close(f64(d["final_state"]), fin, BF16_REL_L2, BF16_MAX_ABS, "final_state")


def test_many_items_per_cta_match_oracle_and_repeat_bit_for_bit():
    """2 x 41 chunks of 32 heads over four prepare CTAs per SM: each prepares four items and more, the next item's token-token product
    following straight on the reads of the previous one (the accumulator is handed back with the tiles)."""
    cfg = get_config("short", B=2, T=64 * 40 + 7, H=32, init_std=0.3, seed=79)
    x = make_inputs(cfg)
    d = to_device(x)
    ws = torch.empty(gdn.gdn_workspace_bytes(cfg.B, cfg.T, cfg.H, cfg.d_k, cfg.d_v, False), dtype=torch.uint8, device="cuda")
    gdn.gdn_set_workspace(ws)
    gdn.lib().gdn_debug_force_segments(1)
    gdn.lib().gdn_debug_set_compact(1)
    first = None
    try:
        for _ in range(6):
            d["out"].zero_(); d["final_state"].zero_()
            gdn.gdn_chunk_prefill(d["q"], d["k"], d["v"], d["log_alpha"], d["beta"], d["initial_state"], d["out"], d["final_state"])
            got = d["out"].clone(), d["final_state"].clone()
            first = first or got
            assert torch.equal(got[0], first[0]) and torch.equal(got[1], first[1])
        assert gdn.gdn_query_status_stream() == 0
    finally:
        gdn.lib().gdn_debug_set_compact(-1)
        gdn.lib().gdn_debug_force_segments(0)
        gdn.gdn_set_workspace(None)
    o, fin = oracle.sequential(widen(x.q), widen(x.k), widen(x.v), x.log_alpha, x.beta, x.initial_state, None)
    assert_close(f64(first[0]), o, BF16_REL_L2, BF16_MAX_ABS, "out")
    assert_close(f64(first[1]), fin, BF16_REL_L2, BF16_MAX_ABS, "final_state")
