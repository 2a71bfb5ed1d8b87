"""A call may read what the call just before it writes.  Every kernel of the library is launched ahead of its predecessor's end and
may start while calls further back still run; here a slow call (two chains in one piece, which leave most SMs free) writes the
initial state and the values of the next one, on one stream and with nothing in between, and the result has to be bit for
bit that of the same two calls with a synchronisation between them."""
import numpy as np
import pytest
import torch

import paper_2607_14568_b200 as gdn
from workloads import epilogue_inputs, get_config, make_inputs
from gdn_testlib import to_device

pytestmark = pytest.mark.gpu

T, H = 64 * 40, 2


@pytest.mark.parametrize("entry,nseg,hooks", [
    ("plain", 5, {}), ("plain", 5, {"gdn_debug_set_scan": 1}), ("plain", 1, {"gdn_debug_set_compact": 0}),
    ("plain", 1, {"gdn_debug_set_compact": 1}), ("plain", 0, {"gdn_debug_set_relay": 3}), ("raw", 4, {}), ("gated", 4, {}),
    ("gated", 1, {}), ("packed", 1, {}), ("snapshots", 3, {}), ("noalloc", 1, {}), ("fused", 1, {}), ("fp32", 1, {}), ("decode", 1, {}),
    ("attention", 1, {})])
def test_inputs_written_by_the_call_before(entry, nseg, hooks):
    L = gdn.lib()
    cfg = get_config("short", B=1, T=T, H=H, init_std=0.3, raw=(entry == "raw"), seed=90)
    first, d = to_device(make_inputs(get_config("short", B=1, T=T, H=H, init_std=0.3, seed=91))), to_device(make_inputs(cfg))
    if entry == "fp32":
        d = {n: x.float() if x is not None and x.dtype == torch.bfloat16 else x for n, x in d.items()}
    e = epilogue_inputs(cfg, (1, T))
    z = torch.from_numpy(e["z"].view(np.int16)).view(torch.bfloat16).cuda().reshape(1, T, H, 128)
    w = torch.from_numpy(e["weight"]).cuda()
    snaps = torch.empty(1, 5, H, 128, 128, device="cuda")
    cu = torch.tensor([0, 64 * 25 + 7, T], dtype=torch.int32, device="cuda")
    s0, v = first["final_state"], first["out"]                       # written by the first call
    fin2 = torch.empty(2, H, 128, 128, device="cuda")
    s02 = torch.empty(2, H, 128, 128, device="cuda")
    row = [d[n][:, 0].contiguous() for n in ("q", "k", "v", "log_alpha", "beta")]
    row_out = torch.empty(1, H, 128, dtype=torch.bfloat16, device="cuda")
    gates = (d["log_alpha"], d["beta"])

    def produce():
        L.gdn_debug_force_segments(1)
        L.gdn_debug_set_compact(0)
        gdn.gdn_chunk_prefill(first["q"], first["k"], first["v"], first["log_alpha"], first["beta"], first["initial_state"], v,
                              s02[1:] if entry == "packed" else s0)
        L.gdn_debug_set_compact(-1)

    def consume():
        L.gdn_debug_force_segments(nseg)
        for name, value in hooks.items():
            getattr(L, name)(value)
        if entry in ("plain", "noalloc", "fused"):
            if entry == "fused":
                L.gdn_debug_force_path(1)
            fn = gdn.gdn_chunk_prefill_noalloc if entry == "noalloc" else gdn.gdn_chunk_prefill
            r = fn(d["q"], d["k"], v, *gates, s0, d["out"], d["final_state"])
            L.gdn_debug_force_path(0)
        elif entry == "raw":
            r = gdn.gdn_chunk_prefill_raw(d["q"], d["k"], v, *gates, 0.05, 1e-6, s0, d["out"], d["final_state"])
        elif entry == "gated":
            r = gdn.gdn_chunk_prefill_gated(d["q"], d["k"], v, *gates, s0, z, w, 1e-6, d["out"], d["final_state"])
        elif entry == "packed":
            r = gdn.gdn_chunk_prefill(d["q"][0], d["k"][0], v[0], gates[0][0], gates[1][0], s02, d["out"][0], fin2, cu)
        elif entry == "snapshots":
            r = gdn.gdn_chunk_prefill_snapshots(d["q"], d["k"], v, *gates, s0, d["out"], d["final_state"], 8, snaps)
        elif entry == "fp32":
            r = gdn.gdn_chunk_prefill_f32(d["q"], d["k"], d["v"], *gates, s0, d["out"], d["final_state"])
        elif entry == "decode":
            r = gdn.gdn_decode_step(*row, s0, row_out)
        else:
            r = gdn.gdn_attn_causal_prefill(d["q"], d["k"], v, d["out"]), s0
        for name in hooks:
            getattr(L, name)(0 if name == "gdn_debug_set_scan" else -1)
        return r

    ws = torch.empty(gdn.gdn_workspace_bytes(1, T, H, 128, 128, False), dtype=torch.uint8, device="cuda")
    gdn.gdn_set_workspace(ws)
    try:
        s02.zero_()
        produce()
        torch.cuda.synchronize()
        want = [x.clone() for x in consume()]
        assert gdn.gdn_query_status() == 0
        for _ in range(10):
            s02.zero_(); s0.fill_(3.0); v.fill_(-2.0)
            d["out"].zero_(); d["final_state"].zero_(); fin2.zero_(); snaps.zero_(); row_out.zero_()
            produce()
            got = consume()
            torch.cuda.synchronize()
            assert gdn.gdn_query_status() == 0
            for a, b in zip(got, want):
                assert torch.equal(a, b)
    finally:
        for name in ("gdn_debug_set_compact", "gdn_debug_set_relay"):
            getattr(L, name)(-1)
        L.gdn_debug_set_scan(0)
        L.gdn_debug_force_path(0)
        L.gdn_debug_force_segments(0)
        gdn.gdn_set_workspace(None)
