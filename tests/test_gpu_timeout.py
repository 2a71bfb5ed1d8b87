"""Failure detection without a GPU fault: a TMA load that never happens makes the bounded waits of
one CTA expire (about a second each); the kernel must come back by itself with GDN_ERR_TIMEOUT in
the status word, leave the context usable, and the next call must be correct."""
import pytest
import torch

import paper_2607_14568_b200 as gdn
from workloads import get_config, make_inputs

from gdn_testlib import BF16_MAX_ABS, BF16_REL_L2, assert_close, f64, prefill_two_kernel, run_oracle, to_device

pytestmark = pytest.mark.gpu


def test_expired_wait_is_reported_and_the_context_survives():
    cfg = get_config("long", T=320, H=2, seed=95)
    x = make_inputs(cfg)
    d = to_device(x)
    L = gdn.lib()
    nbytes = gdn.gdn_workspace_bytes(cfg.B, cfg.T, cfg.H, cfg.d_k, cfg.d_v, False)
    ws = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    gdn.gdn_set_workspace(ws)
    L.gdn_debug_force_path(2)
    L.gdn_debug_force_segments(1)
    L.gdn_debug_drop_chunk(2)                        # chunk 2 of CTA (0,0,0) is never loaded
    try:
        gdn.gdn_chunk_prefill(d["q"], d["k"], d["v"], d["log_alpha"], d["beta"], d["initial_state"], d["out"],
                              d["final_state"])
        assert gdn.gdn_query_status() == 5           # GDN_ERR_TIMEOUT; the kernel returned on its own
    finally:
        L.gdn_debug_drop_chunk(-1)
        L.gdn_debug_force_segments(0)
        L.gdn_debug_force_path(0)
        gdn.gdn_set_workspace(None)
    assert L.gdn_debug_reset_status() == 0
    torch.cuda.synchronize()                         # no sticky CUDA error
    # the context is intact: the same problem now runs correctly
    o_ref, f_ref = run_oracle(x)
    out, fin = prefill_two_kernel(d["q"], d["k"], d["v"], d["log_alpha"], d["beta"], d["initial_state"], d["out"],
                                  d["final_state"])
    assert_close(f64(out), o_ref, BF16_REL_L2, BF16_MAX_ABS, "out after a timed-out call")
    assert_close(f64(fin), f_ref, BF16_REL_L2, BF16_MAX_ABS, "state after a timed-out call")


def test_expired_counter_wait_in_the_merged_kernel_is_reported_and_the_context_survives():
    """The merged scan kernel hands over between its phases through counters in global memory.  A test hook
    makes one CTA not raise its counter; the CTAs of that head that wait for it must give up after about a
    second, report GDN_ERR_TIMEOUT, run to their end, and leave the counters clean for the next call."""
    cfg = get_config("long", T=64 * 12, H=2, seed=96)
    x = make_inputs(cfg)
    d = to_device(x)
    L = gdn.lib()
    ws = torch.empty(gdn.gdn_workspace_bytes(cfg.B, cfg.T, cfg.H, cfg.d_k, cfg.d_v, False), dtype=torch.uint8, device="cuda")
    gdn.gdn_set_workspace(ws)
    L.gdn_debug_force_path(2)
    L.gdn_debug_force_segments(3)
    L.gdn_debug_set_scan(1)
    L.gdn_debug_drop_chunk(-2)                       # CTA (0,0,0) keeps its segment summary to itself
    try:
        gdn.gdn_chunk_prefill(d["q"], d["k"], d["v"], d["log_alpha"], d["beta"], d["initial_state"], d["out"],
                              d["final_state"])
        assert gdn.gdn_query_status() == 5
        L.gdn_debug_drop_chunk(-1)
        assert L.gdn_debug_reset_status() == 0
        torch.cuda.synchronize()
        # same workspace, same counters: the next merged call is correct
        gdn.gdn_chunk_prefill(d["q"], d["k"], d["v"], d["log_alpha"], d["beta"], d["initial_state"], d["out"],
                              d["final_state"])
        assert gdn.gdn_query_status() == 0
    finally:
        L.gdn_debug_drop_chunk(-1)
        L.gdn_debug_force_segments(0)
        L.gdn_debug_set_scan(0)
        L.gdn_debug_force_path(0)
        gdn.gdn_set_workspace(None)
    o_ref, f_ref = run_oracle(x)
    assert_close(f64(d["out"]), o_ref, BF16_REL_L2, BF16_MAX_ABS, "out after a timed-out merged call")
    assert_close(f64(d["final_state"]), f_ref, BF16_REL_L2, BF16_MAX_ABS, "state after a timed-out merged call")


@pytest.mark.parametrize("raw,compact", [(False, 0), (False, 1), (True, 0)])
def test_expired_wait_in_the_prepare_kernel_is_reported_and_the_context_survives(raw, compact):
    """Every CTA expects more bytes than its tiles have: the wait on its first item's runs out, the item is gone through all the
    same, and the roles of the CTA leave their loop together."""
    cfg = get_config("short", B=1, T=64 * 100, H=16, raw=raw, seed=97)     # more items than CTAs
    x = make_inputs(cfg)
    d = to_device(x)
    L = gdn.lib()
    ws = torch.zeros(gdn.gdn_workspace_bytes(cfg.B, cfg.T, cfg.H, cfg.d_k, cfg.d_v, False), dtype=torch.uint8, device="cuda")
    args = (d["q"], d["k"], d["v"], d["log_alpha"], d["beta"])

    def call():
        if raw:
            gdn.gdn_chunk_prefill_raw(*args, cfg.gate_scale, 1e-6, None, d["out"], d["final_state"])
        else:
            gdn.gdn_chunk_prefill(*args, None, d["out"], d["final_state"])

    gdn.gdn_set_workspace(ws)
    L.gdn_debug_force_path(2)
    L.gdn_debug_force_segments(1)
    L.gdn_debug_set_compact(compact)
    try:
        call()
        assert gdn.gdn_query_status() == 0
        want = d["out"].clone(), d["final_state"].clone()
        L.gdn_debug_drop_chunk(-3)
        call()
        assert gdn.gdn_query_status() == 5           # GDN_ERR_TIMEOUT; the kernels returned on their own
        L.gdn_debug_drop_chunk(-1)
        assert L.gdn_debug_reset_status() == 0
        torch.cuda.synchronize()                     # no sticky CUDA error
        gdn.gdn_set_workspace(ws)                    # as the header asks for after a time-out
        d["out"].zero_(); d["final_state"].zero_()
        call()
        assert gdn.gdn_query_status() == 0
        assert torch.equal(d["out"], want[0]) and torch.equal(d["final_state"], want[1])
    finally:
        L.gdn_debug_drop_chunk(-1)
        L.gdn_debug_set_compact(-1)
        L.gdn_debug_force_segments(0)
        L.gdn_debug_force_path(0)
        gdn.gdn_set_workspace(None)


@pytest.mark.parametrize("compact", [0, 1])
def test_expired_counter_wait_of_a_relayed_chain_is_reported_and_the_context_survives(compact):
    """The first piece of one chain does not say that it is done: the piece behind it gives up after a second, reports the time-out
    and runs to its end, so do the others, and the next call on the workspace, set again as the header asks, is correct."""
    cfg = get_config("short", B=1, T=64 * 9 + 3, H=3, seed=98)
    x = make_inputs(cfg)
    d = to_device(x)
    L = gdn.lib()
    ws = torch.zeros(gdn.gdn_workspace_bytes(cfg.B, cfg.T, cfg.H, cfg.d_k, cfg.d_v, False), dtype=torch.uint8, device="cuda")
    call = lambda: gdn.gdn_chunk_prefill(d["q"], d["k"], d["v"], d["log_alpha"], d["beta"], None, d["out"], d["final_state"])
    gdn.gdn_set_workspace(ws)
    L.gdn_debug_force_path(2)
    L.gdn_debug_set_relay(3)
    L.gdn_debug_set_compact(compact)
    L.gdn_debug_drop_chunk(-2)
    try:
        call()
        assert gdn.gdn_query_status() == 5
        L.gdn_debug_drop_chunk(-1)
        assert L.gdn_debug_reset_status() == 0
        torch.cuda.synchronize()
        gdn.gdn_set_workspace(ws)
        call()
        assert gdn.gdn_query_status() == 0
    finally:
        L.gdn_debug_drop_chunk(-1)
        L.gdn_debug_set_compact(-1)
        L.gdn_debug_set_relay(-1)
        L.gdn_debug_force_path(0)
        gdn.gdn_set_workspace(None)
    o_ref, f_ref = run_oracle(x)
    assert_close(f64(d["out"]), o_ref, BF16_REL_L2, BF16_MAX_ABS, "out after a timed-out relay")
    assert_close(f64(d["final_state"]), f_ref, BF16_REL_L2, BF16_MAX_ABS, "state after a timed-out relay")
