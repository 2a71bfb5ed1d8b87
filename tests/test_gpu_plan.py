"""The plans the library makes from the sizes of a call: which kernels run (counted launches), and that what they return is the
oracle's result on both sides of a line."""
import pytest
import torch

import oracle
import paper_2607_14568_b200 as gdn
from workloads import get_config, make_inputs, widen
from gdn_testlib import BF16_MAX_ABS, BF16_REL_L2, F32_REL_L2, assert_close, f64, run_lib, run_oracle, to_device

pytestmark = pytest.mark.gpu


# Two CTAs of a chain share its keys, queries and prepared items (d_v = 256): a split costs them less memory than two chains
@pytest.mark.parametrize("T,H,d_v,launches", [(4096, 16, 256, 4), (10240, 24, 256, 4), (4096, 24, 256, 2), (2048, 16, 256, 2),
                                              (2048, 16, 128, 4), (1024, 16, 128, 2)])
def test_sequence_split_by_the_rule(T, H, d_v, launches):
    cfg = get_config("short", B=1, T=T, H=H, d_v=d_v, init_std=0.02, seed=81)
    x = make_inputs(cfg)
    d = to_device(x)
    ws = torch.empty(gdn.gdn_workspace_bytes(1, T, H, cfg.d_k, d_v, False), dtype=torch.uint8, device="cuda")
    gdn.gdn_set_workspace(ws)
    try:
        n0 = gdn.gdn_launch_count()
        gdn.gdn_chunk_prefill(d["q"], d["k"], d["v"], d["log_alpha"], d["beta"], d["initial_state"], d["out"], d["final_state"])
        assert gdn.gdn_launch_count() - n0 == launches
        assert gdn.gdn_query_status_stream() == 0
    finally:
        gdn.gdn_set_workspace(None)
    o, fin = run_oracle(x)
    assert_close(f64(d["out"]), o, BF16_REL_L2, BF16_MAX_ABS, "out")
    assert_close(f64(d["final_state"]), fin, BF16_REL_L2, BF16_MAX_ABS, "final_state")


# fp32: clusters of eight CTAs up to 60 chains of this size, of four from 61 to 66, of eight again from 67 (rounds on 148 SMs)
@pytest.mark.parametrize("B,H", [(4, 15), (1, 61), (2, 33), (1, 67)])
def test_fp32_clusters_on_both_sides_of_the_line(B, H):
    x = make_inputs(get_config("tiny", B=B, T=64 * 9 + 5, H=H, init_std=0.1, seed=82))
    d = to_device(x)
    out, fin = run_lib(gdn.gdn_chunk_prefill_f32, d)
    o, f = run_oracle(x)
    assert_close(f64(out), o, F32_REL_L2, None, "out")
    assert_close(f64(fin), f, F32_REL_L2, None, "final_state")


# decode: slices of 32 value columns while the slices of 128 are no more than the SMs
@pytest.mark.parametrize("blocks,d_v", [(0, 128), (1, 128), (0, 256), (2, 256)])
def test_decode_on_both_sides_of_the_line(blocks, d_v):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    H = sms * 128 // d_v + blocks * 128 // d_v
    x = make_inputs(get_config("long", B=1, T=1, H=H, d_v=d_v, init_std=0.5, seed=83))
    d = to_device(x)
    state, out = d["initial_state"].clone(), d["out"][:, 0].contiguous()
    gdn.gdn_decode_step(*(d[n][:, 0].contiguous() for n in ("q", "k", "v", "log_alpha", "beta")), state, out)
    torch.cuda.synchronize()
    o, s = oracle.sequential(widen(x.q), widen(x.k), widen(x.v), x.log_alpha, x.beta, x.initial_state)
    assert_close(f64(out), o[:, 0], BF16_REL_L2, BF16_MAX_ABS, "out")      # one rounding of the output to bf16
    assert_close(f64(state), s, F32_REL_L2, None, "state")
