"""The work a user of this library has it do, as cases that can be timed and compared.

Every case goes through the public Python entry points of ``paper_2607_14568_b200`` with caller-owned
buffers, and with the scratch of ``gdn_set_workspace`` in place for the bf16 prefill, which is how a serving
process runs them.  Kinds:

  prefill    gdn_chunk_prefill on equal-length ([B, T, H, .]) or packed ([T, H, .] with cu_seqlens) bf16 input;
             entry "raw" is the call with the norms and gates fused in front of it, "gated" the one with the gated
             norm fused behind it
  f32        gdn_chunk_prefill_f32, the same operation in fp32 throughout
  decode     gdn_decode_step, one token per sequence, the fp32 state updated in place
  attention  gdn_attn_causal_prefill of the softmax layers, equal-length or packed

Inputs are random with the distributions of ``workloads/``: q, k normalised per head, v ~ N(0, 1),
beta = sigmoid(N(0, 1)), log_alpha = -softplus(N(0, 1)) * scale, initial state ~ N(0, 0.02^2).
"""
import math

import torch

import paper_2607_14568_b200 as gdn

CHUNK = 64


def listed():
    return [
        # one user generating: a single sequence's token through one layer (latency of the call is all there is)
        {"name": "decode_1", "kind": "decode", "B": 1, "H": 16, "dk": 128, "dv": 128},
        # a full decode batch: one state read and one state write per sequence and head
        {"name": "decode_256", "kind": "decode", "B": 256, "H": 16, "dk": 128, "dv": 128},
        # the smallest configuration of the benchmark: fp32, narrow heads, a short prompt
        {"name": "tiny_f32", "kind": "f32", "B": 1, "T": 256, "H": 2, "dk": 64, "dv": 64, "scale": 0.1, "s0": False},
        # the 2k-token prompt in fp32, for users who want the precision of the paper
        {"name": "short_f32", "kind": "f32", "B": 1, "T": 2048, "H": 16, "dk": 128, "dv": 128, "scale": 0.05, "s0": False},
        # the 2k-token prompt
        {"name": "short", "kind": "prefill", "entry": "plain", "B": 1, "T": 2048, "H": 16, "dk": 128, "dv": 128, "scale": 0.05, "s0": False},
        # the 10k-token prompt, continued from a state (the configuration the benchmark's headline names)
        {"name": "long", "kind": "prefill", "entry": "plain", "B": 1, "T": 10240, "H": 16, "dk": 128, "dv": 128, "scale": 0.05, "s0": True},
        # a step of continuous batching: a few short prompts of any length packed together, straight from the projections
        {"name": "prompts_raw", "kind": "prefill", "entry": "raw", "lengths": "517,83,1,260,731,64,129", "H": 16, "dk": 128, "dv": 128,
         "scale": 0.05, "s0": True},
        # batched serving: eight prompts of 512 to 8192 tokens packed together
        {"name": "serving", "kind": "prefill", "entry": "plain", "lengths": "6049,1293,7880,3347,590,2715,4411,915", "H": 16, "dk": 128, "dv": 128,
         "scale": 0.05, "s0": True},
        # a small batch of equal, ragged-tailed prompts through the call that also does the output norm and gate
        {"name": "batch_gated", "kind": "prefill", "entry": "gated", "B": 4, "T": 1500, "H": 16, "dk": 128, "dv": 128, "scale": 0.05, "s0": False},
        # the largest configuration of the benchmark: a batch of long documents, wide value heads
        {"name": "large", "kind": "prefill", "entry": "plain", "B": 4, "T": 32768, "H": 32, "dk": 128, "dv": 256, "scale": 0.02, "s0": False},
        # the softmax layers of the same model on the 10k-token prompt
        {"name": "attn_10k", "kind": "attention", "B": 1, "T": 10240, "Hq": 16, "Hkv": 8, "d": 128},
        # the softmax layers on a few packed prompts of any length
        {"name": "attn_packed", "kind": "attention", "lengths": "1711,402,2048,65,977", "Hq": 16, "Hkv": 8, "d": 128},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _lengths(rng, n, lo, hi):
    return ",".join(str(_log(rng, lo, hi)) for _ in range(n))


def draw(rng):
    kind = rng.choice(["decode", "f32", "prefill", "prefill", "prefill", "packed", "packed", "attention"])
    if kind == "decode":
        return {"kind": "decode", "B": _log(rng, 1, 256), "H": rng.choice([8, 12, 16, 24, 32]), "dk": 128, "dv": rng.choice([128, 128, 256])}
    if kind == "f32":
        d = rng.choice([64, 96, 128, 128])
        return {"kind": "f32", "B": 1, "T": _log(rng, 32, 2048), "H": rng.choice([2, 4, 8, 16]), "dk": d, "dv": d,
                "scale": 0.05, "s0": rng.random() < 0.5}
    if kind == "attention":
        hq, hkv = rng.choice([(16, 8), (16, 4), (16, 2), (32, 8), (8, 8)])
        if rng.random() < 0.5:
            return {"kind": "attention", "B": 1, "T": _log(rng, 64, 10240), "Hq": hq, "Hkv": hkv, "d": 128}
        return {"kind": "attention", "lengths": _lengths(rng, rng.randint(2, 8), 32, 4096), "Hq": hq, "Hkv": hkv, "d": 128}
    entry = rng.choice(["plain", "plain", "raw", "gated"])
    H, dv = rng.choice([8, 12, 16, 24, 32]), 128 if entry == "gated" else rng.choice([128, 128, 256])
    case = {"kind": "prefill", "entry": entry, "H": H, "dk": 128, "dv": dv, "scale": rng.choice([0.02, 0.05, 0.1]), "s0": rng.random() < 0.5}
    if kind == "packed":
        return dict(case, lengths=_lengths(rng, rng.randint(2, 12), 32, 8192))
    return dict(case, B=rng.choice([1, 1, 1, 2, 3, 4]), T=_log(rng, 64, 32768))


def _lens(case):
    if "lengths" in case:
        return [int(x) for x in case["lengths"].split(",")]
    return [case["T"]] * case["B"]


_scratch = None


def _workspace(nbytes):
    """One scratch buffer for the process, as large as its largest call needs."""
    global _scratch
    if _scratch is None or _scratch.numel() < nbytes:
        _scratch = None
        gdn.gdn_set_workspace(None)
        _scratch = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
        gdn.gdn_set_workspace(_scratch)


def _unit(x):
    return x.div_(x.square().sum(-1, keepdim=True).sqrt_())


def prepare(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)

    def normal(*shape):
        return torch.randn(*shape, device="cuda", generator=g)

    kind, bf16 = case["kind"], torch.bfloat16
    if kind == "decode":
        lead, H, dk, dv = (case["B"], case["H"]), case["H"], case["dk"], case["dv"]
        s = {"q": _unit(normal(*lead, dk)).to(bf16), "k": _unit(normal(*lead, dk)).to(bf16), "v": normal(*lead, dv).to(bf16),
             "log_alpha": -torch.nn.functional.softplus(normal(*lead)) * 0.05, "beta": torch.sigmoid(normal(*lead)),
             "state": normal(*lead, dk, dv) * 0.1}
        s["out"] = torch.empty_like(s["v"])
        return case, s
    lens = _lens(case)
    packed = "lengths" in case
    lead = (sum(lens),) if packed else (case["B"], case["T"])
    cu = None
    if packed:
        cu = torch.tensor([0] + lens).cumsum(0).to(device="cuda", dtype=torch.int32)
    if kind == "attention":
        q, k, v = (normal(*lead, h, case["d"]).to(bf16) for h in (case["Hq"], case["Hkv"], case["Hkv"]))
        return case, {"q": q, "k": k, "v": v, "out": torch.empty_like(q), "cu": cu}
    H, dk, dv = case["H"], case["dk"], case["dv"]
    io = torch.float32 if kind == "f32" else bf16
    raw = case.get("entry") == "raw"
    if raw:    # projections as they come: any magnitude per token and head
        q, k = ((normal(*lead, H, dk) * (0.5 * normal(*lead, H, 1)).exp_()).to(io) for _ in range(2))
        a, b = normal(*lead, H), normal(*lead, H)
    else:
        q, k = (_unit(normal(*lead, H, dk)).to(io) for _ in range(2))
        a, b = -torch.nn.functional.softplus(normal(*lead, H)) * case["scale"], torch.sigmoid(normal(*lead, H))
    v = normal(*lead, H, dv).to(io)
    s = {"q": q, "k": k, "v": v, "a": a, "b": b, "s0": normal(len(lens), H, dk, dv) * 0.02 if case["s0"] else None,
         "out": torch.empty_like(v), "final": torch.empty(len(lens), H, dk, dv, device="cuda"), "cu": cu}
    if case.get("entry") == "gated":
        s["z"], s["w"] = normal(*lead, H, dv).to(bf16), 1 + 0.1 * normal(dv)
    if kind == "prefill":
        _workspace(gdn.gdn_workspace_bytes(len(lens), lead[0] if packed else case["T"], H, dk, dv, packed))
    return case, s


def run(state):
    case, s = state
    kind = case["kind"]
    if kind == "decode":
        out, st = gdn.gdn_decode_step(s["q"], s["k"], s["v"], s["log_alpha"], s["beta"], s["state"], s["out"])
        return {"out": out, "state": st}
    if kind == "attention":
        return gdn.gdn_attn_causal_prefill(s["q"], s["k"], s["v"], s["out"], cu_seqlens=s["cu"])
    if kind == "f32":
        out, final = gdn.gdn_chunk_prefill_f32(s["q"], s["k"], s["v"], s["a"], s["b"], s["s0"], s["out"], s["final"], s["cu"])
    elif case["entry"] == "raw":
        out, final = gdn.gdn_chunk_prefill_raw(s["q"], s["k"], s["v"], s["a"], s["b"], case["scale"], 1e-6, s["s0"], s["out"], s["final"], s["cu"])
    elif case["entry"] == "gated":
        out, final = gdn.gdn_chunk_prefill_gated(s["q"], s["k"], s["v"], s["a"], s["b"], s["s0"], s["z"], s["w"], 1e-6, s["out"], s["final"], s["cu"])
    else:
        out, final = gdn.gdn_chunk_prefill(s["q"], s["k"], s["v"], s["a"], s["b"], s["s0"], s["out"], s["final"], s["cu"])
    return {"out": out, "final": final}


def work(case):
    kind = case["kind"]
    if kind == "decode":
        n, dk, dv = case["B"] * case["H"], case["dk"], case["dv"]
        return {"bytes": n * (8 * dk * dv + 4 * (dk + dv) + 8), "flops": n * 7 * dk * dv}
    lens = _lens(case)
    tokens = sum(lens)
    if kind == "attention":   # every visible (query, key) pair: one product with K, one with V
        pairs = sum(n * (n + 1) // 2 for n in lens)
        return {"bytes": tokens * case["d"] * 4 * (case["Hq"] + case["Hkv"]), "flops": pairs * case["Hq"] * 4 * case["d"]}
    H, dk, dv = case["H"], case["dk"], case["dv"]
    e = 4 if kind == "f32" else 2
    per_token = (2 * dk + 2 * dv) * e + 8 + (dv * e if case.get("entry") == "gated" else 0)
    states = len(lens) * H * 4 * dk * dv * (2 if case["s0"] else 1)
    # the chunked form with its 64-token chunk: KK^T, QK^T, W, U, then W S, Q S, P v and the state update
    return {"bytes": tokens * H * per_token + states, "flops": tokens * H * (6 * CHUNK * dk + 4 * CHUNK * dv + 6 * dk * dv)}


def tolerance(case):
    kind = case["kind"]
    if kind == "f32":
        return {"rel": 1e-5, "max": 1e-3}
    if kind == "decode":     # fp32 inside; a last bit of the bf16 output may round the other way
        return {"rel": 1e-3, "max": 1e-2}
    return {"rel": 8e-3, "max": 0.1}   # bf16 operands, fp32 accumulation
