"""What users of this library have it do, as timed cases.

A case is one call pattern of a serving or analysis program on top of the public entry points of
`paper_2511_05534_b200.binding` (and `shard`), at sizes of `configs.WORKLOADS` or of the same ranges:

  compress    flowmm_compress_layer right after prefill: one layer at a time as a model's layers finish, or a stack of
              layers in one call
  shard       the same compression on one tensor-parallel rank's KV heads, through the step entry points
  decode      flowmm_decode_attention, one new token per sequence, over a compressed or a full cache
  recompress  flowmm_recompress on a compressed cache that grew while decoding
  flow        flowmm_full_flow, the information-flow statistic over a whole prefill

`prepare` holds what such a program keeps across calls: the tensors, the parameter object, the workspace and the
output tensors.  Inputs are those of `inputs.make_stack_device` (seeded, modality-structured stand-ins for a prefill)."""
import dataclasses
import math

import torch

from paper_2511_05534_b200 import binding as F
from paper_2511_05534_b200 import configs, inputs, shard

DEV = "cuda"


def listed():
    return [
        # the smallest thing anyone compresses: one fp32 layer, four heads of 64, 192 tokens
        dict(name="layer_fp32_small", kind="compress", like="cfg1", layers=1, seqs=1, text0=8, visual=144, text1=40, permille=250),
        # one layer of a LLaVA-1.5-7B-shaped model, called as soon as that layer's prefill is done
        dict(name="layer_mha_image", kind="compress", like="cfg2", layers=1, seqs=1, text0=16, visual=576, text1=48, permille=100),
        # all of its layers in one call
        dict(name="stack_mha_image", kind="compress", like="cfg2", layers=32, seqs=1, text0=16, visual=576, text1=48, permille=100),
        # one layer of a Qwen2-VL-7B-shaped model, two sequences, dynamic-resolution image: ragged token count
        dict(name="layer_gqa_ragged", kind="compress", like="cfg3", layers=1, seqs=2, text0=27, visual=1369, text1=75, permille=100),
        # the whole stack on one image of 2048 tokens
        dict(name="stack_gqa_image", kind="compress", like="cfg3", layers=28, seqs=1, text0=32, visual=2048, text1=96, permille=100),
        # the whole stack on eight interleaved video frames, generous budget
        dict(name="stack_gqa_video", kind="compress", like="cfg4", layers=28, seqs=1, text0=0, visual=1024, text1=32, permille=200),
        # long context, four sequences, four layers per call: the large end of the range
        dict(name="layers_long", kind="compress", like="cfg5", layers=4, seqs=4, text0=128, visual=32768, text1=896, permille=50),
        # one of eight tensor-parallel ranks: its own KV head of two long-context layers, four sequences
        dict(name="rank_long", kind="shard", like="cfg5", layers=2, seqs=4, text0=128, visual=32768, text1=896, permille=50),
        # a decode step of one layer over its compressed cache, a single sequence
        dict(name="decode_layer_compressed", kind="decode", like="cfg3", layers=1, seqs=1, keys=218),
        # ... and of a batch of four sequences over a full long-context cache
        dict(name="decode_layer_full", kind="decode", like="cfg5", layers=1, seqs=4, keys=33792),
        # a stack's compressed caches after 217 decoded tokens, compressed back to their budget
        dict(name="recompress_stack", kind="recompress", like="cfg4", layers=28, seqs=1, kept=423, added=217),
        # information flow of every layer over the whole prefill of a one-image prompt
        dict(name="flow_stack", kind="flow", like="cfg3", layers=28, seqs=1, text0=32, visual=2048, text1=96),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


# Bounds of a drawn case, just below the largest listed one: cache rows in a call, (row, pivot) pairs, and multiply-adds of
# the full-prefill flow.
MAX_ROWS = 15 * 8 * 33792
MAX_PAIRS = MAX_ROWS * 1690
MAX_FLOW = 28 * 28 * 2176 * 2304


def draw(rng):
    kind = rng.choice(["compress"] * 9 + ["decode"] * 4 + ["recompress"] * 2 + ["flow"] * 2 + ["shard"])
    if kind == "compress" and rng.random() < 0.12:               # small fp32 layers with heads of 64
        L = _log_int(rng, 96, 1024)
        t0, t1 = rng.randint(4, 16), rng.randint(20, 48)
        return dict(kind=kind, like="cfg1", layers=1, seqs=rng.randint(1, 4), text0=t0, visual=max(16, L - t0 - t1), text1=t1,
                    permille=rng.choice([100, 200, 250]))
    like = rng.choice(["cfg2", "cfg3", "cfg4", "cfg5"])
    wl = configs.get(like)
    seqs = rng.choice([1, 1, 2, 3, 4])
    layers = rng.choice([1, 1, 2, _log_int(rng, 3, wl.n_layers)])
    permille = rng.choice([50, 100, 200]) if like != "cfg5" else 50
    if kind in ("compress", "shard"):
        heads = 1 if kind == "shard" else wl.n_kv_heads
        if kind == "shard":
            like, wl, heads, permille = "cfg5", configs.get("cfg5"), 1, 50
        lo, hi = {"cfg2": (200, 3000), "cfg3": (400, 8000), "cfg4": (1500, 16000), "cfg5": (6000, 33792)}[like]
        L = _log_int(rng, lo, hi)
        t0 = 0 if wl.ar1_frames else rng.randint(8, 128)
        t1 = rng.randint(17, 64) if wl.ar1_frames else rng.randint(48, 160)
        n = max(1, wl.ar1_frames)
        visual = max(64, L // n - t1 if wl.ar1_frames else L - t0 - t1)
        L = t0 + n * (visual + t1) if wl.ar1_frames else t0 + visual + t1
        per_seq = heads * L * max(1.0, L * permille / 1000 * MAX_ROWS / MAX_PAIRS)
        layers = max(1, min(layers, int(MAX_ROWS / (seqs * per_seq))))
        return dict(kind=kind, like=like, layers=layers, seqs=seqs, text0=t0, visual=visual, text1=t1, permille=permille)
    if kind == "decode":
        keys = _log_int(rng, 32, 33792)
        layers = max(1, min(layers, MAX_ROWS // (seqs * wl.n_kv_heads * keys)))
        return dict(kind=kind, like=like, layers=layers, seqs=seqs, keys=keys)
    if kind == "recompress":
        kept = _log_int(rng, 64, 1690)
        added = max(wl.window, int(kept * rng.uniform(0.2, 1.0)))
        layers = max(1, min(layers, 900 // (seqs * wl.n_kv_heads)))
        return dict(kind=kind, like=like, layers=layers, seqs=seqs, kept=kept, added=added)
    t0, t1 = rng.randint(8, 64), rng.randint(48, 160)
    L = _log_int(rng, 256, 4096)
    visual = max(64, L - t0 - t1)
    L = t0 + visual + t1
    layers = max(1, min(layers, int(MAX_FLOW / (seqs * wl.n_q_heads * L * (L + 128)))))
    return dict(kind=kind, like="cfg3" if wl.ar1_frames else like, layers=layers, seqs=seqs, text0=t0, visual=visual, text1=t1)


def _workload(case):
    """The configuration that the case is like, with the case's own prompt."""
    wl = configs.get(case["like"])
    if "visual" not in case:
        return wl
    if wl.ar1_frames:
        segs = ((configs.VISUAL, case["visual"]), (configs.TEXT, case["text1"])) * wl.ar1_frames
    else:
        segs = ((configs.TEXT, case["text0"]), (configs.VISUAL, case["visual"]), (configs.TEXT, case["text1"]))
    if case["kind"] == "shard":                                  # one KV head of eight, with its query heads
        wl = dataclasses.replace(wl, n_q_heads=wl.group, n_kv_heads=1)
    return dataclasses.replace(wl, segments=segs)


def _units(wl, case):
    """The case's layers spread over the depth of the stack, every sequence of each."""
    step = wl.n_layers / case["layers"]
    return [(int((i + 0.5) * step), s) for i in range(case["layers"]) for s in range(case["seqs"])]


def _params(wl, U, L, B):
    return F.Params(U, wl.n_q_heads, wl.n_kv_heads, wl.head_dim, L, wl.window, B,
                    dtype=F.BF16 if wl.dtype == "bf16" else F.F32, theta=wl.theta, tau=wl.tau_rel, tau_mode=F.TAU_REL)


def _cache(gen, wl, U, n, vis):
    """Key and value rows of a cache; vis [U, Hkv, n]: rows that stand for visual tokens."""
    out = []
    for _ in range(2):
        z = torch.randn((U, wl.n_kv_heads, n, wl.head_dim), generator=gen, device=DEV, dtype=torch.bfloat16)
        out.append(torch.where(vis.unsqueeze(-1), 0.5 + 1.5 * z, z))
    return out


def prepare(case, seed):
    wl = dataclasses.replace(_workload(case), seed=seed % 2003)
    units = _units(wl, case)
    U, Hq, Hkv, D = len(units), wl.n_q_heads, wl.n_kv_heads, wl.head_dim
    kind = case["kind"]
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    s = dict(kind=kind)

    def new(*shape, dtype=torch.float32):
        return torch.zeros(shape, dtype=dtype, device=DEV)

    if kind == "decode":
        n = case["keys"]
        s["q"] = torch.randn((U, Hq, D), generator=gen, device=DEV, dtype=torch.bfloat16)
        s["k"], s["v"] = _cache(gen, wl, U, n, (torch.rand((U, Hkv, n), generator=gen, device=DEV) < 0.9))
        s["out"] = new(U, Hq, D)
        s["ws"] = new(F.flowmm_decode_workspace_bytes(s["q"], s["k"], s["v"]), dtype=torch.uint8)
        return s
    if kind == "recompress":
        n, B = case["kept"] + case["added"], case["kept"]
        vis = torch.rand((U, Hkv, n), generator=gen, device=DEV) < 0.8
        vis[:, :, B:] = False                                    # decoded tokens are text
        s["k"], s["v"] = _cache(gen, wl, U, n, vis)
        s["q"] = torch.randn((U, Hq, wl.window, D), generator=gen, device=DEV, dtype=torch.bfloat16)
        s["m"] = vis.to(torch.uint8)
        s["p"] = p = _params(wl, U, n, B)
        s["k_out"], s["v_out"] = new(U, Hkv, B, D, dtype=torch.bfloat16), new(U, Hkv, B, D, dtype=torch.bfloat16)
        s["m_out"] = new(U, Hkv, B, dtype=torch.uint8)
        s["rho"], s["strategy"] = new(U), new(U, dtype=torch.int32)
        s["ws"] = new(F.flowmm_recompress_workspace_bytes(p), dtype=torch.uint8)
        return s
    q, k, v, m = inputs.make_stack_device(wl, DEV, units)
    s["k"], s["m"] = k, m
    L = wl.seq_len
    s["rho"], s["strategy"] = new(U), new(U, dtype=torch.int32)
    if kind == "flow":
        s["q"] = torch.randn((U, Hq, L, D), generator=gen, device=DEV, dtype=torch.bfloat16)
        s["p"] = p = _params(dataclasses.replace(wl, window=1), U, L, 1)
        s["cross"] = new(U, Hq)
        s["ws"] = new(F.flowmm_full_flow_workspace_bytes(p), dtype=torch.uint8)
        return s
    s["q"], s["v"] = q, v
    B = wl.n_keep(case["permille"])
    s["p"] = p = _params(wl, U, L, B)
    s["k_out"], s["v_out"] = new(U, Hkv, B, D, dtype=k.dtype), new(U, Hkv, B, D, dtype=k.dtype)
    s["retained"] = new(U, Hkv, B, dtype=torch.int32)
    s["ws"] = F.alloc_workspace(p)
    if kind == "shard":
        s["outs"] = dict(importance=new(U, Hkv, L), cross_mass=new(U, Hq), rho=s["rho"], strategy=s["strategy"],
                         rho_local=new(U), strategy_local=new(U, dtype=torch.int32), retained=s["retained"],
                         evicted=new(U, Hkv, L - B, dtype=torch.int32), match=new(U, Hkv, L - B, dtype=torch.int32),
                         match_sim=new(U, Hkv, L - B), k_out=s["k_out"], v_out=s["v_out"])
    return s


def run(s):
    kind = s["kind"]
    if kind == "compress":               # the compressed cache, and the positions and strategy that a program keeps with it
        F.flowmm_compress_layer(s["p"], s["q"], s["k"], s["v"], s["m"], s["k_out"], s["v_out"], s["ws"], rho=s["rho"],
                                strategy=s["strategy"], retained_idx=s["retained"])
        return s["k_out"], s["v_out"], s["rho"], s["strategy"], s["retained"]
    if kind == "shard":
        o = shard.compress_layer_head_sharded(s["p"], s["q"], s["k"], s["v"], s["m"], s["outs"], s["ws"])
        return [o[key] for key in ("k_out", "v_out", "importance", "rho", "strategy", "retained", "evicted", "match", "match_sim")]
    if kind == "decode":
        F.flowmm_decode_attention(s["q"], s["k"], s["v"], s["out"], s["ws"])
        return s["out"]
    if kind == "recompress":
        F.flowmm_recompress(s["p"], s["q"], s["k"], s["v"], s["m"], s["k_out"], s["v_out"], s["m_out"], s["ws"],
                            rho=s["rho"], strategy=s["strategy"])
        return s["k_out"], s["v_out"], s["m_out"], s["rho"], s["strategy"]
    F.flowmm_full_flow(s["p"], s["q"], s["k"], s["m"], s["cross"], s["rho"], s["strategy"], s["ws"])
    return s["cross"], s["rho"], s["strategy"]


def work(case):
    """Inputs once, outputs once.  Of the matching step's (non-pivot, pivot) pairs about half pass the gates of Eq. 10
    under the configurations' thresholds; they alone are counted."""
    wl = _workload(case)
    U, Hq, Hkv, D, W = case["layers"] * case["seqs"], wl.n_q_heads, wl.n_kv_heads, wl.head_dim, wl.window
    e = 2 if wl.dtype == "bf16" else 4
    if case["kind"] == "decode":
        n = case["keys"]
        return {"bytes": U * (2 * Hkv * n * D * e + Hq * D * (e + 4)), "flops": 4 * U * Hq * n * D}
    if case["kind"] == "flow":
        L = wl.seq_len
        return {"bytes": U * ((Hq + Hkv) * L * D * e + L + Hq * 4), "flops": U * Hq * L * (L + 1) * D}
    if case["kind"] == "recompress":
        L, B = case["kept"] + case["added"], case["kept"]
    else:
        L, B = wl.seq_len, wl.n_keep(case["permille"])
    return {"bytes": U * (Hq * W * D * e + 2 * Hkv * (L + B) * D * e + L + Hkv * B * 4),
            "flops": U * (2 * Hq * W * L * D + Hkv * (L - B) * B * D + 4 * Hkv * L * D)}


def tolerance(case):
    if case["kind"] in ("decode", "flow"):                       # fp32 results of bf16 inputs, fp32 accumulation
        return {"rel": 1e-5}
    if configs.get(case["like"]).dtype == "f32":
        return {"rel": 1e-5, "differ": 1e-3}
    return {"rel": 1e-2, "differ": 2e-3}                         # the merged cache is rounded to bf16
