"""The work this framework is timed on: packed variable-length attention through its public calls.

A case is one batch and one entry point.  The batch is described by plain values (how the sequence lengths
are spread, tokens, heads, head size, largest context-parallel degree); its lengths, degrees and spans follow
from these values alone, its tensors from the seed.  `listed()` names the batches that stand for the range,
`draw()` gives further ones of the same range.

Entry points (what one pass calls):
  step       fcp_attn_fwd_fused + fcp_attn_bwd on an uploaded plan: one attention layer of a training step
  forward    fcp_attn_fwd_fused alone: evaluation, or the recomputation under activation checkpointing
  partial    fcp_attn_fwd_merged: the forward pass that goes through the per-rank partial outputs
  heads      one KV-head group of a larger model: the fused forward of its query heads + fcp_attn_bwd_heads
  host       fcp_attn_fwd_bwd_host: forward and backward on pinned host buffers
  new_batch  fcp_plan_strategy + plan + upload + forward + backward: what the first layer of every new batch pays
"""
import math

import numpy as np
import torch

from paper_2602_21788_b200 import costfit, fcp

# compute terms as fitted on this GPU (ms); ring: 4096 bytes of K/V per token over a 25 GB/s link (bytes per ms)
COST = dict(costfit.B200_COEFFS, alpha3=4096.0, beta2=0.05, v=25e6)


def _case(name, entry, mix, tokens, hq, hkv, head_dim, max_degree=8, rank_tokens=4096, layout=0, **mix_args):
    """`rank_tokens`: tokens that one virtual rank holds; degree = ceil(length / rank_tokens), capped."""
    return dict(name=name, entry=entry, mix=mix, tokens=tokens, hq=hq, hkv=hkv, head_dim=head_dim,
                max_degree=max_degree, rank_tokens=rank_tokens, layout=layout, **mix_args)


def listed():
    return [
        # the smallest batch in use: eight short sequences of a small model; launches and host time decide
        _case("tiny_4k_d64_step", "step", "uniform", 4353, 4, 4, 64, max_degree=3, rank_tokens=352, layout=1,
              lo=64, hi=1024),
        # one packed micro-batch of instruction-tuning data on a Llama-3-8B attention layer (32/8 heads)
        _case("short_8k_step", "step", "lognormal", 8192, 32, 8, 128, median=512, cap=4096),
        # a layer of a small model (head size 64, three query heads per KV head), lengths odd, nothing aligned
        _case("ragged_16k_d64_step", "step", "uniform", 16411, 12, 4, 64, max_degree=5, rank_tokens=640, layout=4,
              lo=1, hi=3001),
        # a new batch arrives: strategy search, block plan, upload, then the first layer
        _case("new_batch_16k", "new_batch", "lognormal", 16384, 32, 8, 128, layout=7, median=1024, cap=8192),
        # the ordinary training batch: 64K tokens, log-normal lengths, Llama-3-8B layer
        _case("llama8b_64k_step", "step", "lognormal", 65536, 32, 8, 128, layout=7, median=2048, cap=32768),
        # the same batch in evaluation
        _case("llama8b_64k_forward", "forward", "lognormal", 65536, 32, 8, 128, layout=7, median=2048, cap=32768),
        # the same batch through the partial outputs of every virtual rank and their merge
        _case("llama8b_64k_partial", "partial", "lognormal", 65536, 32, 8, 128, layout=7, median=2048, cap=32768),
        # tensors in host memory: copies over PCIe around the same kernels
        _case("llama8b_32k_host", "host", "lognormal", 32768, 32, 8, 128, layout=7, median=2048, cap=16384),
        # text next to image/video-heavy sequences, no grouped KV heads
        _case("bimodal_128k_step", "step", "bimodal", 131072, 32, 32, 128, max_degree=6, layout=7,
              lo=512, hi=2048, long_lo=16384, long_hi=65536),
        # the same with bidirectional image spans in the long sequences
        _case("bimodal_128k_spans_step", "step", "bimodal", 131072, 32, 32, 128, max_degree=6, layout=7,
              lo=512, hi=2048, long_lo=16384, long_hi=65536, spans=True),
        # one 128K-token document among short ones
        _case("longtail_256k_step", "step", "longtail", 262144, 40, 8, 128, max_degree=7,
              long=131072, lo=256, hi=4096),
        # one 384K-token document: one KV head of a 64/8-head layer (the layer is eight such passes)
        _case("extreme_512k_heads", "heads", "zipf", 524288, 8, 1, 128, max_degree=7,
              long=393216, lo=128, hi=8192),
    ]


def draw(rng):
    """One more case of the ranges above."""
    def log_int(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    layout = rng.randrange(1, 1 << 30)
    shapes = [(4, 4, 64), (12, 4, 64), (16, 2, 64), (8, 8, 128), (32, 8, 128), (28, 4, 128), (40, 8, 128), (32, 32, 128)]
    hq, hkv, head_dim = rng.choice(shapes)
    entry = rng.choice(["step", "step", "step", "forward", "partial", "heads", "host", "new_batch"])
    mix = rng.choice(["uniform", "lognormal", "bimodal", "longtail"])
    if entry in ("host", "new_batch"):
        mix = rng.choice(["uniform", "lognormal"])
        tokens = log_int(2048, 32768)
    elif mix == "longtail":
        tokens = log_int(32768, 262144)
    elif mix == "bimodal":
        tokens = log_int(16384, 131072)
    else:
        tokens = log_int(2048, 65536)
    if entry == "partial":
        tokens = min(tokens, 65537)        # the partial outputs of every rank are held at once
    if entry == "heads":
        g = hq // hkv
        hq, hkv = g, 1
        tokens = log_int(32768, 393216)
        mix = "longtail"
    max_degree = rng.choice([3, 5, 6, 7, 8])
    common = dict(max_degree=max_degree, rank_tokens=rng.choice([512, 2048, 4096]), layout=layout)
    if mix == "uniform":
        hi = log_int(64, 8192)
        args = dict(lo=max(1, hi // rng.choice([2, 8, 64])), hi=hi)
    elif mix == "lognormal":
        args = dict(median=log_int(256, 4096), cap=log_int(4096, 32768))
    elif mix == "bimodal":
        long_hi = max(4096, tokens // 2)
        args = dict(lo=512, hi=2048, long_lo=long_hi // 4, long_hi=long_hi)
        if entry in ("step", "forward", "heads"):
            args["spans"] = rng.random() < 0.5
    else:
        args = dict(long=int(tokens * rng.uniform(0.3, 0.75)), lo=128, hi=4096)
    case = _case("", entry, mix, tokens, hq, hkv, head_dim, **common, **args)
    del case["name"]
    return case


# ---------------------------------------------------------------------------------------------------------
def batch(case):
    """Sequence lengths, degrees and bidirectional spans (or None) of a case."""
    rng = np.random.Generator(np.random.PCG64([case["layout"], 0xBA7C]))
    mix, total = case["mix"], case["tokens"]
    lens = []
    if mix in ("longtail", "zipf"):
        lens.append(case["long"])
    if mix == "zipf":
        support = np.arange(case["lo"], case["hi"] + 1, dtype=np.float64)
        cdf = np.cumsum(support ** -1.2)
        cdf /= cdf[-1]
    remaining = total - sum(lens)
    while remaining > 0:
        if mix == "lognormal":
            n = int(np.clip(round(float(rng.lognormal(math.log(case["median"]), 1.0))), 128, case["cap"]))
        elif mix == "bimodal" and len(lens) % 2 == 1:
            n = int(rng.integers(case["long_lo"], case["long_hi"] + 1))
        elif mix == "zipf":
            n = int(support[min(int(np.searchsorted(cdf, rng.random())), len(support) - 1)])
        else:
            n = int(rng.integers(case["lo"], case["hi"] + 1))
        n = min(n, remaining)
        lens.append(n)
        remaining -= n
    lens = np.asarray(lens, dtype=np.int32)
    degrees = np.minimum(case["max_degree"], -(-lens // case["rank_tokens"])).astype(np.int32)
    if not case.get("spans"):
        return lens, degrees, None
    spans = []
    for length in lens:
        sp, pos = [], 0
        while length >= 4096:      # long sequences: text runs between image spans
            pos += int(rng.integers(64, 513))
            m = int(rng.integers(256, 2049))
            if pos + m > length:
                break
            sp.append((pos, pos + m))
            pos += m
        spans.append(sp)
    return lens, degrees, spans


def prepare(case, seed):
    lens, degrees, spans = batch(case)
    hq, hkv, head_dim, tokens = case["hq"], case["hkv"], case["head_dim"], case["tokens"]
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    st = dict(case=case, lens=lens, degrees=degrees, plan=None)

    def normal(heads):         # attention inputs after normalisation and projection: about N(0, 1), bf16
        return torch.randn((tokens, heads, head_dim), dtype=torch.bfloat16, device="cuda", generator=gen)

    def empty(heads):
        return torch.empty((tokens, heads, head_dim), dtype=torch.bfloat16, device="cuda")

    st.update(q=normal(hq), k=normal(hkv), v=normal(hkv))
    st.update(o=empty(hq), lse=torch.empty((tokens, hq), dtype=torch.float32, device="cuda"))
    backward = case["entry"] not in ("forward", "partial")
    if backward:
        st.update(do=normal(hq), dq=empty(hq), dk=empty(hkv), dv=empty(hkv))
    if case["entry"] == "new_batch":
        return st
    plan = fcp.Plan(lens, degrees, hq, hkv, head_dim, spans=spans).upload()
    st["plan"] = plan
    if case["entry"] == "host":
        for name in ("q", "k", "v", "do"):
            st[name] = st[name].cpu().pin_memory()
        for name in ("o", "lse", "dq", "dk", "dv"):
            st[name] = torch.empty(st[name].shape, dtype=st[name].dtype, pin_memory=True)
        st["workspace_bytes"] = plan.host_workspace_bytes()
        st["workspace"] = torch.empty(st["workspace_bytes"], dtype=torch.uint8, device="cuda")
    elif case["entry"] == "partial":
        o_bytes, lse_bytes, _ = plan.workspace_bytes(hq)
        st["o_part"] = torch.empty(o_bytes // 4, dtype=torch.float32, device="cuda")
        st["lse_part"] = torch.empty(lse_bytes // 4, dtype=torch.float32, device="cuda")
    elif backward:
        st["scratch_bytes"] = plan.bwd_scratch_bytes(hkv)
        st["scratch"] = torch.empty(st["scratch_bytes"], dtype=torch.uint8, device="cuda")
    return st


def run(st):
    case, plan, entry = st["case"], st["plan"], st["case"]["entry"]
    stream = torch.cuda.current_stream().cuda_stream
    if entry == "host":
        fcp.fcp_attn_fwd_bwd_host(plan, st["q"], st["k"], st["v"], st["do"], st["o"], st["lse"], st["dq"], st["dk"],
                                  st["dv"], st["workspace"], st["workspace_bytes"], stream)
        return {n: st[n] for n in ("o", "lse", "dq", "dk", "dv")}
    if entry == "partial":
        fcp.fcp_attn_fwd_merged(plan, st["q"], st["k"], st["v"], st["o_part"], st["lse_part"], st["o"], st["lse"],
                                stream=stream)
        return {n: st[n] for n in ("o", "lse")}
    scratch, scratch_bytes = st.get("scratch"), st.get("scratch_bytes")
    out = {}
    if entry == "new_batch":
        # 32 ranks with room for two `rank_tokens` each (one of them kept free); degrees from the search
        found = fcp.fcp_plan_strategy(st["lens"], 32, 2.0 * case["rank_tokens"], 1.0, 0.0, COST)
        plan = fcp.Plan(st["lens"], found["cp_degree"], case["hq"], case["hkv"], case["head_dim"]).upload(stream)
        scratch_bytes = plan.bwd_scratch_bytes()
        scratch = torch.empty(scratch_bytes, dtype=torch.uint8, device="cuda")
        out["cp_degree"] = found["cp_degree"]
    fcp.fcp_attn_fwd_fused(plan, st["q"], st["k"], st["v"], st["o"], st["lse"], stream=stream)
    out.update({n: st[n] for n in ("o", "lse")})
    if entry == "forward":
        return out
    if entry == "heads":
        fcp.fcp_attn_bwd_heads(plan, st["q"], st["k"], st["v"], st["o"], st["do"], st["lse"], 0, case["hkv"], st["dq"],
                               st["dk"], st["dv"], scratch, scratch_bytes, stream)
    else:
        fcp.fcp_attn_bwd(plan, st["q"], st["k"], st["v"], st["o"], st["do"], st["lse"], st["dq"], st["dk"], st["dv"],
                         scratch, scratch_bytes, stream)
    out.update({n: st[n] for n in ("dq", "dk", "dv")})
    return out


def work(case):
    """Every input tensor read once, every output written once; 4 * head_dim operations per visible
    (query, key) pair and query head forward, 2.5 times that backward."""
    lens, _, spans = batch(case)
    n = lens.astype(np.int64)
    pairs = int((n * (n + 1) // 2).sum())
    for sp in spans or []:
        pairs += sum((e - a) * (e - a - 1) // 2 for a, e in sp)
    q_bytes = case["tokens"] * case["hq"] * case["head_dim"] * 2
    kv_bytes = case["tokens"] * case["hkv"] * case["head_dim"] * 2
    lse_bytes = case["tokens"] * case["hq"] * 4
    flops = 4 * case["head_dim"] * case["hq"] * pairs
    if case["entry"] in ("forward", "partial"):
        return {"bytes": 2 * q_bytes + 2 * kv_bytes + lse_bytes, "flops": flops}
    return {"bytes": 4 * q_bytes + 4 * kv_bytes + lse_bytes, "flops": flops * 7 / 2}


def tolerance(case):
    # bf16 outputs from bf16 inputs with fp32 sums, probabilities and their gradients rounded to bf16 before the
    # second products: measured against fp64, o is off by 2.0e-3, dq and dk by 3.0e-3, dv by 2.3e-3 (2-norm).
    return {"rel": 1e-2}
