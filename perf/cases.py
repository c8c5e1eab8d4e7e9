"""Performance cases of the shared-prefix attention library: what a suffix-search program has it do.

Each case is one pass through the public calls, made the way README.md shows them (results and workspaces
allocated by the call).  The kinds, and where their sizes come from:

  score    pskv_attn_fwd over a batch of candidates: the attention step of candidate scoring, which is most of
           what a search does.  Sizes: the workload table of inputs.py; suffix + target lengths of the paper's
           data (20 suffix tokens, 93 target tokens on average) and the odd lengths around them that a
           tokenizer produces; head layouts 32/32 (Llama-2, Vicuna) and 32/8 (Llama-3, Mistral).
  step     pskv_attn_fwd + pskv_attn_bwd: the same with gradients, from the one current suffix of a search
           up to a whole batch of candidates.
  decode   pskv_attn_fwd_decode: searches that grow every candidate token by token (beam search, sampling).
  multi    pskv_attn_fwd_multi + pskv_attn_bwd_multi: several instructions, one left-padded prefix cache each.
  prefill  pskv_attn_fwd with B = 1 and no prefix: the causal pass that makes a prefix cache.
  ce       pskv_target_ce_fwd: candidate losses over the vocabulary projection.

All tensors are bf16 (the library's one input type), head dimension 128 but for the smallest cases (64).
"""
import math

import torch

import paper_2603_13420_b200 as pskv
from paper_2603_13420_b200.inputs import OUTLIER_CHANNELS, OUTLIER_GAIN

DEVICE = "cuda"


def listed():
    return [
        # the smallest calls: a few candidates of a small model, where launches and host work count
        dict(name="step_small", kind="step", B=8, Hq=4, Hkv=4, d=64, P=32, S=8, outliers=False),
        # gradient of the one current suffix of a search (20 suffix + 93 target tokens behind 78 instruction
        # tokens, the paper's average lengths), Llama-3 heads
        dict(name="grad_single", kind="step", B=1, Hq=32, Hkv=8, d=128, P=78, S=113, outliers=False),
        # candidate scoring on the Llama-2 and Llama-3 layer shapes of the workload table, and with a long prefix
        dict(name="score_mha", kind="score", B=512, Hq=32, Hkv=32, d=128, P=160, S=40, outliers=False),
        dict(name="score_long_prefix", kind="score", B=256, Hq=32, Hkv=8, d=128, P=2048, S=32, outliers=False),
        # the same at lengths that are multiples of nothing, which is how suffix + target usually come out
        dict(name="score_odd", kind="score", B=333, Hq=32, Hkv=8, d=128, P=217, S=53, outliers=False),
        # scoring with gradients: the benchmark's step, the gradient workload of the table, an odd batch with the
        # average target length
        dict(name="step_gqa", kind="step", B=512, Hq=32, Hkv=8, d=128, P=256, S=48, outliers=True),
        dict(name="step_mha", kind="step", B=128, Hq=32, Hkv=32, d=128, P=160, S=40, outliers=False),
        dict(name="step_long_target", kind="step", B=100, Hq=32, Hkv=32, d=128, P=78, S=113, outliers=False),
        # one new token per beam on top of ragged cached suffixes
        dict(name="decode_beams", kind="decode", B=512, Hq=32, Hkv=8, d=128, P=256, Sq=1, Skv=48, outliers=True),
        # eight instructions of different lengths, 64 candidates each, with gradients
        dict(name="multi_8x64", kind="multi", B=512, Bp=8, Hq=32, Hkv=8, d=128, P=256, S=48, outliers=True),
        # the prefix cache of a long prompt
        dict(name="prefill_2048", kind="prefill", B=1, Hq=32, Hkv=8, d=128, P=0, S=2048, outliers=False),
        # losses of 512 candidates over 20 target tokens with the Llama-3 vocabulary
        dict(name="target_ce", kind="ce", N=512, Lr=20, Dm=4096, V=128256),
    ]


HEADS = ((32, 32), (32, 8))
MAX_ROWS = 512 * 32 * 48      # query rows of the largest listed attention case
MAX_SCORES = 2048 * 256 * 32 * 32  # ... and query rows x keys


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choices(("score", "step", "small", "decode", "multi", "prefill", "ce"), (6, 6, 1, 2, 2, 1, 2))[0]
    Hq, Hkv = rng.choice(HEADS)
    outliers = rng.random() < 0.5
    if kind == "small":
        return dict(kind="step", B=_log_int(rng, 2, 64), Hq=4, Hkv=4, d=64, P=_log_int(rng, 16, 256),
                    S=rng.randint(4, 40), outliers=outliers)
    if kind == "prefill":
        return dict(kind="prefill", B=1, Hq=Hq, Hkv=Hkv, d=128, P=0, S=_log_int(rng, 64, 4096), outliers=outliers)
    if kind == "ce":
        return dict(kind="ce", N=_log_int(rng, 16, 512), Lr=rng.randint(1, 20), Dm=4096, V=rng.choice((32000, 128256)))
    if kind == "decode":
        # Sq is 1 for plain decoding; a few for a step that extends every candidate by a short run
        Sq = rng.choice((1, 1, 1, 2, 4))
        return dict(kind="decode", B=_log_int(rng, 16, 2048), Hq=Hq, Hkv=Hkv, d=128, P=_log_int(rng, 32, 2048), Sq=Sq,
                    Skv=rng.randint(max(8, Sq), 128), outliers=outliers)
    S, P = rng.randint(8, 128), _log_int(rng, 32, 2048)
    top = max(2, min(512, MAX_ROWS // (Hq * S), MAX_SCORES // (Hq * S * (P + S))))
    if kind == "multi":
        Bp = rng.randint(2, 16)
        P = min(P, 512)
        Kq = max(1, min(_log_int(rng, 4, 128), MAX_ROWS // (Hq * S * Bp)))
        return dict(kind="multi", B=Bp * Kq, Bp=Bp, Hq=Hq, Hkv=Hkv, d=128, P=P, S=S, outliers=outliers)
    B = _log_int(rng, 1 if kind == "step" else 8, max(8, top))
    return dict(kind=kind, B=B, Hq=Hq, Hkv=Hkv, d=128, P=P, S=S, outliers=outliers)


def _prefix_lens(case):
    """True lengths of the instructions' prefixes: from half of the padded length up to all of it, one of them the longest."""
    n, P = case["Bp"], case["P"]
    return [P - (i * 5 % n) * (P // 2) // n for i in range(n)]


def prepare(case, seed):
    gen = torch.Generator(device=DEVICE)
    gen.manual_seed(seed)

    def normal(*shape, outliers=False, gain=1.0):
        x = torch.randn(shape, generator=gen, device=DEVICE, dtype=torch.float32)
        if gain != 1.0:
            x *= gain
        if outliers:  # a few key channels of large magnitude, as language models have them
            for c in OUTLIER_CHANNELS:
                if c < shape[-1]:
                    x[..., c] *= OUTLIER_GAIN
        return x.to(torch.bfloat16)

    kind = case["kind"]
    if kind == "ce":
        N, Lr, Dm, V = case["N"], case["Lr"], case["Dm"], case["V"]
        mask = torch.rand((N, Lr), generator=gen, device=DEVICE)
        mask = (mask < 0.9).to(torch.float32)  # some positions are padding
        mask[:, 0] = 1.0
        return dict(case=case, hidden=normal(N, Lr, Dm), weight=normal(V, Dm, gain=3.0 / math.sqrt(Dm)),
                    target=torch.randint(0, V, (N, Lr), generator=gen, device=DEVICE, dtype=torch.int32), mask=mask)
    B, Hq, Hkv, d, P, o = (case[k] for k in ("B", "Hq", "Hkv", "d", "P", "outliers"))
    Sq = case["Sq"] if kind == "decode" else case["S"]
    Skv = case["Skv"] if kind == "decode" else case["S"]
    lead = (case["Bp"],) if kind == "multi" else ()
    state = dict(case=case, scale=1.0 / math.sqrt(d), q=normal(B, Hq, Sq, d),
                 prefix_k=normal(*lead, Hkv, P, d, outliers=o) if P else None,
                 prefix_v=normal(*lead, Hkv, P, d) if P else None,
                 suffix_k=normal(B, Hkv, Skv, d, outliers=o), suffix_v=normal(B, Hkv, Skv, d))
    if kind in ("step", "multi"):
        state["dout"] = normal(B, Hq, Sq, d)
    if kind == "multi":
        state["prefix_len"] = _prefix_lens(case)
    if kind == "decode":  # beams differ in how much of their suffix is there
        state["suffix_len"] = torch.randint(max(Sq, Skv // 2), Skv + 1, (B,), generator=gen, device=DEVICE,
                                            dtype=torch.int32)
    return state


def run(state):
    s, kind = state, state["case"]["kind"]
    if kind == "ce":
        nll, lse, loss = pskv.pskv_target_ce_fwd(s["hidden"], s["weight"], s["target"], s["mask"])
        return dict(nll=nll, lse=lse, loss=loss)
    if kind == "decode":
        out, lse = pskv.pskv_attn_fwd_decode(s["q"], s["prefix_k"], s["prefix_v"], s["suffix_k"], s["suffix_v"],
                                             s["suffix_len"], s["scale"])
        return dict(out=out, lse=lse)
    if kind == "multi":
        out, lse = pskv.pskv_attn_fwd_multi(s["q"], s["prefix_k"], s["prefix_v"], s["prefix_len"], s["suffix_k"],
                                            s["suffix_v"], s["scale"])
        dq, dk, dv = pskv.pskv_attn_bwd_multi(s["dout"], s["q"], s["prefix_k"], s["prefix_v"], s["prefix_len"],
                                              s["suffix_k"], s["suffix_v"], out, lse, s["scale"])
        return dict(out=out, lse=lse, dq=dq, dk_suffix=dk, dv_suffix=dv)
    out, lse = pskv.pskv_attn_fwd(s["q"], s["prefix_k"], s["prefix_v"], s["suffix_k"], s["suffix_v"], s["scale"])
    if kind != "step":
        return dict(out=out, lse=lse)
    dq, dk, dv = pskv.pskv_attn_bwd(s["dout"], s["q"], s["prefix_k"], s["prefix_v"], s["suffix_k"], s["suffix_v"],
                                    out, lse, s["scale"])
    return dict(out=out, lse=lse, dq=dq, dk_suffix=dk, dv_suffix=dv)


def work(case):
    """Bytes: each call's inputs read once and its outputs written once.  Flops: causally visible keys only, two
    contractions forward; backward three on the (frozen) prefix keys and five on the suffix keys."""
    kind = case["kind"]
    if kind == "ce":
        rows = case["N"] * case["Lr"]
        return {"bytes": 2 * case["Dm"] * (rows + case["V"]) + 16 * rows + 4 * case["N"],
                "flops": 2.0 * rows * case["Dm"] * case["V"]}
    B, Hq, Hkv, d, P = (case[k] for k in ("B", "Hq", "Hkv", "d", "P"))
    if kind == "decode":
        Sq, Skv = case["Sq"], case["Skv"]
        have = (max(Sq, Skv // 2) + Skv) / 2.0  # cached tokens of a candidate, on average
        rows, visible = B * Hq * Sq, have - (Sq - 1) / 2.0
        return {"bytes": rows * (4 * d + 4) + 4 * d * B * Hkv * have + 4 * d * Hkv * P + 4 * B,
                "flops": 4.0 * d * rows * (P + visible)}
    S = case["S"]
    rows, visible = B * Hq * S, (S + 1) / 2.0
    prefix_rows = P if kind != "multi" else sum(_prefix_lens(case))
    keys = P if kind != "multi" else prefix_rows / case["Bp"]
    kv = 4 * d * (B * Hkv * S + Hkv * prefix_rows)
    bytes_, flops = rows * (4 * d + 4) + kv, 4.0 * d * rows * (keys + visible)
    if kind in ("step", "multi"):
        bytes_ += rows * (8 * d + 4) + kv + 4 * d * B * Hkv * S
        flops += d * rows * (6.0 * keys + 10.0 * visible)
    return {"bytes": bytes_, "flops": flops}


def tolerance(case):
    """About four times the distance of the library's results from the same formulas in 64 bits.  Measured over the
    listed and a dozen drawn cases: out 2.4e-3 (largest single difference 0.05 of max(rms, value), in the first rows
    of a sequence, which see few keys), gradients 2.7e-3 (0.02), 3.6e-3 (0.21) with large key channels, where dQ of a
    row with few keys is a small difference of large terms; probabilities and dS are rounded to bf16 before their
    second contraction.  Losses: fp32 sums of exact bf16 products, 2.3e-6 (4e-6)."""
    if case["kind"] == "ce":
        return {"rel": 1e-5, "max": 2e-5}
    if case["kind"] in ("step", "multi"):
        return {"rel": 1.5e-2, "max": 0.85} if case["outliers"] else {"rel": 1.1e-2, "max": 0.2}
    return {"rel": 1e-2, "max": 0.2}
