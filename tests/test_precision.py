"""Gradients of suffix lengths that are no multiple of 8, or beyond 64, are as exact as fp32 probabilities and dS make them: what is
left is the rounding of the result to bf16.  (dQ of a multiple of 8 up to 128 takes dS rounded to bf16, as up to 64.)
The same of the forward of more than 128 queries whose rows have no divisor between 16 and 128."""
import numpy as np
import pytest
import torch

import oracle
import paper_2603_13420_b200 as pskv
import parity
from paper_2603_13420_b200.inputs import Workload, make_inputs


def _rounding(ref):
    return np.linalg.norm(torch.from_numpy(ref).to(torch.bfloat16).double().numpy() - ref)


@pytest.mark.gpu
@pytest.mark.parametrize("shape", [
    # B, Hq, Hkv, d, P, S
    (2, 8, 2, 128, 78, 113),     # split units, several tiles per candidate
    (9, 8, 2, 128, 256, 30),     # one tile per unit, D formed in the kernel
    (24, 4, 4, 64, 100, 50),
    (300, 4, 4, 128, 200, 21),   # several candidates in a key piece
    (200, 8, 2, 128, 385, 42),   # tiles that straddle candidates
    (160, 8, 2, 64, 40, 77),     # a second pass for the second piece
    (3, 4, 4, 128, 0, 129),
    (6, 4, 2, 128, 90, 72),      # a multiple of 8 beyond one piece
], ids=lambda s: "x".join(map(str, s)))
def test_gradients_are_off_by_the_rounding_of_the_result_alone(shape):
    B, Hq, Hkv, d, P, S = shape
    w = Workload("precision", 300 + sum(shape), B=B, Hq=Hq, Hkv=Hkv, d=d, P=P, S=S)
    t = make_inputs(w, with_dout=True)
    out, lse, dev = parity.run_fwd_gpu(t, w.scale)
    out, lse = out.contiguous(), lse.contiguous()
    prefix = (dev["prefix_k"], dev["prefix_v"]) if P else (None, None)
    grads = pskv.pskv_attn_bwd(dev["dout"], dev["q"], *prefix, dev["suffix_k"], dev["suffix_v"], out, lse, w.scale)
    assert pskv.pskv_poll_device_status() == pskv.PSKV_OK
    cand = sorted({0, 1, B // 2, B - 1})
    f = {k: parity.to_f64(v if k.startswith("prefix") else v[cand]) for k, v in t.items()}
    # D = <dout, out> is formed from the rounded `out`; the oracle's from its own: the difference goes in as a gradient on lse
    ref_out, _ = oracle.attn_fwd(f["q"], f["prefix_k"], f["prefix_v"], f["suffix_k"], f["suffix_v"], w.scale)
    dlse = (f["dout"] * (ref_out - parity.to_f64(out[cand]))).sum(-1)
    refs = oracle.attn_bwd_lse(f["dout"], dlse, f["q"], f["prefix_k"], f["prefix_v"], f["suffix_k"], f["suffix_v"], w.scale)
    for name, g, r in zip(("dq", "dk_suffix", "dv_suffix"), grads, refs):
        if name == "dq" and S % 8 == 0 and S <= 128:
            continue
        err = np.linalg.norm(parity.to_f64(g[cand]) - r)
        # Two bf16 terms hold 16 bits: 2^-17 relative, a few hundredths of the result's own rounding (2^-9) even where the terms
        # of a sum cancel tenfold.  One term (2^-9 again) would give a factor of 1.4.
        assert err <= 1.05 * _rounding(r), (name, err / _rounding(r))


@pytest.mark.gpu
@pytest.mark.parametrize("shape", [
    # B, Hq, Hkv, d, P, S: rows without a divisor between 16 and 128
    (1, 4, 1, 128, 0, 131), (2, 2, 2, 64, 75, 139), (1, 2, 1, 128, 0, 1039), (1, 3, 3, 128, 40, 257),
], ids=lambda s: "x".join(map(str, s)))
def test_forward_of_lengths_without_a_divisor_is_off_by_the_rounding_of_the_result_alone(shape):
    B, Hq, Hkv, d, P, S = shape
    w = Workload("precision", 400 + sum(shape), B=B, Hq=Hq, Hkv=Hkv, d=d, P=P, S=S)
    t = make_inputs(w)
    out, lse, _ = parity.run_fwd_gpu(t, w.scale)
    ref_out, ref_lse = parity.oracle_fwd(t, w.scale)
    assert np.linalg.norm(parity.to_f64(out) - ref_out) <= 1.05 * _rounding(ref_out)
    # fp32 scores of about 10 log2 units, a sum over the keys and the rounding of the result, 2^-24 each
    assert np.linalg.norm(parity.to_f64(lse) - ref_lse) <= 2.0 ** -24 * np.linalg.norm(ref_lse)
