"""The kernels zero only those shared-memory rows that no copy reaches but a contraction reads.  Here every SM's shared memory
is first filled with NaN by calls on NaN inputs, then shapes with and without such rows meet the oracle."""
import pytest
import torch

import oracle
import paper_2603_13420_b200 as pskv
import parity
from paper_2603_13420_b200.inputs import Workload, make_inputs


def leave_nan_behind():
    nan = lambda *shape, dtype=torch.bfloat16: torch.full(shape, float("nan"), dtype=dtype, device="cuda")
    q, pk, sk = nan(192, 8, 64, 128), nan(2, 256, 128), nan(192, 2, 64, 128)
    pskv.pskv_attn_bwd(q, q, pk, pk, sk, sk, q, nan(192, 8, 64, dtype=torch.float32), 0.1)


@pytest.mark.gpu
@pytest.mark.parametrize("shape", [
    # B, Hq, Hkv, d, P, S
    (40, 8, 2, 128, 256, 48),    # every box a multiple of 16 rows and keys
    (7, 2, 2, 128, 200, 40),     # 8-key remainders, 40-row boxes
    (19, 2, 2, 64, 40, 1),
    (9, 3, 3, 128, 100, 24),
    (3, 4, 4, 128, 1200, 56),    # prefix streamed
    (5, 4, 4, 128, 300, 66),     # tiles that straddle candidates
    (2, 2, 2, 128, 70, 129),
], ids=lambda s: "x".join(map(str, s)))
def test_full_suffix_calls(shape):
    B, Hq, Hkv, d, P, S = shape
    w = Workload("unwritten", 300 + sum(shape), B=B, Hq=Hq, Hkv=Hkv, d=d, P=P, S=S)
    t = make_inputs(w, with_dout=True)
    leave_nan_behind()
    out, lse, dev = parity.run_fwd_gpu(t, w.scale)
    ref_out, ref_lse = parity.oracle_fwd(t, w.scale)
    parity.check_tensor("out", parity.to_f64(out), ref_out, strict_abs=P + S >= 128)
    parity.check_lse(parity.to_f64(lse), ref_lse)
    leave_nan_behind()
    grads = pskv.pskv_attn_bwd(dev["dout"], dev["q"], dev["prefix_k"], dev["prefix_v"], dev["suffix_k"], dev["suffix_v"],
                               out.contiguous(), lse.contiguous(), w.scale)
    for name, got, ref in zip(("dq", "dk_suffix", "dv_suffix"), grads, parity.oracle_bwd(t, w.scale)):
        parity.check_tensor(name, parity.to_f64(got), ref)


@pytest.mark.gpu
@pytest.mark.parametrize("Skv", [9, 48, 51])
def test_decode_calls(Skv):
    w = Workload("unwritten", 400 + Skv, B=37, Hq=8, Hkv=2, d=128, P=150, S=Skv)
    t = make_inputs(w)
    q = t["q"][:, :, -1:].contiguous()
    leave_nan_behind()
    out, lse = pskv.pskv_attn_fwd_decode(q.cuda(), t["prefix_k"].cuda(), t["prefix_v"].cuda(), t["suffix_k"].cuda(),
                                         t["suffix_v"].cuda(), None, w.scale)
    f = {k: parity.to_f64(v) for k, v in t.items()}
    ref_out, ref_lse = oracle.attn_fwd_decode(parity.to_f64(q), f["prefix_k"], f["prefix_v"], f["suffix_k"],
                                              f["suffix_v"], w.scale)
    parity.check_tensor("out", parity.to_f64(out), ref_out)
    parity.check_lse(parity.to_f64(lse), ref_lse)
