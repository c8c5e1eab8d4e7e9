"""The backward's row statistic D = <dout, out> formed as the first item of a tile (the diagonal of dO O^T): tiles of one box and of
several, rows that do not exist, several candidates to a key piece, the smallest launch that takes it, several instructions, and both
sides of the lines to the pre-pass; and which results a candidate with NaN queries leaves alone."""
import numpy as np
import pytest
import torch

import oracle
import paper_2603_13420_b200 as pskv
import parity
from paper_2603_13420_b200.inputs import Workload, make_inputs

pytestmark = pytest.mark.gpu

# Launches of a call, and of the same call with a (zero) gradient on lse, which the item does not take and the others do: that
# tells the item from D in the element-wise warps.
ITEM, WARPS, PRE_PASS = (1, 2), (1, 1), (2, 2)


@pytest.mark.parametrize("shape, form", [
    # B, Hq, Hkv, d, P, S
    ((300, 4, 4, 128, 40, 40), ITEM),       # three candidates in one box of 120 rows, 400 units
    ((500, 4, 4, 128, 40, 40), PRE_PASS),   # ... 668 units, more than four per SM
    ((260, 8, 2, 128, 65, 48), ITEM),       # tiles straddle two candidates: boxes of 64 rows
    ((600, 3, 3, 128, 0, 24), ITEM),        # no prefix; two candidates to a key piece
    ((250, 4, 2, 128, 17, 53), ITEM),       # two terms; padded rows and keys
    ((75, 4, 2, 128, 130, 33), ITEM),       # 150 units, two more than SMs; 72 of a tile's 128 rows
    ((74, 4, 2, 128, 130, 33), WARPS),      # ... 148: a tile per SM
    ((290, 8, 2, 128, 100, 51), ITEM),      # two terms, a second tile of 80 rows, two prefix pieces: 580 units
    ((300, 8, 2, 128, 100, 51), PRE_PASS),  # ... 600
    ((300, 8, 2, 128, 100, 57), ITEM),      # ... of 104 rows
    ((300, 4, 4, 128, 40, 72), PRE_PASS),   # two key pieces
    ((300, 4, 4, 64, 40, 40), PRE_PASS),    # head dim 64
], ids=str)
def test_gradients_match_the_oracle(shape, form):
    B, Hq, Hkv, d, P, S = shape
    w = Workload("d_item", 900 + sum(shape), B=B, Hq=Hq, Hkv=Hkv, d=d, P=P, S=S)
    t = make_inputs(w, with_dout=True)
    out, lse, dev = parity.run_fwd_gpu(t, w.scale)
    prefix = (dev["prefix_k"], dev["prefix_v"]) if P else (None, None)
    rest = (dev["q"], *prefix, dev["suffix_k"], dev["suffix_v"], out.contiguous(), lse.contiguous(), w.scale)
    n0 = pskv.pskv_kernel_launches()
    plain = pskv.pskv_attn_bwd(dev["dout"], *rest)
    n1 = pskv.pskv_kernel_launches()
    with_lse = pskv.pskv_attn_bwd_lse(dev["dout"], torch.zeros_like(lse), *rest)
    if torch.cuda.get_device_properties(0).multi_processor_count == 148:
        assert (n1 - n0, pskv.pskv_kernel_launches() - n1) == form
    assert pskv.pskv_poll_device_status() == pskv.PSKV_OK
    pick = [0, 1, 2, B // 2, B - 2, B - 1]
    f = {k: parity.to_f64(v[pick] if v.dim() == 4 and v.shape[0] == B else v) for k, v in t.items()}
    ref = oracle.attn_bwd(f["dout"], f["q"], f["prefix_k"], f["prefix_v"], f["suffix_k"], f["suffix_v"], w.scale)
    for name, g, r in zip(("dq", "dk_suffix", "dv_suffix"), plain, ref):
        parity.check_tensor(name, parity.to_f64(g[pick]), r)
    # zero gradient on lse: the same results up to the order of D's sum
    for a, b in zip(plain, with_lse):
        assert (a.double() - b.double()).norm() <= 1e-3 * b.double().norm()   # single results rounded to the next bf16 value


def test_several_instructions():
    """1248 units of three tiles, one launch; candidates at both ends of each instruction against the oracle."""
    B, Bp, Hq, Hkv, d, P, S, lens = 312, 3, 32, 8, 128, 200, 48, (200, 63, 129)
    w = Workload("d_item_multi", 78, B=B, Hq=Hq, Hkv=Hkv, d=d, P=P, S=S)
    t = make_inputs(w, with_dout=True)
    gen = torch.Generator().manual_seed(79)
    for k in ("prefix_k", "prefix_v"):
        t[k] = torch.randn((Bp, Hkv, P, d), generator=gen).to(torch.bfloat16)
    dev = {k: v.cuda() for k, v in t.items()}
    out, lse = pskv.pskv_attn_fwd_multi(dev["q"], dev["prefix_k"], dev["prefix_v"], lens, dev["suffix_k"], dev["suffix_v"], w.scale)
    n0 = pskv.pskv_kernel_launches()
    grads = pskv.pskv_attn_bwd_multi(dev["dout"], dev["q"], dev["prefix_k"], dev["prefix_v"], lens, dev["suffix_k"],
                                     dev["suffix_v"], out, lse, w.scale)
    if torch.cuda.get_device_properties(0).multi_processor_count == 148:
        assert pskv.pskv_kernel_launches() - n0 == 1
    assert pskv.pskv_poll_device_status() == pskv.PSKV_OK
    K = B // Bp
    pick = [i * K + j for i in range(Bp) for j in (0, K - 1)]
    f = {k: parity.to_f64(v if k.startswith("prefix") else v[pick]) for k, v in t.items()}
    ref = oracle.attn_bwd_multi(f["dout"], f["q"], f["prefix_k"], f["prefix_v"], oracle.left_padding_mask(lens, P),
                                f["suffix_k"], f["suffix_v"], w.scale)
    for name, g, r in zip(("dq", "dk_suffix", "dv_suffix"), grads, ref):
        parity.check_tensor(name, parity.to_f64(g[pick]), np.asarray(r))


def test_what_a_candidate_with_nan_queries_leaves_alone():
    """Candidates 0 to 2 share a tile, with rows 0-39, 40-79 and 80-119, the others its CTA's buffers.  All that
    is not candidate 0's stays as it is, but for candidate 1's dK: dK is summed over rows in steps of 16, so it takes in rows 32-39, which are
    candidate 0's and meet a zero."""
    w = Workload("d_item_nan", 77, B=320, Hq=4, Hkv=4, d=128, P=40, S=33)
    dev = {k: v.cuda() for k, v in make_inputs(w, with_dout=True).items()}

    def step():
        out, lse = pskv.pskv_attn_fwd(dev["q"], dev["prefix_k"], dev["prefix_v"], dev["suffix_k"], dev["suffix_v"], w.scale)
        n0 = pskv.pskv_kernel_launches()
        grads = pskv.pskv_attn_bwd(dev["dout"], dev["q"], dev["prefix_k"], dev["prefix_v"], dev["suffix_k"], dev["suffix_v"],
                                   out, lse, w.scale)
        if torch.cuda.get_device_properties(0).multi_processor_count == 148:
            assert pskv.pskv_kernel_launches() - n0 == 1
        return out, lse, *grads

    clean = step()
    dev["q"][0] = float("nan")
    poisoned = step()
    assert all(bool(torch.isnan(poisoned[i][0]).any()) for i in (0, 1, 2, 3))
    for name, a, b, first in zip(("out", "lse", "dq", "dk_suffix", "dv_suffix"), clean, poisoned, (1, 1, 1, 2, 1)):
        assert torch.equal(a[first:], b[first:]), name
