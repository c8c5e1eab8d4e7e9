"""The backward's row statistic D = <dout, out> formed as the first item of a tile (the diagonal of dO O^T): tiles of one box and of
several, rows that do not exist, several candidates to a key piece, the smallest launch that takes it, several instructions; and
that a candidate with NaN results leaves its neighbours in the same tiles' memory alone."""
import pytest
import torch

import oracle
import paper_2603_13420_b200 as pskv
import parity
from paper_2603_13420_b200.inputs import Workload, make_inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape, launches", [
    # B, Hq, Hkv, d, P, S
    ((300, 4, 4, 128, 40, 40), 1),     # three candidates in one box of 120 rows, 400 units
    ((500, 4, 4, 128, 40, 40), 2),     # ... 668 units, more than four per SM: the pre-pass
    ((260, 8, 2, 128, 65, 48), 1),     # tiles straddle two candidates: boxes of 64 rows
    ((600, 3, 3, 128, 0, 24), 1),      # no prefix; two candidates to a key piece
    ((250, 4, 2, 128, 17, 53), 1),     # two terms; padded rows and keys
    ((149, 1, 1, 128, 130, 64), 1),    # one unit more than SMs, half of each tile's rows do not exist
    ((290, 8, 2, 128, 100, 51), 1),    # two terms, a second tile of 80 rows, two prefix pieces: 580 units
    ((300, 8, 2, 128, 100, 51), 2),    # ... 600: the pre-pass
    ((300, 8, 2, 128, 100, 57), 1),    # ... of 104 rows
    ((300, 4, 4, 128, 40, 72), 2),     # two key pieces: the pre-pass
    ((300, 4, 4, 64, 40, 40), 2),      # head dim 64: the pre-pass
], ids=str)
def test_gradients_match_the_oracle(shape, launches):
    B, Hq, Hkv, d, P, S = shape
    w = Workload("d_item", 900 + sum(shape), B=B, Hq=Hq, Hkv=Hkv, d=d, P=P, S=S)
    t = make_inputs(w, with_dout=True)
    out, lse, dev = parity.run_fwd_gpu(t, w.scale)
    prefix = (dev["prefix_k"], dev["prefix_v"]) if P else (None, None)
    rest = (dev["q"], *prefix, dev["suffix_k"], dev["suffix_v"], out.contiguous(), lse.contiguous(), w.scale)
    n0 = pskv.pskv_kernel_launches()
    plain = pskv.pskv_attn_bwd(dev["dout"], *rest)
    if torch.cuda.get_device_properties(0).multi_processor_count == 148:
        assert pskv.pskv_kernel_launches() - n0 == launches
    assert pskv.pskv_poll_device_status() == pskv.PSKV_OK
    pick = [0, 1, 2, B // 2, B - 2, B - 1]
    f = {k: parity.to_f64(v[pick] if v.dim() == 4 and v.shape[0] == B else v) for k, v in t.items()}
    ref = oracle.attn_bwd(f["dout"], f["q"], f["prefix_k"], f["prefix_v"], f["suffix_k"], f["suffix_v"], w.scale)
    for name, g, r in zip(("dq", "dk_suffix", "dv_suffix"), plain, ref):
        parity.check_tensor(name, parity.to_f64(g[pick]), r)
    # with a gradient on lse D comes from the pre-pass: zero gradient on lse, the same results up to the order of D's sum
    with_lse = pskv.pskv_attn_bwd_lse(dev["dout"], torch.zeros_like(lse), *rest)
    for a, b in zip(plain, with_lse):
        assert (a.double() - b.double()).norm() <= 1e-3 * b.double().norm()   # single results rounded to the next bf16 value


def test_a_candidate_with_nan_results_leaves_the_others_alone():
    w = Workload("d_item_nan", 77, B=320, Hq=4, Hkv=4, d=128, P=40, S=33)
    dev = {k: v.cuda() for k, v in make_inputs(w, with_dout=True).items()}

    def step():
        out, lse = pskv.pskv_attn_fwd(dev["q"], dev["prefix_k"], dev["prefix_v"], dev["suffix_k"], dev["suffix_v"], w.scale)
        return pskv.pskv_attn_bwd(dev["dout"], dev["q"], dev["prefix_k"], dev["prefix_v"], dev["suffix_k"], dev["suffix_v"],
                                  out, lse, w.scale)

    clean = step()
    dev["q"][0] = float("nan")
    poisoned = step()
    assert all(bool(torch.isnan(g[0]).any()) for g in poisoned[:2])
    for a, b in zip(clean, poisoned):  # candidates 1 and 2 share candidate 0's tile, the others its CTA's buffers
        assert torch.equal(a[3:], b[3:])
