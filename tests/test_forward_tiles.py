"""The tensor-core forward at the edges of its tiling: candidates whose rows or keys are no multiple of 8, padded to the next
multiple or as far as a tile's end, boxes that hold padding only, a short last tile, suffixes of one
whole key block, tiles that straddle candidates with suffix keys in several blocks, lengths beyond 128 that have no
divisor."""
import pytest
import torch

import oracle
import paper_2603_13420_b200 as pskv
import parity
from paper_2603_13420_b200.inputs import Workload, make_inputs

SHAPES = [
    # B, Hq, Hkv, d, P, S
    (19, 2, 2, 128, 40, 1),      # one row per candidate: whole candidates, suffix keys in several blocks
    (21, 4, 4, 128, 200, 13),    # 16 rows per candidate, eight to a tile
    (9, 8, 2, 128, 217, 53),     # 212 rows padded to 224: tiles straddle candidates, boxes of 32 rows
    (5, 8, 2, 64, 129, 45),
    (3, 8, 2, 128, 78, 113),     # 452 rows padded to 480: four tiles of 120 rows inside a candidate
    (4, 2, 2, 128, 600, 121),    # prefix streamed
    (3, 7, 1, 128, 100, 35),     # seven heads per KV head
    (2, 8, 2, 128, 0, 127),      # no prefix
    (33, 3, 3, 64, 31, 9),
    (300, 8, 2, 128, 257, 21),   # several tiles per CTA
    (5, 4, 4, 128, 300, 66),     # tiles that straddle candidates, a suffix block per candidate
    (9, 2, 2, 64, 40, 85),
    (300, 2, 2, 128, 200, 70),
    (11, 3, 3, 128, 700, 45),    # ... two candidates to a suffix block
    (1, 4, 2, 128, 0, 131),      # beyond 128 queries: tiles inside one head, heads padded to whole tiles
    (2, 4, 4, 64, 60, 139),
    (1, 2, 1, 128, 0, 1039),
    (1, 8, 2, 128, 33, 513),
    (262, 4, 4, 128, 20, 8),     # tiles of half as many rows as fit, for twice as many SMs
    (9, 7, 1, 128, 34, 8),       # a candidate per tile
    (133, 7, 1, 128, 300, 40),   # boxes of 8 rows, for a round of the SMs less
]


@pytest.mark.gpu
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_forward_matches_the_oracle(shape):
    B, Hq, Hkv, d, P, S = shape
    w = Workload("tiles", 900 + sum(shape), B=B, Hq=Hq, Hkv=Hkv, d=d, P=P, S=S)
    assert pskv.pskv_kernel_family(0, B, Hq, Hkv, S, P, d) == 1
    cand = None if B <= 64 else [0, 1, 2, B // 2 - 1, B // 2, B - 3, B - 2, B - 1]
    parity.fwd_parity(w, cand=cand, strict_abs=(P + S >= 128))


@pytest.mark.gpu
def test_rows_outside_the_safe_exponent_range_next_to_padding_rows():
    """Scores of several hundred nats in the last real rows before a candidate's padding, and in the first after it."""
    w = Workload("tiles", 977, B=6, Hq=8, Hkv=2, d=128, P=90, S=53)
    t = make_inputs(w)
    q = t["q"].float()
    q[1, 3, 52] *= 60.0
    q[2, 0, 0] *= -60.0
    q[5, 7, 52] *= 60.0
    t["q"] = q.to(t["q"].dtype)
    out, lse, _ = parity.run_fwd_gpu(t, w.scale)
    ref_out, ref_lse = parity.oracle_fwd(t, w.scale)
    assert abs(ref_lse).max() > 100.0
    parity.check_tensor("out", parity.to_f64(out), ref_out)
    parity.check_lse(parity.to_f64(lse), ref_lse)


@pytest.mark.gpu
@pytest.mark.parametrize("case", [
    # B, Bp, Hq, Hkv, S, Pmax, d, lens: an instruction is no whole number of tiles, its last tile is short
    (24, 3, 8, 2, 37, 300, 128, (300, 129, 40)),
    (44, 2, 4, 4, 21, 64, 64, (0, 64)),
    (30, 5, 4, 4, 100, 600, 128, (600, 1, 470, 128, 129)),
])
def test_several_instructions_whose_last_tiles_are_short_in_one_launch(case):
    B, Bp, Hq, Hkv, S, Pmax, d, lens = case
    gen = torch.Generator().manual_seed(4242 + S)
    draw = lambda *s: torch.randn(s, generator=gen, dtype=torch.float32).to(torch.bfloat16)
    t = dict(q=draw(B, Hq, S, d), prefix_k=draw(Bp, Hkv, Pmax, d), prefix_v=draw(Bp, Hkv, Pmax, d),
             suffix_k=draw(B, Hkv, S, d), suffix_v=draw(B, Hkv, S, d))
    for i, n in enumerate(lens):
        t["prefix_k"][i, :, : Pmax - n] = 3.0e4
        t["prefix_v"][i, :, : Pmax - n] = -3.0e4
    dev = {k: v.cuda() for k, v in t.items()}
    n0 = pskv.pskv_kernel_launches()
    out, lse = pskv.pskv_attn_fwd_multi(dev["q"], dev["prefix_k"], dev["prefix_v"], lens, dev["suffix_k"], dev["suffix_v"], d ** -0.5)
    assert pskv.pskv_kernel_launches() - n0 == 1
    assert pskv.pskv_poll_device_status() == pskv.PSKV_OK
    f = {k: parity.to_f64(v) for k, v in t.items()}
    ref_out, ref_lse = oracle.attn_fwd_multi(f["q"], f["prefix_k"], f["prefix_v"], oracle.left_padding_mask(lens, Pmax),
                                             f["suffix_k"], f["suffix_v"], d ** -0.5)
    parity.check_tensor("out", parity.to_f64(out), ref_out)
    parity.check_lse(parity.to_f64(lse), ref_lse)
