"""The tensor-core backward at the edges of its tiling: candidates whose rows or keys are no multiple of 8 or 16, several
candidates in one key piece, tiles that straddle candidates, suffixes of several 64-key pieces (taken in turn inside
one tile, or in extra passes over several tiles), the last unit short of candidates, empty and odd prefixes."""
import pytest
import torch

import oracle
import paper_2603_13420_b200 as pskv
import parity
from paper_2603_13420_b200.inputs import Workload, make_inputs

SHAPES = [
    # B, Hq, Hkv, d, P, S
    (19, 2, 2, 128, 40, 1),      # sixteen one-row candidates to a tile
    (17, 4, 4, 128, 64, 5),      # eight candidates to a key piece, short last unit
    (7, 2, 2, 64, 65, 21),       # two candidates to a piece, one key in the last prefix piece
    (5, 3, 3, 128, 1, 33),       # one-key prefix
    (9, 8, 2, 128, 130, 45),     # two tiles per candidate, the second partly empty
    (6, 8, 2, 128, 256, 48),     # tiles straddle two candidates (192 rows each)
    (5, 8, 2, 64, 256, 48),
    (7, 7, 1, 128, 100, 16),     # seven heads per KV head, 112 rows
    (3, 4, 4, 128, 63, 63),
    (3, 4, 4, 128, 0, 64),       # no prefix
    (3, 4, 4, 128, 191, 65),     # second piece with a single key
    (4, 2, 2, 64, 78, 113),
    (2, 8, 2, 128, 78, 113),     # four tiles, two pieces: an extra pass
    (2, 2, 1, 128, 128, 128),
    (2, 2, 2, 128, 70, 129),     # three pieces, two tiles per head
    (1, 4, 1, 64, 33, 200),
]


@pytest.mark.gpu
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_backward_matches_the_oracle(shape):
    B, Hq, Hkv, d, P, S = shape
    w = Workload("units", 700 + sum(shape), B=B, Hq=Hq, Hkv=Hkv, d=d, P=P, S=S)
    assert pskv.pskv_kernel_family(1, B, Hq, Hkv, S, P, d) == 1
    parity.bwd_parity(w)


@pytest.mark.gpu
@pytest.mark.parametrize("shape", [
    # enough candidates that whole candidates are the units (the shapes above are small enough for the split launch,
    # in which every tile's dQ and every suffix piece's dK / dV is a unit of its own)
    (700, 2, 2, 128, 40, 1), (420, 4, 4, 128, 64, 5), (320, 3, 3, 128, 1, 33), (400, 8, 2, 128, 130, 45),
    (400, 8, 2, 128, 256, 48), (401, 8, 2, 64, 256, 48), (400, 4, 4, 128, 191, 65), (400, 8, 2, 128, 78, 113),
    (300, 2, 2, 128, 70, 129), (900, 1, 1, 64, 33, 72),
    (401, 8, 2, 128, 385, 42),   # rows padded so that three tiles hold two candidates (the last unit one)
    (350, 8, 2, 128, 300, 67),   # ... several candidates per unit, two pieces each
], ids=lambda s: "x".join(map(str, s)))
def test_backward_of_many_candidates_matches_the_oracle(shape):
    B, Hq, Hkv, d, P, S = shape
    w = Workload("units", 1700 + sum(shape), B=B, Hq=Hq, Hkv=Hkv, d=d, P=P, S=S)
    assert pskv.pskv_kernel_family(1, B, Hq, Hkv, S, P, d) == 1
    parity.bwd_parity(w, cand=[0, 1, 2, B // 2 - 1, B // 2, B - 3, B - 2, B - 1])


@pytest.mark.gpu
def test_dq_at_a_base_that_is_16_but_not_32_bytes_aligned():
    """dQ leaves in whole 32-byte sectors where its base allows it, else in 16-byte halves: the same bits."""
    w = Workload("units", 899, B=4, Hq=8, Hkv=2, d=128, P=90, S=24)
    t = {k: v.cuda() for k, v in make_inputs(w, with_dout=True).items()}
    out, lse = pskv.pskv_attn_fwd(t["q"], t["prefix_k"], t["prefix_v"], t["suffix_k"], t["suffix_v"], w.scale)
    got = []
    for off in (0, 8):
        buf = torch.full((t["q"].numel() + 64,), float("nan"), dtype=torch.bfloat16, device="cuda")
        dq = buf[off:off + t["q"].numel()].view(t["q"].shape)
        assert dq.data_ptr() % 32 == 2 * off
        pskv.pskv_attn_bwd(t["dout"], t["q"], t["prefix_k"], t["prefix_v"], t["suffix_k"], t["suffix_v"], out, lse, w.scale, dq=dq)
        assert torch.isnan(buf[:off]).all() and torch.isnan(buf[off + dq.numel():]).all()
        got.append(dq.clone())
    assert torch.equal(got[0], got[1])


@pytest.mark.gpu
@pytest.mark.parametrize("case", [
    # B, Bp, Hq, Hkv, S, Pmax, d, lens: units never reach into the next instruction
    (14, 2, 4, 4, 13, 150, 128, (150, 70)),
    (9, 3, 8, 2, 45, 100, 128, (100, 0, 33)),
    (6, 2, 4, 2, 70, 129, 64, (129, 64)),
])
def test_instructions_with_odd_sizes_in_one_launch(case):
    B, Bp, Hq, Hkv, S, Pmax, d, lens = case
    gen = torch.Generator().manual_seed(4711 + S)
    draw = lambda *s: torch.randn(s, generator=gen, dtype=torch.float32).to(torch.bfloat16)
    t = dict(q=draw(B, Hq, S, d), prefix_k=draw(Bp, Hkv, Pmax, d), prefix_v=draw(Bp, Hkv, Pmax, d),
             suffix_k=draw(B, Hkv, S, d), suffix_v=draw(B, Hkv, S, d), dout=draw(B, Hq, S, d))
    for i, n in enumerate(lens):
        t["prefix_k"][i, :, : Pmax - n] = 3.0e4
        t["prefix_v"][i, :, : Pmax - n] = -3.0e4
    scale = d ** -0.5
    dev = {k: v.cuda() for k, v in t.items()}
    out, lse = pskv.pskv_attn_fwd_multi(dev["q"], dev["prefix_k"], dev["prefix_v"], lens, dev["suffix_k"], dev["suffix_v"], scale)
    got = []
    try:
        for form in ("one", "passes"):
            pskv.pskv_set_multi_form(form)
            got.append(pskv.pskv_attn_bwd_multi(dev["dout"], dev["q"], dev["prefix_k"], dev["prefix_v"], lens, dev["suffix_k"],
                                                dev["suffix_v"], out, lse, scale))
    finally:
        pskv.pskv_set_multi_form("auto")
    assert pskv.pskv_poll_device_status() == pskv.PSKV_OK
    f = {k: parity.to_f64(v) for k, v in t.items()}
    ref = oracle.attn_bwd_multi(f["dout"], f["q"], f["prefix_k"], f["prefix_v"], oracle.left_padding_mask(lens, Pmax),
                                f["suffix_k"], f["suffix_v"], scale)
    for name, a, b, r in zip(("dq", "dk_suffix", "dv_suffix"), got[0], got[1], ref):
        parity.check_tensor(name, parity.to_f64(a), r)
        parity.check_tensor(name + " (passes)", parity.to_f64(b), r)
