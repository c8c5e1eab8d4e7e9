"""The extension module takes what the ctypes binding took, and refuses what it refused."""
import math

import pytest
import torch

import paper_2603_13420_b200 as pskv


def _inputs():
    gen = torch.Generator().manual_seed(99)
    draw = lambda *s: torch.randn(s, generator=gen).to(torch.bfloat16).cuda()
    return draw(4, 4, 8, 64), draw(2, 2, 24, 64), draw(2, 2, 24, 64), draw(4, 2, 8, 64), draw(4, 2, 8, 64)


@pytest.mark.gpu
def test_forms_of_the_arguments():
    q, pk, pv, sk, sv = _inputs()
    scale = 0.125
    ref = pskv.pskv_attn_fwd(q, pk[0], pv[0], sk, sv, scale)
    same = lambda r: all(torch.equal(x, y) for x, y in zip(r, ref))
    for form in ("0.125", torch.tensor(0.125), torch.tensor([0.125]).numpy()[0]):
        assert same(pskv.pskv_attn_fwd(q, pk[0], pv[0], sk, sv, form))
    # sizes are read off q and the leading dimensions of the caches, whose last ones may be merged
    assert same(pskv.pskv_attn_fwd(q, pk[0].view(2, 24, 8, 8), pv[0].view(2, 24, 8, 8), sk.view(4, 2, 512), sv.view(4, 2, 512), scale))
    lens = [24, 9]
    multi = pskv.pskv_attn_fwd_multi(q, pk, pv, lens, sk, sv, scale)
    for form in (tuple(lens), torch.tensor(lens), torch.tensor(lens).numpy(), [24.0, "9"], [2 ** 64 + 24, 9]):
        assert all(torch.equal(x, y) for x, y in zip(pskv.pskv_attn_fwd_multi(q, pk, pv, form, sk, sv, scale), multi))


@pytest.mark.gpu
def test_what_is_refused():
    q, pk, pv, sk, sv = _inputs()
    with pytest.raises(TypeError):
        pskv.pskv_attn_fwd_multi(q, pk, pv, (n for n in (24, 9)), sk, sv, 0.125)
    with pytest.raises(ValueError):
        pskv.pskv_attn_fwd(q[0], pk[0], pv[0], sk, sv, 0.125)
    with pytest.raises(ValueError):
        pskv.pskv_attn_fwd(q.transpose(1, 2), pk[0], pv[0], sk, sv, 0.125)
    with pytest.raises(IndexError):
        pskv.pskv_attn_fwd(q, pk[0], pv[0], sk.view(-1), sv, 0.125)
    with pytest.raises(ValueError):
        pskv.pskv_attn_fwd(q, pk[0], pv[0], sk, sv, "scale")
    with pytest.raises(pskv.PskvError):
        pskv.pskv_attn_fwd_multi(q, pk, pv, [], sk, sv, 0.125)
    assert math.isfinite(float(pskv.pskv_attn_fwd(q, pk[0], pv[0], sk, sv, 0.125)[1].sum()))


def test_host_tensors_are_refused():
    t = torch.zeros((1, 1, 1, 64), dtype=torch.bfloat16)
    with pytest.raises(ValueError):
        pskv.pskv_attn_fwd(t, None, None, t, t, 0.1)


def test_a_module_built_for_another_torch_is_stale_and_refused(monkeypatch):
    from paper_2603_13420_b200 import _native, binding, build

    assert _native.built_for == build.built_for() and torch.__version__ in _native.built_for
    assert not build._native_stale()
    monkeypatch.setattr(build, "built_for", lambda: "cpython-312 torch 0.0.1")
    assert build._native_stale() and build.is_stale()
    monkeypatch.setattr(binding, "_native", None)
    monkeypatch.setattr(torch, "__version__", "0.0.1")
    with pytest.raises(RuntimeError, match="built for"):
        binding.native()
