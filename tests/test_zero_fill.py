"""The rows a cache build leaves for later (free slots, room for decode steps) are zero, whatever the allocator hands out.
torch.empty is made to return 0xFF bytes, so an array that is not zeroed where the build does not write shows."""
import pytest
import torch

import paper_2402_18096_gb300 as pkg
from paper_2402_18096_gb300.layer import MixedPrecisionLayer

VARIANTS = {"bf16": dict(bits=2), "int3": dict(bits=3), "coded8": dict(bits=2, hi_bits=8),
            "coded2": dict(bits=4, hi_bits=2), "per-channel": dict(bits=2, k_channel_group=64), "evict": dict(bits=0)}


@pytest.fixture
def poisoned(monkeypatch):
    """torch.empty gives 0xFF; every array takes the way of a large one. Yields the poisoned allocations."""
    made, empty = [], torch.empty

    def dirty(*size, **kw):
        t = empty(*size, **kw)
        if t.numel():
            t.view(-1).view(torch.uint8).fill_(0xFF)
        made.append(t)
        return t

    monkeypatch.setattr(torch, "empty", dirty)
    monkeypatch.setattr(pkg, "FILL_WHOLE", 0)
    return made


def _shape(bits, hi_bits=16, k_channel_group=0, context=333, B=2, H=2):
    return pkg.shape_for_context(B, H, H, bits, 32, context, 0.2, 40, hi_bits=hi_bits, k_channel_group=k_channel_group)


def _is_zero(t):
    return not t.numel() or not bool(t.contiguous().view(torch.uint8).any())


@pytest.mark.parametrize("variant", list(VARIANTS))
def test_rows_past_the_filled_ones_are_zero(variant, poisoned):
    """The arrays alone, on the CPU: of each, exactly the rows that the caller said it writes are left as allocated."""
    shape = _shape(**VARIANTS[variant])
    hi, lo = shape.hi_cap - 1, 333 - (shape.hi_cap - 1) if shape.bits else 0
    cache = pkg.LayerCache(shape, device="cpu", filled=(hi, lo))
    assert poisoned
    groups = lo // 64
    first = dict.fromkeys(("k_hi", "v_hi", "k_hi_params", "v_hi_params", "hi_tok", "acc"), hi)
    first.update(dict.fromkeys(("k_codes", "v_codes", "v_params", "lo_tok"), 64 * groups if shape.k_channel_group else lo))
    first["k_params"] = groups if shape.k_channel_group else lo
    for name, n in first.items():
        t = getattr(cache, name)
        if t is not None:
            assert _is_zero(t[:, :, n:]), name
            written = t[:, :, :n].contiguous().view(torch.uint8) if t[:, :, :n].numel() else None
            assert written is None or bool((written == 0xFF).all()), name  # (the rows the build writes are not filled too)


@pytest.mark.gpu
@pytest.mark.parametrize("variant", list(VARIANTS))
def test_build_overwrites_or_zeroes_everything(variant, monkeypatch, request):
    """A whole build over poisoned allocations leaves the arrays of a build over zeros."""
    gen = torch.Generator().manual_seed(9)
    k, v = (torch.randn(2, 2, 333, 128, generator=gen).bfloat16().cuda() for _ in range(2))
    scores = torch.rand(2, 2, 333, generator=gen).cuda()
    shape = _shape(**VARIANTS[variant])
    want = vars(MixedPrecisionLayer.from_prefill(shape, k, v, scores).cache)
    poisoned = request.getfixturevalue("poisoned")
    got = vars(MixedPrecisionLayer.from_prefill(shape, k, v, scores).cache)
    assert len(poisoned) > 4
    for name, t in want.items():
        if isinstance(t, torch.Tensor) and t.numel():
            assert torch.equal(t.contiguous().view(torch.uint8), got[name].contiguous().view(torch.uint8)), name


@pytest.mark.gpu
def test_build_at_the_real_threshold():
    """Arrays of 32 MiB and more, over blocks of their sizes that were filled with 0xFF and freed."""
    B, H, T = 32, 8, 5300
    shape = _shape(2, context=T, B=B, H=H)
    k, v = (torch.randn(B, H, T, 128, device="cuda", dtype=torch.bfloat16) for _ in range(2))
    scores = torch.rand(B, H, T, device="cuda")
    sizes = [t.numel() * t.element_size() for t in vars(pkg.LayerCache(shape, device="cuda")).values()
             if isinstance(t, torch.Tensor)]
    assert sum(n >= pkg.FILL_WHOLE for n in sizes) >= 4
    junk = [torch.full((n,), 0xFF, dtype=torch.uint8, device="cuda") for n in sizes]
    del junk
    cache = MixedPrecisionLayer.from_prefill(shape, k, v, scores).cache
    hi, lo = shape.hi_cap - 1, T - (shape.hi_cap - 1)
    for name, n in (("k_hi", hi), ("v_hi", hi), ("hi_tok", hi), ("acc", hi), ("k_codes", lo), ("v_codes", lo),
                    ("k_params", lo), ("v_params", lo), ("lo_tok", lo)):
        assert _is_zero(getattr(cache, name)[:, :, n:]), name
