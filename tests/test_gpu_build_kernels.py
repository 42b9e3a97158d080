"""GPU parity of the cache-build kernels at the edges of their tiles: the bulk quantizer's rounds, the balancer's
row chunks and its path for unaligned inputs, the bulk selection's rounds and ties, the gather's row groups, and the
rows a build leaves zero. Everything here is bit-exact."""
import numpy as np
import pytest
import torch

import oracle
import paper_2402_18096_gb300 as pkg
from paper_2402_18096_gb300.layer import MixedPrecisionLayer
from _cases import bits16, new_workspace

pytestmark = pytest.mark.gpu
D = 128


def _rand_bf16(*shape, gen, scale=1.0):
    return (torch.randn(*shape, generator=gen) * scale).to(torch.bfloat16)


def _unaligned(t, dev):
    """The tensor on the device, 4 elements into its allocation (8 bytes for bf16)."""
    store = torch.empty(t.numel() + 4, dtype=t.dtype, device=dev)
    out = store[4:].view(t.shape)
    out.copy_(t)
    assert out.data_ptr() % 16 != 0 and out.is_contiguous()
    return out


@pytest.mark.parametrize("n_rows", [1, 15, 16, 17, 127, 128, 129, 260])
@pytest.mark.parametrize("bits,group", [(2, 32), (3, 64), (4, 128), (3, 128), (4, 32)])
def test_quantize_pack_row_counts(n_rows, bits, group):
    gen = torch.Generator().manual_seed(n_rows * 10 + bits)
    B, Hkv, n_src = 1, 3, 300
    shape = pkg.Shape(B, Hkv, Hkv, bits, group, hi_cap=1, lo_cap=272)
    k = _rand_bf16(B, Hkv, n_src, D, gen=gen, scale=3.0)
    v = _rand_bf16(B, Hkv, n_src, D, gen=gen)
    k[0, 0, ::7] *= 1e-6   # spans far below an fp16 step
    v[0, 1, ::5] *= 1e5    # scales beyond fp16
    v[0, 2, ::3] = 2.5     # zero span
    bal = (torch.rand(Hkv, D, generator=gen) * 3 + 0.2).float()
    rows = torch.stack([torch.randperm(n_src, generator=gen)[:n_rows] for _ in range(Hkv)]).view(B, Hkv, n_rows).int()
    dev = torch.device("cuda")
    cache = pkg.LayerCache(shape, device=dev, balancer=bal.to(dev))
    for name in ("k_codes", "v_codes"):
        getattr(cache, name).fill_(0xA5)
    pkg.mikv_quantize_pack(cache, k.to(dev), v.to(dev), rows.to(dev), 3)
    ref = oracle.empty_cache(B, Hkv, D, bits, group, 1, 272)
    oracle.quantize_pack(ref, bits16(k), bits16(v), rows.numpy(), 3, balancer_=bal.numpy())
    sl = slice(3, 3 + n_rows)
    for name in ("k_codes", "v_codes", "lo_tok"):
        np.testing.assert_array_equal(getattr(cache, name)[:, :, sl].cpu().numpy(), ref[name][:, :, sl], err_msg=name)
    for name in ("k_params", "v_params"):
        got = getattr(cache, name)[:, :, sl].cpu().view(torch.int16).numpy().view(np.uint16)
        np.testing.assert_array_equal(got, ref[name][:, :, sl], err_msg=name)
    for name in ("k_codes", "v_codes"):  # nothing outside the rows is written
        rest = getattr(cache, name).clone()
        rest[:, :, sl] = 0xA5
        assert bool((rest == 0xA5).all())


@pytest.mark.parametrize("T", [1, 15, 16, 17, 127, 128, 129, 1023, 1024, 1025, 2300])
@pytest.mark.parametrize("aligned", [True, False], ids=["aligned", "unaligned"])
def test_balancer_row_counts(T, aligned):
    gen = torch.Generator().manual_seed(T)
    B, Hq, Hkv = 2, 4, 2
    q = _rand_bf16(B, Hq, T, D, gen=gen, scale=2.0)
    k = _rand_bf16(B, Hkv, T, D, gen=gen, scale=2.0)
    q[:, :, T // 2, 3] = -60.0   # the maximum sits in one row
    k[1, 1, T - 1, 4] = 90.0     # the last row of the last head
    k[:, 0, :, 5] = -0.0
    shape = pkg.Shape(B, Hq, Hkv, 2, 32, hi_cap=1, lo_cap=16)
    dev = torch.device("cuda")
    place = (lambda t: t.to(dev)) if aligned else (lambda t: _unaligned(t, dev))
    out = torch.empty(Hkv, D, dtype=torch.float32, device=dev)
    pkg.mikv_compute_balancer(shape, place(q), place(k), out, new_workspace(shape, pkg.WS_BALANCER, 0))
    ref = oracle.balancer(bits16(q), bits16(k))
    np.testing.assert_array_equal(out.cpu().numpy().view(np.uint32), ref.view(np.uint32))


def test_balancer_passes_over_nan_and_keeps_infinity():
    """NaN entries do not count and infinities do, the same on both paths."""
    gen = torch.Generator().manual_seed(5)
    q, k = _rand_bf16(1, 2, 200, D, gen=gen), _rand_bf16(1, 2, 200, D, gen=gen)
    q[0, 0, ::3, 1] = float("nan")
    q[0, 0, :, 2] = float("nan")
    q[0, 1, 7, 3] = float("inf")
    k[0, 1, 9, 4] = float("-inf")
    shape = pkg.Shape(1, 2, 2, 2, 32, hi_cap=1, lo_cap=16)
    dev = torch.device("cuda")
    outs = []
    for place in (lambda t: t.to(dev), lambda t: _unaligned(t, dev)):
        out = torch.empty(2, D, dtype=torch.float32, device=dev)
        pkg.mikv_compute_balancer(shape, place(q), place(k), out, new_workspace(shape, pkg.WS_BALANCER, 0))
        outs.append(out.cpu())
    assert torch.equal(outs[0], outs[1]) and not bool(outs[0].isnan().any())
    assert outs[0][0, 2] == 1.0 and outs[0][1, 3] == float("inf") and outs[0][1, 4] == 0.0
    want = torch.sqrt(q[0, 0, :, 1].float().abs().nan_to_num(0.0).amax() / k[0, 0, :, 1].float().abs().amax())
    assert outs[0][0, 1] == want


@pytest.mark.parametrize("n,n_demote", [(2, 2), (1023, 2), (1024, 1023), (1025, 600), (32767, 30000), (32768, 2),
                                        (32769, 32768), (40001, 20000)])
@pytest.mark.parametrize("kind", ["spread", "ties", "equal"])
def test_select_demote_rounds_and_ties(n, n_demote, kind):
    """Sizes around the block and the rounds of 32768 entries; scores drawn from a handful of values or all equal, so
    that the boundary falls among equal scores and the ids decide."""
    gen = torch.Generator().manual_seed(n + n_demote)
    B, H = 1, 2
    scores = torch.randn(B, H, n, generator=gen).exp() if kind == "spread" else \
        torch.randint(-2, 3, (B, H, n), generator=gen).float() * 0.5 if kind == "ties" else torch.full((B, H, n), -0.0)
    if kind == "ties":
        scores[0, 1, ::3] = -0.0
    ids = torch.stack([torch.randperm(n, generator=gen) - n // 2 for _ in range(H)]).view(B, H, n).int()
    dev = torch.device("cuda")
    for with_ids in (False, True):
        dem = torch.full((B, H, n_demote), -7, dtype=torch.int32, device=dev)
        kept = torch.full((B, H, n - n_demote), -7, dtype=torch.int32, device=dev)
        pkg.mikv_select_demote(scores.to(dev), n, n_demote, dem, kept, ids=ids.to(dev) if with_ids else None)
        rd, rk = oracle.select_demote(scores.numpy(), n_demote, ids.numpy() if with_ids else None)
        np.testing.assert_array_equal(dem.cpu().numpy(), rd)
        np.testing.assert_array_equal(kept.cpu().numpy(), rk)


@pytest.mark.parametrize("n_rows", [1, 3, 4, 5, 31, 32, 33, 70])
@pytest.mark.parametrize("aligned", [True, False], ids=["aligned", "unaligned"])
def test_gather_row_counts(n_rows, aligned):
    gen = torch.Generator().manual_seed(n_rows)
    B, Hkv, n_src = 2, 2, 90
    shape = pkg.Shape(B, Hkv, Hkv, 2, 32, hi_cap=n_rows + 1, lo_cap=16)
    k, v = _rand_bf16(B, Hkv, n_src, D, gen=gen), _rand_bf16(B, Hkv, n_src, D, gen=gen)
    sc = torch.rand(B, Hkv, n_src, generator=gen)
    rows = torch.stack([torch.randperm(n_src, generator=gen)[:n_rows] for _ in range(B * Hkv)]).view(B, Hkv, n_rows).int()
    dev = torch.device("cuda")
    place = (lambda t: t.to(dev)) if aligned else (lambda t: _unaligned(t, dev))
    cache = pkg.LayerCache(shape, device=dev)
    bad = rows.clone()
    bad[1, 1, 0] = n_src  # skipped
    pkg.mikv_gather_hi(cache, place(k), place(v), bad.to(dev), src_scores=sc.to(dev))
    ref = oracle.empty_cache(B, Hkv, D, 2, 32, n_rows + 1, 16)
    oracle.gather_hi(ref, bits16(k), bits16(v), rows.numpy(), src_scores=sc.numpy())
    for name in ("k_hi", "v_hi"):
        ref[name][1, 1, 0] = 0
        np.testing.assert_array_equal(bits16(getattr(cache, name)[:, :, :n_rows + 1]), ref[name])
    ref["hi_tok"][1, 1, 0] = ref["acc"][1, 1, 0] = 0
    np.testing.assert_array_equal(cache.hi_tok[:, :, :n_rows].cpu().numpy(), ref["hi_tok"][:, :, :n_rows])
    np.testing.assert_array_equal(cache.acc[:, :, :n_rows].cpu().numpy(), ref["acc"][:, :, :n_rows])


@pytest.mark.parametrize("bits,hi_bits,kch", [(2, 16, 0), (3, 8, 0), (2, 16, 64), (0, 16, 0)],
                         ids=["bf16", "coded", "per-channel", "evict"])
def test_build_zeroes_what_it_does_not_write(bits, hi_bits, kch, monkeypatch):
    """A build that zeroes only the rows it does not write leaves the same arrays as one that zeroes everything."""
    gen = torch.Generator().manual_seed(9)
    B, H, T = 2, 2, 333
    dev = torch.device("cuda")
    k, v = _rand_bf16(B, H, T, D, gen=gen).to(dev), _rand_bf16(B, H, T, D, gen=gen).to(dev)
    scores = torch.rand(B, H, T, generator=gen).to(dev)
    shape = pkg.shape_for_context(B, H, H, bits, 32, T, 0.2, 40, hi_bits=hi_bits, k_channel_group=kch)
    built = []
    for whole in (1 << 60, 0):
        monkeypatch.setattr(pkg, "FILL_WHOLE", whole)
        junk = torch.full((64 << 20,), 0xFF, dtype=torch.uint8, device=dev)  # what the allocator hands out next
        del junk
        cache = MixedPrecisionLayer.from_prefill(shape, k, v, scores, device=dev).cache
        built.append({n: t.clone() for n, t in vars(cache).items() if isinstance(t, torch.Tensor)})
    for name, want in built[0].items():
        got = built[1][name]
        as_bytes = lambda t: t.contiguous().view(torch.uint8) if t.numel() else t  # noqa: E731
        assert torch.equal(as_bytes(got), as_bytes(want)), name
