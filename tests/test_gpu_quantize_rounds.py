"""The bulk quantizer's rounds: a block of quantize_pack_kernel walks up to sixteen rounds of 16 rows when a call has many
rows, with the next round's rows in flight. Sizes around the ends of rounds and blocks, skipped rows in a later round;
codes, parameters and token ids of K and V bit for bit against the oracle on sampled heads, and nothing written past the
rows."""
import numpy as np
import pytest
import torch

import oracle
import paper_2402_18096_gb300 as pkg
from _cases import bits16

pytestmark = pytest.mark.gpu
D = 128
HEADS = (64, 8)  # with 512 heads a call of n rows has n / 16 * 512 rounds in all: 2, 3 and 16 a block at the sizes below
NAMES = ("k_codes", "v_codes", "k_params", "v_params", "lo_tok")


def _bytes(t):
    return t.contiguous().view(torch.uint8)


@pytest.mark.parametrize("n_rows", [65, 79, 80, 81, 112, 113, 127, 128, 129, 144, 593, 608, 767, 768, 769, 1025])
@pytest.mark.parametrize("bits,group", [(2, 32), (3, 64), (4, 128)])
def test_rounds_match_oracle(n_rows, bits, group):
    B, H = HEADS
    dev = torch.device("cuda")
    n_src, start = n_rows + 7, 5
    shape = pkg.Shape(B, H, H, bits, group, hi_cap=1, lo_cap=(start + n_rows + 33) // 16 * 16)
    gen = torch.Generator(device=dev).manual_seed(1000 * bits + n_rows)
    k, v = (torch.randn(B, H, n_src, D, generator=gen, device=dev).mul_(3).bfloat16() for _ in range(2))
    bal = torch.rand(H, D, generator=gen, device=dev) * 3 + 0.2
    rows = torch.rand(B, H, n_src, generator=gen, device=dev).argsort(-1)[:, :, :n_rows].int().contiguous()
    tok = torch.randint(0, 1 << 20, (B, H, n_src), generator=gen, device=dev, dtype=torch.int32)
    skipped = sorted({17, n_rows // 2, n_rows - 1})  # in the second, a middle and the last round
    rows[:, :, skipped] = torch.tensor([-1, n_src, n_src + 5], dtype=torch.int32, device=dev)[:len(skipped)]
    cache = pkg.LayerCache(shape, device=dev, balancer=bal)
    for name in NAMES:
        _bytes(getattr(cache, name)).fill_(0xA5)
    pkg.mikv_quantize_pack(cache, k, v, rows, start, src_tok=tok)

    whole = torch.ones(shape.lo_cap, dtype=torch.bool, device=dev)  # rows no call may touch
    whole[start:start + n_rows] = False
    whole[[start + i for i in skipped]] = True
    for name in NAMES:
        t = getattr(cache, name)
        assert bool((_bytes(t[:, :, whole]) == 0xA5).all()), name
    good = [i for i in range(n_rows) if i not in skipped]
    sl = [start + i for i in good]
    for b, h in [(0, 0), (17, 3), (40, 6), (B - 1, H - 1)]:
        ref = oracle.empty_cache(1, 1, D, bits, group, 1, shape.lo_cap)
        rr = rows[b:b + 1, h:h + 1].cpu().numpy().copy()
        rr[0, 0, skipped] = 0  # (the oracle takes valid rows only; these are not compared)
        oracle.quantize_pack(ref, bits16(k[b:b + 1, h:h + 1].cpu()), bits16(v[b:b + 1, h:h + 1].cpu()), rr, start,
                             balancer_=bal[h:h + 1].cpu().numpy(), src_tok=tok[b:b + 1, h:h + 1].cpu().numpy())
        for name in NAMES:
            got = getattr(cache, name)[b, h, sl].cpu()
            got = got.view(torch.int16).numpy().view(np.uint16) if got.dtype == torch.float16 else got.numpy()
            np.testing.assert_array_equal(got, ref[name][0, 0][sl], err_msg=f"{name} of head {b}, {h}")
