"""The prefill importance repeats itself bit for bit: passes over several inputs back to back, at lengths of odd and even
numbers of tiles and with many short items per block, where the hand-over of tiles between the kernels' warps is
busiest. Every pass has to give the bits of the first one on the same inputs, and every KV head's scores have to sum to
G T (each query's weights sum to one)."""
import math

import numpy as np
import pytest
import torch

import mikv_inputs as mi
import oracle
import paper_2402_18096_gb300 as pkg
from paper_2402_18096_gb300.layer import workspace
from _cases import bits16
from test_gpu_prefill import _gpu_scores, prefill_rtol

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,Hq,Hkv,T,passes", [
    (1, 32, 8, 32768, 60), (1, 32, 8, 20001, 60), (4, 32, 32, 4096, 120),
    (30, 32, 32, 600, 400), (16, 32, 8, 257, 400), (8, 32, 32, 300, 400), (16, 32, 32, 128, 400), (40, 8, 8, 256, 400),
    (2, 40, 40, 777, 400), (1, 40, 40, 513, 400), (3, 32, 4, 999, 400),
], ids=lambda x: str(x))
def test_prefill_repeats(B, Hq, Hkv, T, passes):
    dev = torch.device("cuda")
    shape = pkg.Shape(B, Hq, Hkv, 2, 32, 1, 16)
    G, states = Hq // Hkv, []
    for seed in (T, T + 1):
        w = mi.Workload("pfr", B, Hq, Hkv, T, 1, 2, 32, 0.2, seed=seed)
        q, k = mi.prefill_queries(w, 0, dev), mi.prefill_kv(w, 0, dev)[0]
        out = torch.zeros(B, Hkv, T, device=dev)
        ws = workspace(pkg.mikv_workspace_bytes(shape, pkg.WS_PREFILL, T), dev)
        top = [bits16(x.abs().amax((0, 1, 2))[None].cpu()) for x in (q, k)]
        states.append((q, k, out, ws, prefill_rtol(*top, T, G)))
    first, wrong = [None, None], torch.zeros((), dtype=torch.int64, device=dev)
    for i in range(passes):
        n = int(i % 3 != 0)  # either input after itself and after the other
        q, k, out, ws, _ = states[n]
        pkg.mikv_prefill_scores(shape, q, k, out, ws)
        if first[n] is None:
            first[n] = out.clone()
        else:
            wrong += (out != first[n]).any()
    assert int(wrong) == 0, f"{int(wrong)} of {passes} passes differ from the first on the same inputs"
    for (_, _, _, ws, rtol), scores in zip(states, first):
        pkg.mikv_workspace_check(ws)
        np.testing.assert_allclose(scores.double().sum(-1).cpu().numpy(), G * T, rtol=rtol)


@pytest.mark.parametrize("B,Hq,Hkv,T", [
    (1, 40, 40, 513),   # one-tile items, more of them than blocks
    (3, 32, 4, 999),    # two-tile items in the pass over queries, one-tile items in the pass over keys
    (30, 8, 8, 600),    # two-tile items of an odd number of tiles: one is left alone, at the short end
    (1, 80, 80, 140),   # a last group of heads of another size
], ids=lambda x: str(x))
def test_prefill_items_match_oracle(B, Hq, Hkv, T):
    """The items of either size against the oracle, on the first and last head and one between."""
    w = mi.Workload("pfi", B, Hq, Hkv, T, 1, 2, 32, 0.2, seed=T + Hq)
    q, k, G = mi.prefill_queries(w, 0), mi.prefill_kv(w, 0)[0], Hq // Hkv
    got = _gpu_scores(w, q, k)
    for b, h in [(0, 0), (B // 2, Hkv // 2), (B - 1, Hkv - 1)]:
        qh, kh = bits16(q[b:b + 1, h * G:(h + 1) * G]), bits16(k[b:b + 1, h:h + 1])
        ref = oracle.prefill_scores(qh, kh, 1 / math.sqrt(128))[0, 0]
        np.testing.assert_allclose(got[b, h], ref, rtol=prefill_rtol(qh, kh, T, G), atol=1e-30)
