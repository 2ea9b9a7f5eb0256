"""Decode attention at the sizes where its launches are streamed (many KV heads or long caches): every number of CTAs
per head that the launch rule chooses (16 down to 1, and several heads per CTA), lengths around the edges of a 16-row
tile, rings of one row, caches without sink or without selected rows, all group sizes, both group modes, the
log-sum-exps, launches back to back in every overlap mode.  Tolerance of the outputs as everywhere: 1e-2 absolute + 1e-2
relative (bf16 output and bf16 softmax weights); log-sum-exp 1e-3 (scores are fp32 sums of 128 products, the weights
bf16: relative 2^-9 each, averaged over the rows)."""

import numpy as np
import pytest
import torch

from oracle import sagekv_oracle as O
from helpers import bits

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2503_08879_b200 import binding
    return binding


# batch, KV heads, G, S, k_q, R (L = S + G*k_q + R + 1), overlap, pooled
CASES = [
    (1, 8, 4, 4, 2015, 128, 2, 0),      # 8193 rows: 16 CTAs per head
    (1, 4, 7, 4, 580, 131, 0, 0),       # 4196 rows, seven heads
    (2, 8, 8, 0, 512, 0, 1, 0),         # 4097 rows: the window is the last token alone, in a tile of its own
    (3, 8, 4, 3, 700, 12, 2, 0),        # 2816 rows: whole tiles
    (6, 8, 4, 5, 250, 10, 0, 0),        # 1016 rows
    (12, 8, 1, 4, 400, 111, 2, 0),      # one query head per KV head
    (10, 8, 2, 0, 100, 56, 1, 0),       # 257 rows: one row beyond a tile
    (9, 8, 8, 16, 0, 239, 2, 0),        # nothing selected: sink and window
    (20, 8, 4, 4, 60, 10, 0, 0),        # 255 rows: one short of a tile
    (40, 8, 4, 4, 61, 8, 2, 0),         # more heads than CTAs: several whole heads per CTA
    (75, 4, 4, 1, 4, 14, 1, 0),         # 32 rows: fewer tiles than warps
    (80, 4, 2, 0, 3, 9, 2, 0),          # one tile
    (5, 8, 4, 4, 1003, 24, 0, 1),       # pooled: every head sees every selected row
    (1, 8, 4, 4, 8100, 90, 2, 1),
]


@pytest.mark.parametrize("Bt,Hkv,G,S,k_q,R,overlap,pooled", CASES)
def test_streamed_launches_match_the_oracle(B, Bt, Hkv, G, S, k_q, R, overlap, pooled):
    H, n_sel = G * Hkv, k_q if pooled else G * k_q
    L = S + n_sel + R + 1
    gen = torch.Generator(device="cuda").manual_seed(L + Bt)
    rnd = lambda *s: torch.randn(*s, generator=gen, device="cuda").to(torch.bfloat16)
    layers, rows = 2, L + 3                                       # rows beyond L are not the call's
    Kc, Vc = rnd(layers, Bt, Hkv, rows, 128), rnd(layers, Bt, Hkv, rows, 128)
    step = torch.full((layers, 1), R, dtype=torch.int32, device="cuda")       # the next slot is the last of the ring
    q, kn, vn = rnd(3, layers, Bt, H, 128), rnd(3, layers, Bt, Hkv, 128), rnd(3, layers, Bt, Hkv, 128)
    out = torch.zeros_like(q)
    lse = torch.zeros(3, layers, Bt, H, device="cuda")
    ref_K, ref_V = bits(Kc), bits(Vc)
    sk = B.SageKV(H, Hkv, 128, Bt, max_ctx=max(L, 64), max_len=L)
    sk.set_overlap(overlap)
    B.sagekv_set_group_mode(sk.ctx, pooled)
    for t in range(3):                                            # the last one appends nothing
        for l in range(layers):
            st = B.CacheState(S, k_q, n_sel, R, R + 1, L, step[l].data_ptr())
            new = (kn[t, l], vn[t, l]) if t < 2 else (None, None)
            B.sagekv_decode_attn(sk.ctx, q[t, l], *new, Kc[l], Vc[l], st, out[t, l], lse[t, l])
    torch.cuda.synchronize()
    assert sk.status() == 0
    assert step.flatten().tolist() == [R + 2] * layers
    got, got_lse = out.float().cpu().numpy().astype(np.float64), lse.cpu().numpy()
    for l in range(layers):
        for b in sorted({0, Bt // 2, Bt - 1}):
            rk, rv, s = ref_K[l, b, :, :L], ref_V[l, b, :, :L], R
            for t in range(3):
                new = (bits(kn[t, l, b]), bits(vn[t, l, b])) if t < 2 else (None, None)
                if pooled:
                    ref, ref_lse, s = O.decode_step_pooled(bits(q[t, l, b]), *new, rk, rv, s, S, k_q, R)
                else:
                    ref, ref_lse, s = O.decode_step(bits(q[t, l, b]), *new, rk, rv, s, S, k_q, R)
                assert np.all(np.abs(got[t, l, b] - ref) <= 1e-2 + 1e-2 * np.abs(ref)), (l, b, t)
                assert np.all(np.abs(got_lse[t, l, b] - ref_lse) <= 1e-3 + 1e-3 * np.abs(ref_lse)), (l, b, t)
        for b in range(Bt):                                       # the appended rows and nothing else
            for t in range(2):
                slot = S + n_sel + (R + t) % (R + 1)
                ref_K[l, b, :, slot], ref_V[l, b, :, slot] = bits(kn[t, l, b]), bits(vn[t, l, b])
    assert np.array_equal(bits(Kc), ref_K) and np.array_equal(bits(Vc), ref_V)
    sk.close()
