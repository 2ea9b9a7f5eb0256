"""Score step at the edges of the first pass's tiles (16 tokens), warps (48) and CTAs (384), and of the second pass's
rounds (8192 scores of a slice), for several group sizes; rows sum to 1 and nothing behind them is written.  Tolerance as
everywhere: relative 1e-3 (bf16 products summed in fp32 over 128 terms, approximate exponentials)."""

import numpy as np
import pytest
import torch

from oracle import sagekv_oracle as O
from helpers import bits

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("G", [1, 4, 7, 8])
@pytest.mark.parametrize("E", [1, 15, 16, 17, 47, 48, 49, 383, 384, 385, 767, 769, 8191, 8193])
def test_edges_match_the_oracle(E, G):
    from paper_2503_08879_b200 import binding as B
    Hkv, S, R = 2, 3, 5
    H, N = G * Hkv, S + E + R + 1
    gen = torch.Generator(device="cuda").manual_seed(E * 16 + G)
    K = torch.randn(1, Hkv, N, 128, generator=gen, device="cuda").to(torch.bfloat16)
    q = (2 * torch.randn(1, H, 128, generator=gen, device="cuda")).to(torch.bfloat16)
    K[:, :, :S] = K[:, :, S + E:] = float("inf")                # rows outside the eviction region are not read
    sk = B.SageKV(H, Hkv, 128, 1, max_ctx=N, max_len=64)
    buf = torch.full((H, (E + 3) // 4 * 4 + 4), 7.5, device="cuda")
    sk.score(q, K, S, R, scores=buf)
    torch.cuda.synchronize()
    K[:, :, :S] = K[:, :, S + E:] = 0
    got = buf[:, :E].cpu().numpy().astype(np.float64)
    np.testing.assert_allclose(got, O.score(bits(q[0]), bits(K[0]), S, R), rtol=1e-3, atol=1e-30)
    np.testing.assert_allclose(got.sum(axis=1), 1.0, atol=1e-4)
    assert (buf[:, E:] == 7.5).all() and sk.status() == 0
    sk.close()
