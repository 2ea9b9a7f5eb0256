"""Score step at the edges of the first pass's tiles (16 tokens), warps (48) and CTAs (384), for several group sizes, and of the
second pass's rounds: 8192 scores of a slice (a slice is that long where there are more rows than the device takes at once), 16384
where the histogram is left behind the row.  Rows sum to 1 and nothing behind them is written.  Tolerance as everywhere: relative
1e-3 (bf16 products summed in fp32 over 128 terms, approximate exponentials)."""

import numpy as np
import pytest
import torch

from oracle import sagekv_oracle as O
from helpers import HINT_WORDS, bits, hint_of

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


@pytest.mark.parametrize("E", [8188, 8191, 8192, 8193, 16387])
def test_rounds_of_the_second_pass(E):
    from paper_2503_08879_b200 import binding as B
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    Hkv, G, S, R = 4, 8, 3, 5
    H, N = Hkv * G, S + E + R + 1
    Bt = (4 * n_sm + H - 1) // H                                 # four slices per SM: one per row
    gen = torch.Generator(device="cuda").manual_seed(E)
    K = torch.randn(Bt, Hkv, N, 128, generator=gen, device="cuda").to(torch.bfloat16)
    q = (2 * torch.randn(Bt, H, 128, generator=gen, device="cuda")).to(torch.bfloat16)
    sk = B.SageKV(H, Hkv, 128, Bt, max_ctx=N, max_len=64)
    buf = torch.full((Bt * H, (E + 3) // 4 * 4 + 4), 7.5, device="cuda")
    sk.score(q, K, S, R, scores=buf)
    torch.cuda.synchronize()
    assert (buf[:, E:] == 7.5).all() and sk.status() == 0
    assert ((buf[:, :E].double().sum(1) - 1).abs() < 1e-4).all()
    for b in (0, Bt - 1):
        np.testing.assert_allclose(buf[b * H:(b + 1) * H, :E].cpu().numpy().astype(np.float64),
                                   O.score(bits(q[b]), bits(K[b]), S, R), rtol=1e-3, atol=1e-30)
    sk.close()


@pytest.mark.parametrize("E", [131068, 131070, 131072, 131073, 131079, 262147])
def test_rounds_of_the_second_pass_with_the_histogram(E):
    from paper_2503_08879_b200 import binding as B
    S, R, H = 3, 5, 2
    N = S + E + R + 1
    gen = torch.Generator(device="cuda").manual_seed(E)
    K = torch.randn(1, 1, N, 128, generator=gen, device="cuda").to(torch.bfloat16)
    q = (2 * torch.randn(1, H, 128, generator=gen, device="cuda")).to(torch.bfloat16)
    sk = B.SageKV(H, 1, 128, 1, max_ctx=N, max_len=64)
    sk.set_select_hint(1)
    buf = torch.full((H, sk.score_stride(N, S, R) + 4), 7.5, device="cuda")
    sk.score(q, K, S, R, scores=buf)
    torch.cuda.synchronize()
    got, E4 = buf.cpu().numpy(), (E + 3) // 4 * 4
    np.testing.assert_allclose(got[:, :E].astype(np.float64), O.score(bits(q[0]), bits(K[0]), S, R), rtol=1e-3, atol=1e-30)
    assert np.array_equal(got[:, E4:E4 + HINT_WORDS].view(np.uint32), hint_of(got[:, :E], E))
    assert (got[:, E:E4] == 7.5).all() and (got[:, E4 + HINT_WORDS:] == 7.5).all() and sk.status() == 0
    sk.close()
