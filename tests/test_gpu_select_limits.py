"""Selections at the ends of their range: slices of many iterations that the prefilter does not take (their shared memory may
not grow with the slice) in every way such a launch comes about, and a selection too large for the shared memory, which is
refused before anything is written.  Bit-exact against the oracle."""

import numpy as np
import pytest
import torch

from oracle import sagekv_oracle as O
from test_gpu_select_static import run

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2503_08879_b200 import binding
    return binding


@pytest.mark.parametrize("H,E,k_q", [(8, 200000, 24000), (2, 1000000, 23000), (1, 13000001, 1000)])
def test_long_slices_without_the_prefilter(B, H, E, k_q):
    gen = torch.Generator(device="cuda").manual_seed(E)
    buf = torch.rand(H, (E + 3) // 4 * 4, generator=gen, device="cuda")
    idx = torch.full((1, H, k_q), -1, dtype=torch.int32, device="cuda")
    sk = B.SageKV(H, H, 128, 1, max_ctx=E, max_len=64)
    B.sagekv_select_topk(sk.ctx, buf, buf.stride(0), E, k_q, idx)
    torch.cuda.synchronize()
    assert sk.status() == 0
    sk.close()
    for h in sorted({0, H - 1}):
        assert np.array_equal(idx[0, h:h + 1].cpu().numpy(), O.select(buf[h:h + 1, :E].cpu().numpy(), k_q, 0))


def test_more_rows_than_sms_with_the_histogram_hint(B):
    Hkv, G, E, k_q, S, R = 20, 8, 1500001, 2000, 1, 2           # one CTA per row
    N, H = S + E + R + 1, 160
    gen = torch.Generator(device="cuda").manual_seed(3)
    K = torch.randn(1, 1, N, 128, generator=gen, device="cuda", dtype=torch.bfloat16).expand(1, Hkv, N, 128)
    sk = B.SageKV(H, Hkv, 128, 1, max_ctx=N, max_len=S + G * k_q + R + 1)
    sk.set_select_hint(1)
    scores = sk.new_scores(N, S, R).uniform_(generator=gen)     # no histogram behind them
    cache = sk.select_compact(scores, K, K, S, R, G * k_q)
    torch.cuda.synchronize()
    assert sk.status() == 0
    idx = cache.indices()[0].cpu().numpy()
    for h in (0, 159):
        assert np.array_equal(idx[h:h + 1], O.select(scores[h:h + 1, :E].cpu().numpy(), k_q, S))
    rows = torch.from_numpy(idx[159].astype(np.int64)).cuda()
    assert torch.equal(cache.Kc[0, 19, S + 7 * k_q: S + 8 * k_q], K[0, 0, rows])
    sk.close()


def test_a_single_cta_per_candidate_list(B):
    run(B, 1, 1, 1, 1600003, 64, 3, 5, hint=2, overlap=2, layers=2)


def test_too_large_a_selection_is_refused_before_anything_is_written(B):
    E, k_q, S, R = 200000, 26000, 4, 300                         # a window that is copied by a kernel of its own
    N = S + E + R + 1
    sk = B.SageKV(1, 1, 128, 1, max_ctx=N, max_len=S + k_q + R + 1)
    K = torch.ones(1, 1, N, 128, dtype=torch.bfloat16, device="cuda")
    scores, cache = torch.rand(1, E, device="cuda"), sk.new_layer(S, R, k_q)
    cache.step.fill_(9)
    with pytest.raises(B.SagekvError) as e:
        sk.select_compact(scores, K, K, S, R, k_q, cache)
    assert e.value.code == B.ERR_CUDA
    torch.cuda.synchronize()
    assert sk.status() == 0 and int(cache.step.item()) == 9 and cache.state.len == 0
    assert not cache.Kc.any() and not cache.Vc.any() and not cache.idx.any()
    sk.close()
