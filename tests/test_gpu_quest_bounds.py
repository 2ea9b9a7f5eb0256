"""Block bounds at the edges of the kernel's 16-block tiles and 64-block CTAs, for every group size, on summaries as
sagekv_quest_build leaves them and on arrays that are no minima and maxima (the formula holds for those too), with
infinities and zeros.  Tolerance: 128 fp32 additions of exact products, 128 * 2^-24 < 1e-5 of the sum of their magnitudes."""

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("G", [1, 2, 3, 4, 7, 8])
@pytest.mark.parametrize("n_blocks,ordered,special", [(1, True, False), (15, True, False), (16, True, False), (17, False, False),
                                                      (63, False, False), (64, True, True), (65, True, False), (127, True, True), (128, False, True), (300, True, False)])
def test_bounds_match_the_formula(G, n_blocks, ordered, special):
    from paper_2503_08879_b200 import binding as B
    Bt, Hkv = 2, 3
    gen = torch.Generator(device="cuda").manual_seed(n_blocks * 16 + G)
    rnd = lambda *s: torch.randn(*s, generator=gen, device="cuda").to(torch.bfloat16)
    a, b, q = rnd(Bt, Hkv, n_blocks, 128), rnd(Bt, Hkv, n_blocks, 128), rnd(Bt, Hkv * G, 128)
    kmin, kmax = (torch.minimum(a, b), torch.maximum(a, b)) if ordered else (a, b)
    q[:, 0, ::5] = 0
    if special:
        kmin[0, 1, n_blocks // 2, 3] = float("-inf")
        kmax[1, 2, n_blocks - 1, 127] = float("inf")
        q[:, Hkv * G - 1, 3] = -1.0
    q = q.contiguous()
    sk = B.SageKV(Hkv * G, Hkv, 128, Bt, max_ctx=16 * n_blocks + 1, max_len=64)
    stride = n_blocks + 5
    out = torch.full((Bt * Hkv * G, stride), 7.5, device="cuda")
    B.sagekv_quest_bounds(sk.ctx, q, kmin, kmax, n_blocks, out, stride)
    torch.cuda.synchronize()
    f = lambda t: t.double().cpu().numpy()
    qv = f(q).reshape(Bt, Hkv, G, 1, 128)
    with np.errstate(invalid="ignore"):
        lo, hi = qv * f(kmin)[:, :, None], qv * f(kmax)[:, :, None]
        terms = np.fmax(lo, hi)
        ref, mag = terms.sum(-1) / np.sqrt(128.0), np.abs(terms).sum(-1) / np.sqrt(128.0)
        got = out[:, :n_blocks].cpu().numpy().astype(np.float64).reshape(ref.shape)
        fine = np.isfinite(ref)
        assert np.all(np.abs(got - ref)[fine] <= 1e-5 * mag[fine])
    assert np.array_equal(got[~fine], ref[~fine], equal_nan=True)
    assert (out[:, n_blocks:] == 7.5).all()
    sk.close()
