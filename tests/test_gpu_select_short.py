"""Selection from rows that fit one CTA's registers: at the edges of the row lengths its instances take (2048, 4096, 8192, 16384 and
32768 scores, with 4, 8, 16, 32 and 64 per thread), of a thread's and a warp's share, and of the numbers of kept scores at which the way
changes (a thread's or a vector's maximum as a group, every score by itself).  Rows of equal scores, few values, infinities, NaN,
large scores side by side.  Indices and gathered rows bit-exact against the oracle."""

import numpy as np
import pytest
import torch

from oracle import sagekv_oracle as O
from helpers import bits

pytestmark = pytest.mark.gpu

KINDS = ["softmax", "few", "equal", "infinite", "nan", "side by side", "close"]


def rows_of(kind, H, E, rng):
    x = rng.standard_normal((H, E)).astype(np.float32)
    if kind == "softmax":
        x = np.exp(1.5 * x - 12)
    elif kind == "few":
        x = np.round(x)
    elif kind == "equal":
        x[:] = -0.0
        x[:, ::3] = 0.0
    elif kind == "infinite":
        x[x < 1] = -np.inf
        x[:, E // 2] = np.inf
    elif kind == "nan":                                          # never kept while there are numbers
        x[:, rng.random(E) < 0.1] = np.nan
    elif kind == "side by side":
        x[:, E // 3: E // 3 + E // 8] += 8
    elif kind == "close":
        x = np.float32(1) + np.abs(x) * np.float32(2 ** -20)
    return x


def check(E, k, kind, S, R, Hkv, G, seed):
    from paper_2503_08879_b200 import binding as B
    rng = np.random.default_rng(seed)
    H, N, k = Hkv * G, S + E + R + 1, min(k, E)
    x = rows_of(kind, H, E, rng)
    if kind == "nan":
        k = min(k, int((~np.isnan(x)).sum(axis=1).min()))
    buf = torch.full((H, (E + 3) // 4 * 4 + 4), float("inf"), device="cuda")
    buf[:, :E] = torch.from_numpy(x).cuda()
    gen = torch.Generator(device="cuda").manual_seed(seed)
    K, V = (torch.randn(1, Hkv, N, 128, generator=gen, device="cuda").to(torch.bfloat16) for _ in range(2))
    sk = B.SageKV(H, Hkv, 128, 1, max_ctx=N, max_len=S + G * k + R + 1)
    cache = sk.select_compact(buf, K, V, S, R, G * k)
    top = torch.full((1, H, k), -1, dtype=torch.int32, device="cuda")
    B.sagekv_select_topk(sk.ctx, buf, buf.stride(0), E, k, top)
    torch.cuda.synchronize()
    assert sk.status() == 0
    want = O.select(x, k, S)
    idx = cache.indices()[0].cpu().numpy()
    assert np.array_equal(idx, want) and np.array_equal(top[0].cpu().numpy(), want - S)
    got = [bits(t[0]) for t in cache.cache()]
    for a, b in zip(got, O.compact(bits(K[0]), bits(V[0]), idx, S, R)):
        assert np.array_equal(a, b)
    sk.close()


@pytest.mark.parametrize("E", [1, 3, 4, 127, 129, 2047, 2048, 2049, 4096, 4097, 8191, 8193, 16383, 16385, 32767, 32768, 32769])
def test_row_lengths(E):
    for i, kind in enumerate(KINDS):
        check(E, max(1, E // (50 + 7 * i)), kind, 2, 3, 1, 2, E + i)


@pytest.mark.parametrize("E", [1000, 3000, 8184, 12001, 30002])
@pytest.mark.parametrize("part", ["one", "thread", "thread + 1", "vector", "vector + 1", "most", "all"])
def test_how_many_are_kept(E, part):
    per = {1000: 1, 3000: 2, 8184: 4, 12001: 8, 30002: 16}[E]   # vectors of four scores a thread has
    k = {"one": 1, "thread": E // (8 * per), "thread + 1": E // (8 * per) + 1, "vector": E // 8, "vector + 1": E // 8 + 1,
         "most": E - 1, "all": E}[part]
    for i, kind in enumerate(("softmax", "few", "side by side")):
        check(E, k, kind, 1, 2, 1, 2, 7 * E + i)


@pytest.mark.parametrize("Hkv,G,E,k,S,R", [(1, 1, 4000, 40, 40, 700), (2, 4, 8000, 300, 1000, 1100), (1, 8, 16000, 512, 2048, 2047),
                                           (40, 4, 3000, 70, 4, 128), (20, 8, 9000, 33, 2, 60)])
def test_with_the_other_rows_along_and_beside(Hkv, G, E, k, S, R):
    check(E, k, "softmax", S, R, Hkv, G, E + R)
