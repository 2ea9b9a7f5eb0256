"""Which kernel a selection takes, on both sides of every line of the rule for rows of 8193 to 16384 scores: few and many kept scores,
up to and beyond one CTA per SM, with and without a gather, many static rows beside it, a histogram behind the rows; and of that for the
large selections' instance that leaves room for the static rows' kernel.  The lines are where one way became slower than the other when
measured; results are the same, bit-exact against the oracle."""

import numpy as np
import pytest
import torch

from oracle import sagekv_oracle as O
from helpers import bits, kernels_of

pytestmark = pytest.mark.gpu

SHORT, CLUSTER, GENERAL = "select_short_kernel", "select_compact_kernel", "select_general_kernel"


def select(rows, E, k, S, R, G, hint, gather, kernel):
    from paper_2503_08879_b200 import binding as B
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    H = {"half": n_sm // 2, "one": n_sm, "more": n_sm + 8, "13/10": 13 * n_sm // 10 + 4, "two": 2 * n_sm, "three": 3 * n_sm, "3+": 3 * n_sm + 8}.get(rows, rows)
    H -= H % G
    Hkv, N = H // G, S + E + R + 1
    gen = torch.Generator(device="cuda").manual_seed(E + k)
    sk = B.SageKV(H, Hkv, 128, 1, max_ctx=N, max_len=S + G * k + R + 1)
    sk.set_select_hint(hint)
    scores = torch.exp(1.5 * torch.randn(H, sk.score_stride(N, S, R), generator=gen, device="cuda") - 12)
    if gather:
        K = torch.randint(-9999, 9999, (1, 1, N, 128), generator=gen, device="cuda", dtype=torch.int16).view(torch.bfloat16).expand(1, Hkv, N, 128)
        cache = sk.new_layer(S, R, G * k)
        names = kernels_of(lambda: sk.select_compact(scores, K, K, S, R, G * k, cache))
        idx = cache.indices()[0]
    else:
        idx = torch.full((1, H, k), -1, dtype=torch.int32, device="cuda")
        names = kernels_of(lambda: B.sagekv_select_topk(sk.ctx, scores, scores.stride(0), E, k, idx))
        idx = idx[0] + S
    assert sk.status() == 0
    assert names[-1].startswith(kernel) and names[:-1] in ([], ["copy_static_kernel"]), names
    some = sorted({0, H // 2, H - 1})
    want = O.select(scores[some, :E].cpu().numpy(), k, S)
    assert np.array_equal(idx[some].cpu().numpy(), want)
    if gather:
        for i, h in enumerate(some):
            j = S + h % G * k
            assert np.array_equal(bits(cache.Kc[0, h // G, j:j + k]), bits(K[0, 0])[want[i]])
        last = torch.cat([K[0, 0, :S], K[0, 0, S + E:]])
        got = torch.cat([cache.Vc[0, -1, :S], cache.Vc[0, -1, S + G * k:cache.state.len]])
        assert torch.equal(got.view(torch.int16), last.view(torch.int16))
    sk.close()
    return names


@pytest.mark.parametrize("rows,E,k,R,kernel", [
    (640, 8192, 256, 20, SHORT), ("one", 8193, 256, 20, SHORT), ("more", 8193, 256, 20, CLUSTER), ("one", 16384, 40, 20, SHORT),
    ("more", 16384, 40, 20, CLUSTER), ("half", 16384, 512, 20, SHORT), ("more", 16384, 257, 20, SHORT), (400, 8193, 512, 124, SHORT),
    ("one", 16384, 384, 125, SHORT), ("one", 16384, 385, 125, CLUSTER), (96, 16384, 512, 125, SHORT), (112, 16384, 512, 125, CLUSTER),
    (192, 16384, 512, 125, SHORT), ("13/10", 9000, 257, 125, CLUSTER), ("13/10", 9000, 512, 125, CLUSTER), ("13/10", 16384, 513, 125, SHORT),
    (32, 16385, 512, 20, SHORT), ("one", 16385, 64, 20, CLUSTER), (16, 33000, 2049, 20, GENERAL)])
def test_with_a_gather(rows, E, k, R, kernel):               # 3 + R + 1 static rows: 128 are copied along by one CTA per row
    select(rows, E, k, 3, R, 4, 0, True, kernel)


@pytest.mark.parametrize("rows,E,k,kernel", [
    ("more", 14336, 256, SHORT), ("two", 14336, 256, SHORT), ("two", 14337, 256, CLUSTER), ("three", 16384, 256, SHORT), ("3+", 9000, 256, CLUSTER),
    ("3+", 9000, 257, SHORT)])
def test_without_a_gather(rows, E, k, kernel):
    select(rows, E, k, 0, 20, 1, 0, False, kernel)


@pytest.mark.parametrize("rows,S,R,k,kernel", [(80, 1999, 2000, 256, SHORT), (80, 2000, 2000, 256, CLUSTER), (80, 2000, 2000, 513, SHORT),
                                                     (112, 300, 300, 512, SHORT), (160, 64, 191, 300, SHORT), (160, 64, 192, 300, CLUSTER)])
def test_many_static_rows(rows, S, R, k, kernel):
    names = select(rows, 9000, k, S, R, 4, 0, True, kernel)
    assert names[0] == "copy_static_kernel", names


@pytest.mark.parametrize("rows,E,k,kernel", [("half", 14337, 1500, SHORT), ("one", 14337, 128, SHORT), ("one", 16384, 129, CLUSTER), ("more", 16384, 40, CLUSTER),
                                             ("more", 14337, 600, CLUSTER), (16, 16385, 40, CLUSTER)])
def test_with_a_histogram_behind_the_rows(rows, E, k, kernel):
    select(rows, E, k, 3, 20, 4, 1, True, kernel)


@pytest.mark.parametrize("rows,E,k,S,R,kernel", [
    (32, 17000, 8192, 2048, 2047, GENERAL + "<true>"), (32, 17000, 8193, 2048, 2047, GENERAL + "<false>"), (32, 50002, 2100, 600, 449, GENERAL + "<true>"),
    (32, 60002, 4300, 2048, 2048, GENERAL + "<false>"),
    (8, 50002, 2100, 2048, 2048, GENERAL + "<false>"), (32, 100001, 4096, 2048, 2048, GENERAL + "<false>"), (32, 50002, 2100, 4, 20, GENERAL + "<false>")])
def test_large_selections_beside_static_rows(rows, E, k, S, R, kernel):
    select(rows, E, k, S, R, 1, 0, True, kernel)
