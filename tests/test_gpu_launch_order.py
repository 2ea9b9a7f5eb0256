"""What a call finds when the kernel directly before it on the stream has written its inputs, where the selection reads them
while its own static rows are copied by a kernel beside it (by clusters, and by single CTAs); alone, and with calls of another
context put on the same stream from a second thread, between a call's launches too.  And a decode that reads its cache ahead, behind two select calls that
run ahead.  Bit-exact against the same calls one at a time."""

import threading

import pytest
import torch

from helpers import kernels_of

pytestmark = pytest.mark.gpu

Bt, Hkv, G, k_q, S, R = 2, 4, 4, 300, 600, 3000                  # 3601 static rows per head: copied beside the selection
H = Hkv * G


@pytest.fixture(scope="module")
def B():
    from paper_2503_08879_b200 import binding
    return binding


def inputs(gen, E):
    N = S + E + R + 1
    rnd = lambda *s: torch.randn(*s, generator=gen, device="cuda").to(torch.bfloat16)
    return rnd(Bt, Hkv, N, 128), rnd(Bt, Hkv, N, 128), torch.rand(Bt * H, (E + 3) // 4 * 4, generator=gen, device="cuda")


class Selection:
    def __init__(self, B, seed, E, kernel):
        gen = torch.Generator(device="cuda").manual_seed(seed)
        self.sets = [inputs(gen, E) for _ in range(3)]
        self.sk = B.SageKV(H, Hkv, 128, Bt, max_ctx=S + E + R + 1, max_len=S + G * k_q + R + 1)
        self.now = [torch.empty_like(x) for x in self.sets[0]]
        self.cache = self.sk.new_layer(S, R, G * k_q)
        self.want = []
        for i in range(3):
            self.write(i)
            torch.cuda.synchronize()
            self.select()
            torch.cuda.synchronize()
            self.want.append([x.clone() for x in (self.cache.idx, self.cache.Kc, self.cache.Vc)])
        names = kernels_of(self.select)
        assert names[0] == "copy_static_kernel" and names[1].startswith(kernel) and len(names) == 2, names

    def write(self, i):
        for x, y in zip(self.now, self.sets[i]):
            torch.add(y, 0, out=x)                               # a kernel, scores last: the selection needs them first

    def select(self):
        K, V, scores = self.now
        self.sk.select_compact(scores, K, V, S, R, G * k_q, self.cache)

    def rounds(self, n, bad):
        for t in range(n):
            i = t * t % 3
            self.write(i)
            self.select()
            bad += sum((x != y).any() for x, y in zip((self.cache.idx, self.cache.Kc, self.cache.Vc), self.want[i]))
            for x in (self.cache.idx, self.cache.Kc, self.cache.Vc):
                x.zero_()


ROWS = pytest.mark.parametrize("E,kernel", [(25001, "select_compact_kernel"), (12001, "select_short_kernel"), (3001, "select_short_kernel")])


@ROWS
def test_inputs_written_directly_before(B, E, kernel):
    s, bad = Selection(B, 1, E, kernel), torch.zeros((), dtype=torch.int64, device="cuda")
    s.rounds(60, bad)
    torch.cuda.synchronize()
    assert int(bad) == 0 and s.sk.status() == 0
    s.sk.close()


@ROWS
def test_another_context_on_the_same_stream(B, E, kernel):
    s, bad = Selection(B, 2, E, kernel), torch.zeros((), dtype=torch.int64, device="cuda")
    n2, k2 = 16500, 40                                           # short selections from candidate lists, which release early
    sk = B.SageKV(8, 2, 128, 1, max_ctx=n2, max_len=4 + 4 * k2 + 8)
    sk.set_select_hint(2, 4 * k2)
    sk.set_select_overlap(2)
    K, q = torch.randn(1, 2, n2, 128, device="cuda").to(torch.bfloat16), torch.randn(1, 8, 128, device="cuda").to(torch.bfloat16)
    scores, caches = sk.new_scores(n2, 4, 7), [sk.new_layer(4, 7, 4 * k2) for _ in range(2)]
    sk.score(q, K, 4, 7, scores)
    torch.cuda.synchronize()
    stop, errors = threading.Event(), []

    def other():
        try:
            while not stop.is_set():
                for _ in range(20):
                    for cache in caches:
                        sk.select_compact(scores, K, K, 4, 7, 4 * k2, cache)
                torch.cuda.current_stream().synchronize()
        except Exception as e:                                   # (shown by the assertion below)
            errors.append(e)

    t = threading.Thread(target=other)
    t.start()
    try:
        s.rounds(60, bad)
    finally:
        stop.set()
        t.join()
    torch.cuda.synchronize()
    assert not errors and int(bad) == 0 and s.sk.status() == 0 and sk.status() == 0
    assert torch.equal(caches[0].idx, caches[1].idx) and torch.equal(caches[0].Kc, caches[1].Kc)
    s.sk.close()
    sk.close()


@pytest.mark.parametrize("kq2,heads", [(20, 1), (300, 2), (1000, 8)])
def test_decode_behind_two_select_calls_that_run_ahead(B, kq2, heads):
    n, s0, r0, layers = 16500, 4, 60, 2
    gen = torch.Generator(device="cuda").manual_seed(kq2)
    rnd = lambda *s: torch.randn(*s, generator=gen, device="cuda").to(torch.bfloat16)
    sk = B.SageKV(4 * heads, heads, 128, 1, max_ctx=n, max_len=s0 + 4 * kq2 + r0 + 1)
    sk.set_select_hint(2, 4 * kq2)
    K, V = rnd(layers, 1, heads, n, 128), rnd(layers, 1, heads, n, 128)
    q, kn, vn = rnd(layers, 1, 4 * heads, 128), rnd(layers, 1, heads, 128), rnd(layers, 1, heads, 128)
    scores = [sk.score(q[l], K[l], s0, r0) for l in range(layers)]
    caches, out = [sk.new_layer(s0, r0, 4 * kq2) for _ in range(layers)], torch.empty_like(q)

    def calls(between=lambda: None):
        for l in range(layers):
            sk.select_compact(scores[l], K[l], V[l], s0, r0, 4 * kq2, caches[l])
            between()
        for l in range(layers):
            sk.decode_attn(q[l], kn[l], vn[l], caches[l], out[l])
            between()

    sk.set_select_overlap(2)
    sk.set_overlap(2)
    calls(torch.cuda.synchronize)
    want = out.clone()
    bad = torch.zeros((), dtype=torch.int64, device="cuda")
    for _ in range(50):
        for c in caches:
            c.Kc.fill_(3.0)
            c.Vc.fill_(float("nan"))
        out.zero_()
        calls()
        bad += (out != want).any()
    torch.cuda.synchronize()
    assert int(bad) == 0 and sk.status() == 0
    sk.close()
