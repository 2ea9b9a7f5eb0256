"""The calls in their default modes where their launches do not simply follow one another: captured into a CUDA graph behind
copies, behind a join of two streams, on a stream forked off in between and behind a memset; and from two threads at once, each
with a context and a stream of its own.  Bit-exact against the same calls one at a time."""

import threading

import pytest
import torch

pytestmark = pytest.mark.gpu

Hkv, G, N, S, R, k = 4, 4, 6000, 4, 64, 444
H, E = Hkv * G, N - S - R - 1


class Layer:
    def __init__(self, B, seed):
        gen = torch.Generator(device="cuda").manual_seed(seed)
        rnd = lambda *s: torch.randn(*s, generator=gen, device="cuda").to(torch.bfloat16)
        self.sk = B.SageKV(H, Hkv, 128, 1, max_ctx=N, max_len=S + k + R + 1)
        self.K0, self.V0, self.q = rnd(1, Hkv, N, 128), rnd(1, Hkv, N, 128), rnd(1, H, 128)
        self.K, self.V = torch.zeros_like(self.K0), torch.zeros_like(self.V0)
        self.kn, self.vn = rnd(1, Hkv, 128), rnd(1, Hkv, 128)
        self.scores, self.cache, self.out = self.sk.new_scores(N, S, R).zero_(), self.sk.new_layer(S, R, k), torch.zeros_like(self.q)
        self.results = (self.scores, self.cache.idx, self.cache.Kc, self.cache.Vc, self.cache.step, self.out)

    def score(self):
        self.sk.score(self.q, self.K, S, R, self.scores)

    def select(self):
        self.sk.select_compact(self.scores, self.K, self.V, S, R, k, self.cache)

    def decode(self):
        self.sk.decode_attn(self.q, self.kn, self.vn, self.cache, self.out)

    def clear(self):
        for x in (self.K, self.V, *self.results):
            x.zero_()


@pytest.fixture(scope="module")
def B():
    from paper_2503_08879_b200 import binding
    return binding


@pytest.mark.parametrize("kind", ["copies", "join", "fork", "memset"])
def test_captured_calls(B, kind):
    lay, side = Layer(B, 1), torch.cuda.Stream()

    def work():
        cur = torch.cuda.current_stream()
        if kind == "join":                                       # two streams write the inputs
            side.wait_stream(cur)
            with torch.cuda.stream(side):
                torch.add(lay.V0, 0, out=lay.V)
            torch.add(lay.K0, 0, out=lay.K)
            cur.wait_stream(side)
        else:                                                    # copy nodes
            lay.V.copy_(lay.V0)
            lay.K.copy_(lay.K0)
        lay.score()
        if kind == "fork":                                       # the selection on a stream of its own, work beside it
            side.wait_stream(cur)
            with torch.cuda.stream(side):
                lay.select()
            lay.V0.float().sum()
            cur.wait_stream(side)
        else:
            lay.select()
        lay.decode()
        if kind == "memset":
            lay.out.zero_()
            lay.decode()

    work()
    torch.cuda.synchronize()
    want = [x.clone() for x in lay.results]
    assert int(want[4]) == (2 if kind == "memset" else 1) and want[5].any()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        work()
    for _ in range(5):
        lay.clear()
        graph.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(x, y) for x, y in zip(lay.results, want))
    assert lay.sk.status() == 0
    del graph
    lay.sk.close()


def test_two_threads_with_a_stream_each(B):
    layers, errors = [Layer(B, seed) for seed in (2, 3)], []
    want = []
    for lay in layers:
        lay.K.copy_(lay.K0)
        lay.V.copy_(lay.V0)
        lay.score(), lay.select(), lay.decode()
        torch.cuda.synchronize()
        want.append([x.clone() for x in lay.results])

    def work(lay, ref):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                bad = torch.zeros((), dtype=torch.int64, device="cuda")
                for _ in range(50):
                    lay.clear()
                    torch.add(lay.V0, 0, out=lay.V)
                    torch.add(lay.K0, 0, out=lay.K)
                    lay.score(), lay.select(), lay.decode()
                    bad += sum((x != y).any() for x, y in zip(lay.results, ref))
                torch.cuda.current_stream().synchronize()
                assert int(bad) == 0 and lay.sk.status() == 0
        except BaseException as e:                               # (shown by the assertion below)
            errors.append(e)

    threads = [threading.Thread(target=work, args=a) for a in zip(layers, want)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors
    for lay in layers:
        lay.sk.close()
