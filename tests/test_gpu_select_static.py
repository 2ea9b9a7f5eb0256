"""select+compact where the sink, recent and last rows are many: from two rows per warp of the head's CTAs on (both sides
of that line, in the kernels for short rows, for long ones and for large selections) a kernel of their own copies them beside the selection.
Every hint and overlap mode, several layers back to back, row strides beyond 128 elements; and the shapes of the score row at which the
cluster size changes.  Bit-exact."""

import numpy as np
import pytest
import torch

from oracle import sagekv_oracle as O
from helpers import bits, kernels_of

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2503_08879_b200 import binding
    return binding


def run(B, Bt, Hkv, G, E, k_q, S, R, hint=0, overlap=0, pad=0, layers=3, kernels=()):
    H, N = Hkv * G, S + E + R + 1
    gen = torch.Generator(device="cuda").manual_seed(E + R)
    rnd = lambda *s: torch.randn(*s, generator=gen, device="cuda").to(torch.bfloat16)
    sk = B.SageKV(H, Hkv, 128, Bt, max_ctx=N, max_len=S + G * k_q + R + 1)
    sk.set_select_hint(hint, G * k_q)
    sk.set_select_overlap(overlap)
    lays = []
    for _ in range(layers):
        K, V = rnd(Bt, Hkv, N, 128 + pad)[..., :128], rnd(Bt, Hkv, N, 128 + pad)[..., :128]
        lay = dict(q=rnd(Bt, H, 128), K=K, V=V, scores=sk.new_scores(N, S, R), cache=sk.new_layer(S, R, G * k_q, spare_rows=2))
        lay["cache"].Kc.view(torch.int16).fill_(0x5A5A)
        lay["cache"].Vc.view(torch.int16).fill_(0x5A5A)
        lay["cache"].step.fill_(9)
        lays.append(lay)
    for lay in lays:
        sk.score(lay["q"], lay["K"], S, R, lay["scores"])
    for lay in lays:
        sk.select_compact(lay["scores"], lay["K"], lay["V"], S, R, G * k_q, lay["cache"])
    torch.cuda.synchronize()
    assert sk.status() == 0
    names = [] if not kernels else kernels_of(lambda: sk.select_compact(lay["scores"], lay["K"], lay["V"], S, R, G * k_q, lay["cache"]))
    assert len(names) == len(kernels) and all(n.startswith(k) for n, k in zip(names, kernels)), names
    for lay in lays:
        c = lay["cache"]
        assert int(c.step.item()) == 0
        rows = lay["scores"].view(Bt, H, -1)[..., :E].cpu().numpy()
        assert (c.Kc[:, :, c.state.len:].view(torch.int16) == 0x5A5A).all()
        for b in range(Bt):
            idx = c.indices()[b].cpu().numpy()
            assert np.array_equal(idx, O.select(rows[b], k_q, S))
            Kc, Vc = O.compact(bits(lay["K"][b]), bits(lay["V"][b]), idx, S, R)
            got = c.cache()
            assert np.array_equal(bits(got[0][b]), Kc) and np.array_equal(bits(got[1][b]), Vc)
    sk.close()


@pytest.mark.parametrize("Bt,Hkv,G,E,k_q,S,R,pad", [
    (1, 1, 1, 3000, 40, 40, 87, 0),      # (a short row takes as many CTAs as copy 128 to 257 rows along)
    (1, 1, 1, 3000, 40, 41, 214, 0),
    (1, 1, 1, 3000, 40, 41, 215, 8),
    (2, 4, 2, 5000, 300, 512, 900, 0),
    (1, 2, 4, 2001, 7, 0, 1500, 16),     # no sink
    (1, 2, 4, 2001, 7, 1500, 0, 0),      # no recent rows
    (1, 2, 7, 900, 900, 700, 699, 0),    # everything is kept
])
def test_many_static_rows(B, Bt, Hkv, G, E, k_q, S, R, pad):
    run(B, Bt, Hkv, G, E, k_q, S, R, pad=pad)


ALONG_LONG, ALONG_SHORT, ALONG_LARGE = (["select_%s_kernel" % n] for n in ("compact", "short", "general"))
BESIDE_LONG, BESIDE_SHORT, BESIDE_LARGE = (["copy_static_kernel"] + n for n in (ALONG_LONG, ALONG_SHORT, ALONG_LARGE))


@pytest.mark.parametrize("Bt,Hkv,G,E,k_q,S,R,pad,kernels", [
    (1, 1, 1, 40001, 40, 40, 87, 0, ALONG_LONG),         # 128 rows over a cluster of 8 x 16 warps: one per warp
    (1, 1, 1, 40001, 40, 41, 214, 0, ALONG_LONG),        # 256: two per warp
    (1, 1, 1, 40001, 40, 41, 215, 8, BESIDE_LONG),       # 257
    (1, 2, 4, 33001, 7, 0, 1500, 16, BESIDE_LONG),
    (1, 2, 4, 33001, 7, 1500, 0, 0, BESIDE_LONG),
    (1, 1, 1, 33003, 2100, 40, 215, 0, ALONG_LARGE),
    (1, 1, 1, 33003, 2100, 40, 216, 8, BESIDE_LARGE),
    (2, 16, 1, 33003, 2100, 600, 500, 0, BESIDE_LARGE),  # two CTAs and the copying one on an SM
    (4, 8, 4, 2000, 40, 2000, 47, 0, BESIDE_SHORT),      # short rows, one to sixteen vectors of four scores per thread
    (4, 8, 4, 4001, 40, 900, 47, 8, BESIDE_SHORT),
    (2, 8, 4, 8001, 300, 900, 147, 0, BESIDE_SHORT),     # four, with the histogram of every score
    (2, 8, 4, 8190, 40, 900, 147, 0, BESIDE_SHORT),      # and with that of the vectors' maxima
    (2, 8, 4, 12001, 300, 1100, 1047, 0, BESIDE_SHORT),  # eight
    (1, 8, 4, 16384, 33, 1100, 1047, 16, BESIDE_SHORT),
    (2, 8, 4, 30002, 300, 2, 100, 0, ALONG_SHORT),       # (sixteen: never beside)
])
def test_along_and_beside_by_kernel(B, Bt, Hkv, G, E, k_q, S, R, pad, kernels):
    run(B, Bt, Hkv, G, E, k_q, S, R, pad=pad, layers=2, kernels=kernels)


@pytest.mark.parametrize("hint,overlap", [(0, 0), (0, 2), (1, 0), (1, 1), (2, 0), (2, 1), (2, 2)])
@pytest.mark.parametrize("R", [127, 1100])
def test_modes_of_long_rows(B, hint, overlap, R):
    run(B, 1, 2, 4, 33003, 200, 4, R, hint=hint, overlap=overlap, layers=4)


@pytest.mark.parametrize("hint,overlap", [(0, 0), (0, 2), (1, 0), (1, 1), (2, 0), (2, 1), (2, 2)])
@pytest.mark.parametrize("R", [127, 1100])
def test_modes(B, hint, overlap, R):
    run(B, 1, 2, 4, 15003, 200, 4, R, hint=hint, overlap=overlap, layers=4)


@pytest.mark.parametrize("Bt,E,k_q", [(1, 512, 20), (1, 513, 20), (2, 16384, 100), (2, 16385, 100), (4, 33000, 300), (3, 9000, 257),
                                      (1, 65537, 512)])
def test_row_lengths(B, Bt, E, k_q):
    run(B, Bt, 8, 4, E, k_q, 3, 20, layers=1)


@pytest.mark.parametrize("Bt,Hkv,E,k_q", [(20, 8, 9000, 20), (5, 8, 16385, 100), (5, 8, 16385, 257), (3, 8, 32769, 30), (2, 8, 32769, 512), (1, 8, 65537, 1025),
                                          (1, 8, 65536, 300), (1, 8, 131073, 20)])
def test_cluster_sizes(B, Bt, Hkv, E, k_q):                      # one to eight CTAs
    run(B, Bt, Hkv, 4, E, k_q, 3, 20, layers=1, kernels=ALONG_LONG)
