"""Decode attention around the line between the ninth warp asking for the copies alone and all nine sharing them: few and many tiles per CTA,
one row beyond and short of a tile, every overlap mode (in modes 1 and 2 some of these shapes are streamed).  Then the resident kernel's
instances by name, with V tiles that wait for a slot among them: there the first row that is replaced, the last of the cache, lies in such
a tile, and the second, the oldest of the window, in one that is there from the start.  Checks and tolerances of the streamed launches' test."""

import pytest
import torch

from helpers import kernels_of
from test_gpu_decode_stream import B, test_streamed_launches_match_the_oracle as check  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("overlap", [0, 1, 2])
@pytest.mark.parametrize("Bt,Hkv,G,S,k_q,R", [(1, 1, 4, 4, 20, 27), (1, 2, 8, 4, 60, 90), (1, 8, 4, 4, 90, 148), (1, 8, 4, 4, 250, 20),
                                              (1, 8, 4, 4, 470, 144), (4, 4, 7, 4, 270, 130), (1, 1, 2, 4, 1300, 200), (2, 8, 4, 1, 60, 14)])
def test_resident_launches(B, Bt, Hkv, G, S, k_q, R, overlap):  # noqa: F811
    check(B, Bt, Hkv, G, S, k_q, R, overlap, 0)


# S = 4, R = 200.  Behind the number of rows: tiles of the CTA that has most, its V tiles that wait
@pytest.mark.parametrize("Bt,Hkv,G,k_q,overlap,is_long,shared", [
    (1, 2, 8, 46, 0, False, False),      # 573 rows
    (1, 2, 8, 46, 1, False, False),
    (1, 8, 4, 205, 0, False, True),      # 1025
    (1, 8, 4, 205, 1, False, True),
    (1, 8, 4, 205, 2, False, True),
    (1, 8, 8, 360, 0, True, True),       # 3085: 25 tiles, none waits
    (3, 4, 4, 720, 1, True, True),
    (1, 2, 4, 720, 2, True, True),
    (1, 1, 8, 376, 0, True, True),       # 3213: 26, two
    (1, 1, 4, 752, 2, True, True),
    (1, 4, 8, 400, 2, True, True),       # 3405: 27, four
    (1, 1, 8, 400, 2, True, True),
    (3, 4, 4, 800, 0, True, False),
    (3, 4, 8, 400, 1, True, False),
    (5, 4, 8, 380, 1, True, False),      # 3245: clusters of six, 34 tiles, eighteen
    (17, 1, 8, 294, 0, True, False),     # 2557; from this many heads on the older costs hold
    (19, 1, 8, 102, 1, False, False),    # 1021
])
def test_instances(B, Bt, Hkv, G, k_q, overlap, is_long, shared):  # noqa: F811
    check(B, Bt, Hkv, G, 4, k_q, 200, overlap, 0)
    L = 4 + G * k_q + 201
    sk = B.SageKV(G * Hkv, Hkv, 128, Bt, max_ctx=L, max_len=L)
    sk.set_overlap(overlap)
    kv, q = torch.zeros(Bt, Hkv, L, 128, dtype=torch.bfloat16, device="cuda"), torch.zeros(Bt, G * Hkv, 128, dtype=torch.bfloat16, device="cuda")
    step, kv2, new, out = torch.zeros(1, dtype=torch.int32, device="cuda"), kv.clone(), kv[:, :, 0].contiguous(), torch.empty_like(q)
    state = B.CacheState(4, k_q, G * k_q, 200, 201, L, step.data_ptr())
    names = kernels_of(lambda: B.sagekv_decode_attn(sk.ctx, q, new, new, kv, kv2, state, out))
    assert names == ["decode_attn_kernel<%s, %s>" % (str(is_long).lower(), str(shared).lower())], names
    sk.close()
