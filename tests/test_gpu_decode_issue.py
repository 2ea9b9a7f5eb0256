"""Decode attention with the cache brought in whole, on both sides of the line between the ninth warp asking for the copies alone and all
nine sharing them: few and many tiles per CTA, one row beyond and short of a tile, V tiles that wait for a slot, every overlap mode.
Checks and tolerances of the streamed launches' test."""

import pytest

from test_gpu_decode_stream import B, test_streamed_launches_match_the_oracle as check  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("overlap", [0, 1, 2])
@pytest.mark.parametrize("Bt,Hkv,G,S,k_q,R", [(1, 1, 4, 4, 20, 27), (1, 2, 8, 4, 60, 90), (1, 8, 4, 4, 90, 148), (1, 8, 4, 4, 250, 20),
                                              (1, 8, 4, 4, 470, 144), (4, 4, 7, 4, 270, 130), (1, 1, 2, 4, 1300, 200), (2, 8, 4, 1, 60, 14)])
def test_resident_launches(B, Bt, Hkv, G, S, k_q, R, overlap):  # noqa: F811
    check(B, Bt, Hkv, G, S, k_q, R, overlap, 0)
