"""The checked build skips a static row whose token lies outside the extent it was given: the row of the cache stays as it
was, the other rows arrive, the status word says so.  (The memory behind it holds every position: nothing is out of bounds.)"""

import ctypes as C

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_ctx", [131, 130, 100, 90, 30])
def test_rows_outside_the_extent_are_skipped(n_ctx):
    from paper_2503_08879_b200 import binding as B
    if B.lib.sagekv_checked_build() != 1:
        pytest.skip("runs on the checked build (test_gpu_checked_build.py)")
    S, E, R, n_sel = 33, 60, 37, 7                               # tokens 0..32 and 93..130, rows 0..32 and 40..77
    K = torch.randn(S + E + R + 1, 128, device="cuda").to(torch.bfloat16)
    V = torch.randn_like(K)
    Kc = torch.full((S + n_sel + R + 1, 128), 7.0, dtype=torch.bfloat16, device="cuda")
    Vc, words = Kc.clone(), torch.full((2,), 9, dtype=torch.int32, device="cuda")
    words[1] = 0
    p = lambda t: C.c_void_p(t.data_ptr())
    code = B.lib.sagekv_checked_copy_static(p(K), p(V), p(Kc), p(Vc), n_ctx, S, E, R, n_sel, p(words), p(words[1:]),
                                            C.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert code == 0
    torch.cuda.synchronize()
    want_K, want_V = torch.full_like(Kc, 7.0), torch.full_like(Kc, 7.0)
    for r in range(S + R + 1):
        tok, row = (r, r) if r < S else (E + r, n_sel + r)
        if tok < n_ctx:
            want_K[row], want_V[row] = K[tok], V[tok]
    assert torch.equal(Kc, want_K) and torch.equal(Vc, want_V)
    assert words.tolist() == [0, 2 if n_ctx < S + E + R + 1 else 0]
