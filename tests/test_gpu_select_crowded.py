"""Selection where many scores crowd around the cut: the second histogram over the cut's bin (from 49 candidates on), equal
scores inside it, keys one unit apart, outliers that stretch the first histogram; and rows long enough for several
iterations of the passes over a slice.  Indices bit-exact against the oracle."""

import numpy as np
import pytest
import torch

from oracle import sagekv_oracle as O

pytestmark = pytest.mark.gpu


def select(rows, k_q, hint=0):
    from paper_2503_08879_b200 import binding as B
    H, E = rows.shape
    sk = B.SageKV(H, H, 128, 1, max_ctx=E, max_len=64)
    buf = torch.zeros(H, (E + 3) // 4 * 4, device="cuda")
    buf[:, :E] = torch.from_numpy(rows).cuda()
    idx = torch.full((1, H, k_q), -1, dtype=torch.int32, device="cuda")
    B.sagekv_select_topk(sk.ctx, buf, buf.stride(0), E, k_q, idx)
    torch.cuda.synchronize()
    assert sk.status() == 0
    sk.close()
    assert np.array_equal(idx[0].cpu().numpy(), O.select(rows, k_q, 0))


@pytest.mark.parametrize("crowd", [47, 48, 49, 200, 511, 513])
@pytest.mark.parametrize("spread", ["equal", "ulps", "narrow"])
def test_crowded_cut(crowd, spread):
    rng = np.random.default_rng(crowd)
    H, E, k_q = 4, 20011, 300
    rows = (rng.random((H, E)) * 1e-6).astype(np.float32)
    for h in range(H):
        at = rng.permutation(E)
        above = at[: k_q - crowd // 2] if crowd // 2 < k_q else at[:0]
        rows[h, above] = rng.random(above.size, dtype=np.float32) + 1.0
        mid = at[above.size: above.size + crowd]
        base = np.float32(0.5)
        if spread == "equal":
            rows[h, mid] = base
        elif spread == "ulps":
            rows[h, mid] = (base.view(np.int32) + rng.integers(0, 40, crowd).astype(np.int32)).view(np.float32)
        else:
            rows[h, mid] = base + rng.random(crowd, dtype=np.float32) * np.float32(1e-3)
        rows[h, at[-1]] = 1e4
    select(rows, k_q)


@pytest.mark.parametrize("H,E,k_q", [(1, 140003, 900), (2, 600001, 1500), (40, 70001, 64)])
def test_long_slices(H, E, k_q):
    rng = np.random.default_rng(E)
    rows = np.exp(rng.standard_normal((H, E)) * 2).astype(np.float32)
    rows[:, 1000:1400] = rows[:, 1000:1001]                     # equal scores in a run
    select(np.ascontiguousarray(rows / rows.sum(axis=1, keepdims=True)), k_q)
