"""Selections that the prefilter does not take (more than 2048 kept scores of a long row): every row length that changes a slice's last
vector or the number of its iterations, scores staged and not, equal scores, few values, infinities, NaN, and the other rows copied
along and beside.  Bit-exact against the oracle."""

import pytest

from test_gpu_select_short import check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("E,k", [(33000, 2100), (40001, 5000), (65535, 65535), (65538, 40000), (131071, 2049), (131073, 3000), (300003, 9000)])
@pytest.mark.parametrize("kind", ["softmax", "few", "equal", "infinite", "nan", "side by side", "close"])
def test_many_kept_of_long_rows(E, k, kind):
    check(E, k, kind, 2, 3, 1, 1, E)


@pytest.mark.parametrize("Hkv,G,E,k,S,R", [(2, 2, 50000, 2500, 600, 700), (24, 1, 33003, 2300, 4, 128), (4, 1, 600001, 2200, 0, 0)])
def test_with_the_other_rows_along_and_beside(Hkv, G, E, k, S, R):
    check(E, k, "softmax", S, R, Hkv, G, E + R)
