"""Elias encodes of so many CTAs that the sums of their runs are added up over two levels of groups: messages bit for bit against the
oracle, by tiles and by teams, on both sides of the line."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1610_02132_b200 import inputs as I
from parity_util import encode_parity

pytestmark = pytest.mark.gpu

MANY = 4 * 64 * 64


@pytest.mark.parametrize("n,d,s,norm,code", [
    (MANY * 2080, 2080, 16, O.NORM_MAX, O.CODE_ELIAS_DENSE),             # tiles of one bucket: the last with one level of groups
    ((MANY + 64) * 2080 + 1, 2080, 16, O.NORM_MAX, O.CODE_ELIAS_DENSE),  # two levels, a last group of one CTA
    ((MANY + 1) * 8192 - 31, 32, 1, O.NORM_MAX, O.CODE_ELIAS),           # teams
])
def test_messages(n, d, s, norm, code):
    g = np.tile(I.gaussian(2 ** 20, 1.0, seed=3), -(-n // 2 ** 20))[:n]
    g[n // 2: n // 2 + 4096 * d // 4] = 0.0
    encode_parity(g, d, s, norm, code, 7, 3, 1)
