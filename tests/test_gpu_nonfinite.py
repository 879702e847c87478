"""Coordinates that are no numbers in the tile code (bucket sizes that are no power of two, vectors shorter than a
tile, ragged tails): a NaN, and an infinity in its own infinite scale, have level 0 and no sign, as has every
other coordinate of a bucket with an infinite scale."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_1610_02132_b200 import inputs as I
from parity_util import gpu_encode, scales_from_message

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,d", [(1000, 128), (3 * 4032 + 17, 96), (31, 32), (2 * 4096, 4064)])
@pytest.mark.parametrize("s", [1, 3, 15, 255])
@pytest.mark.parametrize("norm", [O.NORM_L2, O.NORM_MAX])
@pytest.mark.parametrize("code", [O.CODE_FIXED, O.CODE_ELIAS, O.CODE_ELIAS_DENSE])
def test_nan_and_infinity_have_level_zero(n, d, s, norm, code):
    g = I.gaussian(n, 0.01, seed=3)
    r = np.random.default_rng(n)
    g[r.integers(0, n, 1 + n // 200)] = np.nan
    g[r.integers(0, n, 1 + n // 900)] = r.choice([np.inf, -np.inf])
    big, info, st, _ = gpu_encode(torch.from_numpy(g).cuda(), d, s, norm, code, 7, 1, 2)
    assert st == 0
    msg = big[: info[2]].cpu().numpy()
    A = scales_from_message(msg, info, n, d, s, code)
    ref, ref_info = O.encode(np.where(np.isfinite(g), g, np.float32(0.0)), d, s, norm, code, 7, 1, 2, A_ext=A)
    assert info == ref_info and np.array_equal(msg, ref)
