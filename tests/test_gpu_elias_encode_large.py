"""Elias encodes beyond the 1000 tiles of the small path, on both sides of the line between teams and tiles and where runs of
strings are added up over several groups of CTAs: whole messages bit for bit against the oracle, and a buffer too small for
the message left alone."""
import numpy as np
import pytest
import torch

import paper_1610_02132_b200 as Q
from oracle import oracle as O
from paper_1610_02132_b200 import inputs as I
from parity_util import encode_parity, gpu_encode

pytestmark = pytest.mark.gpu

L2, MAX, ELIAS, DENSE = O.NORM_L2, O.NORM_MAX, O.CODE_ELIAS, O.CODE_ELIAS_DENSE
N = 1000 * 4096


@pytest.mark.parametrize("n,d,s,norm,code", [
    (N + 1, 512, 255, L2, ELIAS), (N + 31, 480, 255, MAX, ELIAS), (N + 4095, 4096, 16, MAX, ELIAS), (N + 777, 512, 15, MAX, ELIAS),
    (N + 65, 96, 15, MAX, ELIAS), (N + 33, 32, 3, L2, ELIAS), (N + 4096, 4096, 1, MAX, ELIAS), (N + 9, 4064, 3, L2, ELIAS),
    (N + 1, 4096, 64, L2, DENSE), (N + 17, 32, 16, MAX, DENSE), (N + 2047, 2080, 255, MAX, DENSE), (N + 100, 512, 15, MAX, DENSE),
    (N + 3, 1056, 3, L2, DENSE), (N + 129, 128, 1, MAX, DENSE), (3 * N + 5, 64, 7, L2, ELIAS)])
def test_messages(n, d, s, norm, code):
    g = I.gaussian(n, 1.0, seed=3)
    g[n // 2: n // 2 + 3 * d] = 0.0                       # long gaps, whole empty buckets, single nonzeros at both ends
    g[n // 3: n // 3 + 2 * d: max(d // 2 - 1, 70)] = 5.0
    encode_parity(g, d, s, norm, code, 7, 3, 1)


@pytest.mark.parametrize("d,s,code", [(512, 15, ELIAS), (1024, 255, ELIAS), (4096, 64, DENSE)])
def test_a_buffer_too_small(d, s, code):
    n = N + 4097
    g = torch.from_numpy(I.gaussian(n, 1.0, seed=4)).cuda()
    _, info, st, _ = gpu_encode(g, d, s, L2, code, 7, 0, 0)
    assert st == 0
    for cap in (info[2] - 1, info[2] // 2):
        big, short, st, _ = gpu_encode(g, d, s, L2, code, 7, 0, 0, capacity=cap)
        assert st == Q.binding.DEV_CAPACITY and short == info
        assert np.all(big.cpu().numpy() == 0xAB)
