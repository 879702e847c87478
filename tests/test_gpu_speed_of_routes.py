"""Calls that a rule of a dispatch, or a kernel's split of the work, must not leave behind others of the same size: ratios of
times of one and the same run, with room for noise."""
import pytest
import torch

import paper_1610_02132_b200 as Q
from oracle import oracle as O
from paper_1610_02132_b200 import inputs as I
from test_gpu_relative_speed import decode, time_of

pytestmark = pytest.mark.gpu

L2, MAX, FIXED, ELIAS, DENSE = O.NORM_L2, O.NORM_MAX, O.CODE_FIXED, O.CODE_ELIAS, O.CODE_ELIAS_DENSE


def encode(g, d, s, norm, code):
    n, status = g.numel(), Q.new_status()
    out = torch.empty(Q.qsgd_message_capacity(n, d, s, code), dtype=torch.uint8, device="cuda")
    info = torch.zeros(4, dtype=torch.int64, device="cuda")
    ws = torch.empty(Q.qsgd_workspace_bytes(n, d, s, code), dtype=torch.uint8, device="cuda")
    return lambda: Q.qsgd_encode(g, d, s, norm, code, 7, 0, 0, out, info, ws, status)


def test_elias_encode_of_mostly_small_values_with_many_levels():
    """22 levels against 15, of which messages are hardly shorter."""
    g = I.gaussian_mixture_device(40 * 2 ** 20, seed=3)
    fewer, more = time_of(*(encode(g, 512, s, L2, ELIAS) for s in (15, 22)), repeats=4)
    assert more < 1.55 * fewer                             # 1.34; 1.76 by tiles


def test_encodes_of_more_ctas_grow_no_faster_than_their_length():
    """Four times the coordinates, with so many CTAs that what each does to find its place must not grow along."""
    n, d, s = 2 ** 28, 2080, 16
    g = I.gaussian_device(4 * n, 1.0, seed=3)
    less, more = time_of(*(encode(g[:m], d, s, L2, DENSE) for m in (n, 4 * n)), repeats=1, replays=4)
    assert more < 4.4 * less                               # 4.0; 4.8 where every CTA reads the sums of all groups



def test_short_strings_where_long_ones_are_shared_by_warps():
    """Eight peers' strings of mostly small values against seventeen peers', too many to be shared."""
    n, d, s = 15792, 4096, 255
    eight, many = time_of(*(decode(n, d, s, L2, ELIAS, K, lambda w: I.gaussian_mixture_device(n, seed=w)) for K in (8, 17)))
    assert eight < 0.48 * many                             # 0.42; 0.54 where first parts share schedulers


def test_one_peer_against_eight():
    """A CTA with a single string has its tables to make all the same."""
    n, d, s = 3871, 4096, 15
    one, eight = time_of(*(decode(n, d, s, L2, DENSE, K) for K in (1, 8)))
    assert one < 0.9 * eight


@pytest.mark.parametrize("n,d,K,other", [(6973756, 480, 4, 512), (2753820, 96, 7, 128)])
def test_many_levels_in_buckets_of_many_sizes(n, d, K, other):
    """A lane per string against buckets a little longer, which another decoder reads or another split fits."""
    here, there = time_of(*(decode(n, m, 255, L2, ELIAS, K) for m in (d, other)))
    assert here < 1.05 * there


@pytest.mark.parametrize("d,s,K", [(128, 64, 64), (64, 100, 32)])
def test_a_few_chunks_more_than_a_round_of_warps(d, s, K):
    """Fixed-width decode of 8-bit levels: 32 chunks of 512 coordinates on each of 148 SMs, and an eighth more."""
    n = 512 * 148 * 32
    round_, more = time_of(*(decode(m, d, s, MAX, FIXED, K) for m in (n, n + n // 8)))
    assert more < 1.55 * round_                            # 1.3; 1.9 where a few SMs get all of the rest
