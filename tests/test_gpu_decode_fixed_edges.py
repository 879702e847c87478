"""The fixed-width decoder at the edges of its chunks (512 coordinates a warp), its groups of four messages and its CTAs:
sums and steps bit for bit against the oracle, in flat form and through a bucket map."""
import pytest

from oracle import oracle as O
from paper_1610_02132_b200 import inputs as I
from parity_util import decode_parity, encode_parity
from test_gpu_policy import run_case

pytestmark = pytest.mark.gpu


# one scale per chunk and several, every field width; remainders of chunk, lane and group; with 8-bit levels the CTA grows
# at 8 and 16 chunks per SM (148)
@pytest.mark.parametrize("n,d,s,K", [(511, 512, 255, 1), (512, 512, 255, 5), (513, 512, 15, 4), (4096 + 16, 1024, 15, 3), (4095, 96, 15, 6),
                                     (512 * 1184 - 1, 2048, 255, 4), (512 * 1185, 512, 255, 2), (512 * 2369 + 3, 32, 255, 3),
                                     (512 * 9, 4096, 1, 7), (512 * 9 - 500, 64, 1, 8), (8191, 512, 3, 9), (8193, 160, 3, 4)])
def test_sums_and_steps(n, d, s, K):
    sent = [encode_parity(I.gaussian(n, 1.0, seed=w), d, s, O.NORM_MAX, O.CODE_FIXED, 7, 3, w) for w in range(min(K, 3))]
    decode_parity([sent[k % 3][0] for k in range(K)], [sent[k % 3][1] for k in range(K)], n, d, s, O.CODE_FIXED, eta=0.05,
                  x0=I.gaussian(n, 1.0, seed=9))


# buckets that lie off 16-byte boundaries and short ones: chunks that go out in whole lines beside others
@pytest.mark.parametrize("d,s", [(512, 255), (512, 15), (1024, 255), (2048, 3), (128, 255)])
def test_buckets_through_a_map(d, s):
    run_case([16384, 10001, 7, 12288, 20002, 10240], d, s, O.NORM_MAX, O.CODE_FIXED, K=5)
