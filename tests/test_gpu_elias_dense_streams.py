"""The dense code read by streams (a lane per run of buckets and peer): well-formed messages bit for bit against the oracle in
every form of the call, with symbols of every length, short and long buckets, few and many peers; and messages with one peer's
strings malformed: flagged, nothing written out of bounds, and where only one string is bad the other buckets come out right."""
import numpy as np
import pytest
import torch

import paper_1610_02132_b200 as Q
from oracle import oracle as O
from paper_1610_02132_b200 import inputs as I
from parity_util import decode_parity, encode_parity
from test_gpu_elias_decoders import worker

pytestmark = pytest.mark.gpu

L2, MAX, DENSE = O.NORM_L2, O.NORM_MAX, O.CODE_ELIAS_DENSE

# (buckets, coordinates missing in the last, d, s, norm, K)
SHAPES = [
    (9000, 27, 32, 15, MAX, 5), (4200, 1, 96, 32, MAX, 16), (8300, 63, 64, 1, L2, 4), (2100, 255, 512, 64, MAX, 32), (2800, 1, 512, 15, L2, 12),
    (4200, 0, 160, 3, L2, 8), (2000, 4095, 4096, 64, L2, 17), (50000, 0, 128, 15, MAX, 1), (1000, 2047, 2080, 64, L2, 32), (4200, 5, 480, 7, MAX, 8),
]


def gradient(n, d, w):
    g = I.gaussian(n, 1.0, seed=50 + w)
    if w % 3 == 1:
        g[:: d] = 40.0                                    # most levels 0, some the longest
    if w % 3 == 2:
        g[np.random.default_rng(w).random(n) < 0.9] = 0.0
    return g


@pytest.mark.parametrize("B,missing,d,s,norm,K", SHAPES)
def test_sums_of_well_formed_messages(B, missing, d, s, norm, K):
    n = B * d - missing
    sent = [encode_parity(gradient(n, d, w), d, s, norm, DENSE, 7, 3, w) for w in range(min(K, 3))]
    msgs, infos = [sent[k % 3][0] for k in range(K)], [sent[k % 3][1] for k in range(K)]
    x0 = I.gaussian(n, 1.0, seed=9)
    decode_parity(msgs, infos, n, d, s, DENSE, eta=0.05, x0=x0)
    decode_parity(msgs, infos, n, d, s, DENSE, eta=-0.05, x0=x0, tables_first=True)
    words = [torch.tensor(i, dtype=torch.int64, device="cuda") for i in infos]
    acc, status = torch.empty(n, device="cuda"), Q.new_status()
    assert worker(lambda: Q.qsgd_decode_accumulate_packed(msgs, words, n, d, s, DENSE, acc, status)) == "decode_elias_dense"


@pytest.mark.parametrize("B,missing,d,s,norm,K", [c for c in SHAPES if c[0] * c[2] < 2 * 10 ** 6])
def test_malformed_messages(B, missing, d, s, norm, K):
    n = B * d - missing
    good, info = O.encode(gradient(n, d, 0), d, s, norm, DENSE, 7, 0, 0)
    table = O.message_table(good, info, n, d)
    noise = good.copy()
    noise[: info[1]] = np.random.default_rng(1).integers(0, 256, info[1], dtype=np.uint8)
    ones, zeros = good.copy(), good.copy()
    ones[: info[1]] = 255
    zeros[: info[1]] = 0
    cut, swapped, above = table.copy(), table.copy(), table.copy()
    cut[B // 2] -= 3
    swapped[[B // 3, B // 3 + 1]] = swapped[[B // 3 + 1, B // 3]]
    above[-1] += 1 << 33
    one, bad = good.copy(), B // 2                             # ones behind the scale of one string
    for t in range(int(table[bad]) + 32, int(table[bad]) + 56):
        one[4 * (t // 32) + 3 - (t % 32) // 8] |= 1 << (7 - t % 8)
    ref = O.decode_accumulate([good] * K, [table] * K, n, d, s, DENSE)[1]
    words = torch.tensor(info, dtype=torch.int64, device="cuda")
    for msg, tab, only in ((good, table, -1), (noise, table, None), (ones, table, None), (zeros, table, None), (good, cut, None),
                           (good, swapped, None), (good, above, None), (one, table, bad)):
        bufs = []
        for m, t in ((msg, tab), (good, table)):
            m = m.copy()
            m[info[1]: info[1] + t.nbytes] = t.view(np.uint8)
            bufs.append(torch.from_numpy(np.concatenate([m, np.zeros(64, np.uint8)])).cuda())
        acc = torch.full((n + 256,), 7.0, device="cuda")
        status = Q.new_status()
        Q.qsgd_decode_accumulate_packed([bufs[i] for i in [1] * (K - 1) + [0]], [words] * K, n, d, s, DENSE, acc[:n], status)
        assert bool((acc[n:] == 7.0).all())
        assert (int(status.item()) != 0) == (only != -1)
        if only is not None:
            same = acc[:n].cpu().numpy().view(np.uint32) == ref.view(np.uint32)
            if only >= 0:
                same[only * d: (only + 1) * d] = True
            assert same.all()
