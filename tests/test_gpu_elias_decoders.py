"""Each Elias decoder on shapes that its line gives to it, which the kernel that did the work is checked against: a
change of a line that takes a shape elsewhere fails here. Well-formed messages, bit for bit against the oracle in every
form of the call; and messages with one peer's strings malformed: flagged, nothing written out of bounds, and where
only one string is bad the other buckets come out right."""
import numpy as np
import pytest
import torch

import paper_1610_02132_b200 as Q
from oracle import oracle as O
from paper_1610_02132_b200 import inputs as I
from parity_util import decode_parity, encode_parity

pytestmark = pytest.mark.gpu

L2, MAX, ELIAS = O.NORM_L2, O.NORM_MAX, O.CODE_ELIAS

# more than 24 K strings for a lane each; (decoder, buckets, coordinates missing in the last, d, s, norm, K, long gaps in every other peer)
SHAPES = [
    ("decode_elias", 15000, 27, 32, 15, MAX, 9, True), ("decode_elias", 2700, 1, 96, 3, MAX, 17, True),
    ("decode_elias", 6700, 0, 160, 15, L2, 4, True), ("decode_elias", 3200, 223, 224, 7, MAX, 8, True),
    ("decode_elias", 3100, 247, 256, 15, MAX, 8, True), ("decode_elias", 1500, 509, 512, 15, L2, 17, True),
    ("decode_elias", 800, 1017, 1024, 1, MAX, 32, False), ("decode_elias", 2800, 1, 2048, 15, L2, 9, True),
    ("decode_elias", 1030, 5, 512, 15, MAX, 24, True), ("decode_elias", 1600, 3, 4096, 15, MAX, 16, False),
    ("decode_elias_bytes", 40000, 27, 32, 15, MAX, 1, True), ("decode_elias_bytes", 1000, 1, 32, 3, L2, 30, False),
    ("decode_elias_bytes", 13000, 63, 64, 15, MAX, 2, True), ("decode_elias_bytes", 5200, 0, 96, 7, MAX, 5, True),
    ("decode_elias_bytes", 1600, 13, 160, 3, MAX, 17, False),
    # decided by the strings: 0.25 to 0.7 bits per coordinate behind the scale, ranges shorter and longer than a bucket
    ("decode_elias_bytes", 16600, 0, 256, 1, L2, 16, False), ("decode_elias_bytes", 19000, 99, 224, 1, L2, 16, False),
    ("decode_elias_bytes", 14700, 250, 288, 1, L2, 16, False),
    ("decode_elias_fields", 25000, 95, 96, 255, L2, 1, False), ("decode_elias_fields", 5000, 3, 480, 16, MAX, 5, False),
    ("decode_elias_fields", 800, 31, 32, 255, MAX, 32, False), ("decode_elias_fields", 3200, 0, 256, 255, L2, 8, False),
    ("decode_elias_teams", 3, 7, 4096, 255, MAX, 5, False), ("decode_elias_teams", 1000, 0, 64, 3, L2, 24, True),
    # few buckets of a size that is no power of two: lists of 29 and of 19 entries, rounded up
    ("decode_elias_sparse", 7000, 0, 928, 1, L2, 2, None), ("decode_elias_sparse", 7000, 3, 608, 1, L2, 2, None),
    ("decode_elias_sparse", 1000, 4001, 4096, 1, L2, 8, None), ("decode_elias_sparse", 7000, 9, 1024, 1, L2, 4, None),
]


def worker(call):
    """The Elias decoder that did the work of a call: the others only stand down. The call's launches queue up behind
    other work, so that their times hold no time of the host."""
    other = torch.empty(2 ** 28, device="cuda")
    Q.qsgd_profile_enable(True)
    try:
        Q.qsgd_profile_collect()
        for _ in range(4):
            other.zero_()
        call()
        torch.cuda.synchronize()
    finally:
        Q.qsgd_profile_enable(False)
    ms = {name: v[0] for name, v in Q.qsgd_profile_collect().items() if name.startswith("decode_elias") and v[1]}
    return max(ms, key=ms.get)


def gradient(n, d, long_gaps, w):
    if long_gaps is None:
        return I.sparse_laplace(n, 1e-3, 0.6, seed=w)
    if not long_gaps or w % 2 == 0:
        return I.gaussian(n, 1.0, seed=50 + w)
    g = I.sparse_laplace(n, 1e-3, 0.3, seed=50 + w)
    g[np.random.default_rng(w).random(n) < 0.97] = 0.0
    g[n // 3: n // 3 + 3 * d] = 0.0
    return g


@pytest.mark.parametrize("name,B,missing,d,s,norm,K,long_gaps", SHAPES)
def test_sums_of_well_formed_messages(name, B, missing, d, s, norm, K, long_gaps):
    n = B * d - missing
    sent = [encode_parity(gradient(n, d, long_gaps, w), d, s, norm, ELIAS, 7, 3, w) for w in range(min(K, 3))]
    msgs, infos = [sent[k % 3][0] for k in range(K)], [sent[k % 3][1] for k in range(K)]
    x0 = I.gaussian(n, 1.0, seed=9)
    decode_parity(msgs, infos, n, d, s, ELIAS, eta=0.05, x0=x0)
    decode_parity(msgs, infos, n, d, s, ELIAS, eta=-0.05, x0=x0, tables_first=True)
    words = [torch.tensor(i, dtype=torch.int64, device="cuda") for i in infos]
    acc, status = torch.empty(n, device="cuda"), Q.new_status()
    assert worker(lambda: Q.qsgd_decode_accumulate_packed(msgs, words, n, d, s, ELIAS, acc, status)) == name


@pytest.mark.parametrize("name,B,missing,d,s,norm,K,long_gaps", [c for c in SHAPES if c[1] * c[3] < 5 * 10 ** 6])
def test_malformed_messages(name, B, missing, d, s, norm, K, long_gaps):
    n = B * d - missing
    good, info = O.encode(gradient(n, d, long_gaps, 0), d, s, norm, ELIAS, 7, 0, 0)
    table = O.message_table(good, info, n, d)
    noise = good.copy()
    noise[: info[1]] = np.random.default_rng(1).integers(0, 256, info[1], dtype=np.uint8)
    ones = good.copy()
    ones[: info[1]] = 255
    cut, swapped, above = table.copy(), table.copy(), table.copy()
    cut[B // 2] -= 3
    swapped[[B // 3, B // 3 + 1]] = swapped[[B // 3 + 1, B // 3]]
    above[-1] += 1 << 33
    one = good.copy()                                          # ones behind the scale of one string that is long enough
    bad = int(np.flatnonzero(np.diff(table.astype(np.int64)) > 64)[0])
    for t in range(int(table[bad]) + 32, int(table[bad]) + 56):
        one[4 * (t // 32) + 3 - (t % 32) // 8] |= 1 << (7 - t % 8)
    ref = O.decode_accumulate([good] * K, [table] * K, n, d, s, ELIAS)[1]
    words = torch.tensor(info, dtype=torch.int64, device="cuda")
    for msg, tab, only in ((good, table, -1), (noise, table, None), (ones, table, None), (good, cut, None), (good, swapped, None),
                           (good, above, None), (one, table, bad)):
        bufs = []
        for m, t in ((msg, tab), (good, table)):
            m = m.copy()
            m[info[1]: info[1] + t.nbytes] = t.view(np.uint8)
            bufs.append(torch.from_numpy(np.concatenate([m, np.zeros(64, np.uint8)])).cuda())
        order = [1] * (K - 1) + [0]
        acc = torch.full((n + 256,), 7.0, device="cuda")
        status = Q.new_status()
        ran = worker(lambda: Q.qsgd_decode_accumulate_packed([bufs[i] for i in order], [words] * K, n, d, s, ELIAS, acc[:n], status))
        assert bool((acc[n:] == 7.0).all())
        if tab is not above:                                   # (whose strings count as long)
            assert ran == name
        assert (int(status.item()) != 0) == (only != -1)
        if only is not None:
            same = acc[:n].cpu().numpy().view(np.uint32) == ref.view(np.uint32)
            if only >= 0:
                same[only * d: (only + 1) * d] = True
            assert same.all()


@pytest.mark.parametrize("n,d,s,K,name", [(54272, 1024, 1, 4, "decode_elias_sparse"), (431883, 4096, 1, 1, "decode_elias_sparse"),
                                          (13345 * 480, 480, 1, 1, "decode_elias_sparse"), (57037, 1024, 1, 17, "decode_elias_teams")])
def test_short_strings_of_small_problems(n, d, s, K, name):
    """The sizes read off the pointers (a table right behind its payload) choose, in one launch."""
    sent = [encode_parity(I.gaussian_mixture(n, seed=w), d, s, L2, ELIAS, 7, 3, w) for w in range(min(K, 3))]
    msgs, infos = [sent[k % 3][0] for k in range(K)], [sent[k % 3][1] for k in range(K)]
    decode_parity(msgs, infos, n, d, s, ELIAS, eta=0.05)
    B = O.n_buckets(n, d)
    tables = [m[i[1]: i[1] + 8 * (B + 1)].view(torch.int64) for m, i in zip(msgs, infos)]
    acc, status, before = torch.empty(n, device="cuda"), Q.new_status(), Q.qsgd_launch_count()
    assert worker(lambda: Q.qsgd_decode_accumulate(msgs, tables, n, d, s, ELIAS, acc, status)) == name
    assert Q.qsgd_launch_count() == before + 1
