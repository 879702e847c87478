"""Elias Encode and Decode at the edges of their dispatch rules: problems read by teams of lanes (parts of a
string shorter and longer than a lane's least part, peers in several passes, codes on which a reader that
starts out of step stays out of step; long gaps, empty buckets and malformed strings among many strings) and encoded in
tiles (tiles of whole buckets, sizes around a tile, both sides of the line to the team kernels). Bit for bit against the
oracle. The decoders with a lane per string have their shapes in test_gpu_elias_decoders.py."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_1610_02132_b200 import inputs as I
from parity_util import decode_parity, encode_parity

pytestmark = pytest.mark.gpu

L2, MAX = O.NORM_L2, O.NORM_MAX
ELIAS, DENSE = O.CODE_ELIAS, O.CODE_ELIAS_DENSE


def run(n, d, s, norm, code, K, make=None):
    make = make or (lambda w: I.gaussian(n, 1.0, seed=50 + w))
    msgs, infos = [], []
    for w in range(K):
        m, info = encode_parity(make(w), d, s, norm, code, 7, 3, w)
        msgs.append(m)
        infos.append(info)
    x0 = I.gaussian(n, 1.0, seed=9)
    decode_parity(msgs, infos, n, d, s, code, eta=0.05, x0=x0)
    decode_parity(msgs, infos, n, d, s, code, eta=-0.05, x0=x0, tables_first=True)


@pytest.mark.parametrize("n,d,s,norm,code,K", [
    (32, 32, 1, L2, ELIAS, 1), (31, 32, 15, MAX, DENSE, 2),              # one string, shorter than a part
    (4096, 4096, 64, L2, DENSE, 8), (4064, 4064, 63, L2, DENSE, 3),      # 32 lanes a string
    (3 * 4096 + 5, 4096, 15, MAX, ELIAS, 5), (5 * 1024 + 1, 1024, 127, MAX, ELIAS, 17),
    (2 * 4096 + 77, 4096, 255, MAX, ELIAS, 17), (4096 + 40, 4096, 255, MAX, DENSE, 33),   # several passes over the peers
    (2 * 4096, 4096, 15, MAX, ELIAS, 64), (3000, 992, 128, L2, ELIAS, 40),
    (70 * 96 + 11, 96, 255, L2, ELIAS, 5), (1000, 160, 31, L2, DENSE, 4),
    # the dense code by table and symbol by symbol, codes of 5, 8 and 9 bits, words that lanes share
    (4096 + 33, 4096, 255, L2, DENSE, 3), (2 * 2048 + 1, 2048, 127, MAX, DENSE, 2), (999, 992, 15, L2, DENSE, 7),
    (3 * 64 + 2, 64, 255, L2, DENSE, 9), (2 * 4096 - 1, 4096, 1, L2, DENSE, 4), (5 * 512 + 3, 512, 128, MAX, DENSE, 6),
])
def test_teams(n, d, s, norm, code, K):
    run(n, d, s, norm, code, K)


@pytest.mark.parametrize("code,s,value", [(DENSE, 1, 0.0), (DENSE, 1, 1.0), (ELIAS, 1, 1.0), (ELIAS, 255, 1.0)])
def test_teams_out_of_step(code, s, value):
    """Strings of one repeated symbol (all levels 0, or every level s at gap 1): a lane that starts inside a
    symbol never falls into step and every part has to be read again from its predecessor's end."""
    n, d = 2 * 4096 + 100, 4096

    def make(w):
        g = np.full(n, value, np.float32)
        g[::d] = 1.0 + w
        return g
    run(n, d, s, MAX, code, 3, make)


@pytest.mark.parametrize("n,d,s,norm,K", [
    (13000 * 32 + 5, 32, 15, MAX, 1), (6500 * 96 + 95, 96, 3, L2, 2), (3200 * 160, 160, 15, L2, 4), (1800 * 224 + 1, 224, 7, MAX, 8),
    (1600 * 256 + 9, 256, 15, MAX, 8), (800 * 512 + 3, 512, 15, L2, 17), (500 * 1024 + 7, 1024, 1, MAX, 32), (1600 * 2048 + 2047, 2048, 15, L2, 9),
])
def test_streams(n, d, s, norm, K):
    """Many strings, up to half of those that get a lane each. Every other peer's strings have long gaps and empty
    buckets."""
    def make(w):
        if w % 2 == 0:
            return I.gaussian(n, 1.0, seed=50 + w)
        g = I.sparse_laplace(n, 1e-3, 0.3, seed=50 + w)
        g[np.random.default_rng(w).random(n) < 0.97] = 0.0
        g[n // 3: n // 3 + 3 * d] = 0.0
        return g
    run(n, d, s, norm, ELIAS, K, make)


@pytest.mark.parametrize("d,K", [(32, 1), (512, 16), (1024, 24)])
def test_malformed_streams(d, K):
    """Noise, strings cut short and offsets out of order in one peer's message: flagged, nothing
    written out of bounds, and where only one string is bad the buckets of the others come out right."""
    import paper_1610_02132_b200 as Q
    B = 13000 // K + 1
    n, s = B * d - d // 2, 3
    good, info = O.encode(I.gaussian(n, 1.0, seed=4), d, s, MAX, ELIAS, 7, 0, 0)
    table = O.message_table(good, info, n, d)
    noise = good.copy()
    noise[: info[1]] = np.random.default_rng(1).integers(0, 256, info[1], dtype=np.uint8)
    cut, swapped, above = table.copy(), table.copy(), table.copy()
    cut[B // 2] -= 3
    swapped[[B // 3, B // 3 + 1]] = swapped[[B // 3 + 1, B // 3]]
    above[-1] += 1 << 33
    one = good.copy()                                          # a level above s in one string: its first sign and level all ones
    lo = int(table[5]) + 32
    for t in range(lo, min(lo + 24, int(table[6]))):
        one[4 * (t // 32) + 3 - (t % 32) // 8] |= 1 << (7 - t % 8)
    for msg, tab, only in ((noise, table, None), (good, cut, None), (good, swapped, None), (good, above, None), (one, table, 5)):
        bufs = [torch.from_numpy(np.concatenate([m, np.zeros(64, np.uint8)])).cuda() for m in (msg, good)]
        tabs = [torch.from_numpy(x.view(np.int64)).cuda() for x in (tab, table)]
        order = [0] + [1] * (K - 1)
        status = Q.new_status()
        acc = torch.full((n + 256,), 7.0, device="cuda")
        Q.qsgd_decode_accumulate([bufs[i] for i in order], [tabs[i] for i in order], n, d, s, ELIAS, acc[:n], status,
                                 payload_bytes=[info[1]] * K)
        torch.cuda.synchronize()
        assert int(status.item()) != 0 and bool((acc[n:] == 7.0).all())
        if only is not None:
            ref = O.decode_accumulate([good] * K, [table] * K, n, d, s, ELIAS)[1]
            same = acc[:n].cpu().numpy().view(np.uint32) == ref.view(np.uint32)
            same[only * d: (only + 1) * d] = True
            assert same.all()


@pytest.mark.parametrize("n,d,s,K", [(3072 * 512, 512, 15, 8), (3072 * 512 + 1, 512, 15, 8), (6144 * 480, 480, 200, 4), (6144 * 480 + 1, 480, 200, 4), (2 ** 22, 128, 3, 2), (2 ** 25, 4096, 3, 2), (2 ** 20, 4096, 1, 8), (2 ** 20 + 4096, 4096, 1, 8),
                                     (10000 * 32 + 7, 32, 16, 5), (9000 * 64, 64, 101, 5), (9000 * 96 + 1, 96, 127, 5), (1400 * 480, 480, 255, 32)])
def test_lines_between_decoders(n, d, s, K):
    """Both sides of the lines between a lane and a team per string and between one and two launches, against
    the sum of the messages decoded one by one (K = 1 goes through another decoder or another split)."""
    import paper_1610_02132_b200 as Q
    msgs, infos = [], []
    for w in range(K):
        g = I.sparse_laplace_device(n, seed=w) if s == 1 else I.gaussian_device(n, 1.0, seed=w)
        out, bits, st = Q.encode_alloc(g, d, s, L2, ELIAS, 7, 0, w)
        msgs.append(out)
        infos.append(bits)
    status = Q.new_status()
    acc = torch.empty(n, device="cuda")
    Q.qsgd_decode_accumulate_packed(msgs, infos, n, d, s, ELIAS, acc, status)
    fixed, ref = [], torch.empty(n, device="cuda")
    for w in range(K):
        g = I.sparse_laplace_device(n, seed=w) if s == 1 else I.gaussian_device(n, 1.0, seed=w)
        fixed.append(Q.encode_alloc(g, d, s, L2, O.CODE_FIXED, 7, 0, w)[0])
    Q.qsgd_decode_accumulate_packed(fixed, None, n, d, s, O.CODE_FIXED, ref, status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    assert torch.equal(acc.view(torch.int32), ref.view(torch.int32))


@pytest.mark.parametrize("n,d,s,code", [
    (1, 32, 15, ELIAS), (4095, 32, 3, ELIAS), (4096, 64, 1, ELIAS), (4097, 512, 15, ELIAS), (42 * 96, 96, 255, ELIAS), (42 * 96 + 1, 96, 255, ELIAS),
    (2 * 4032, 2016, 15, DENSE), (3 * 4096, 4096, 64, DENSE), (4096000, 512, 15, ELIAS), (4096001, 512, 15, ELIAS), (1000 * 4032, 96, 7, ELIAS),
    (1000 * 4032 + 1, 96, 7, ELIAS), (2 ** 22 + 5, 4096, 64, DENSE), (2 ** 22 + 5, 128, 255, ELIAS), (2 ** 22 + 5, 32, 15, ELIAS),
    (2 ** 22 + 37, 480, 7, ELIAS), (2 ** 22 + 37, 2080, 3, DENSE), (7 * 2 ** 20 + 3, 160, 255, ELIAS),
])
def test_tiles(n, d, s, code):
    encode_parity(I.gaussian_mixture(n, seed=3), d, s, MAX, code, 7, 1, 2)
