"""Calls that must not fall behind others of the same size: ratios of times of one and the same run, with room for
noise. What is compared is device time (a graph of several calls, replayed; the shortest replay)."""
import pytest
import torch

import paper_1610_02132_b200 as Q
from oracle import oracle as O
from paper_1610_02132_b200 import inputs as I

pytestmark = pytest.mark.gpu


def time_of(*calls, repeats=8, replays=7):
    """Shortest time of each call, taken in turn."""
    graphs, best = [], [float("inf")] * len(calls)
    for call in calls:
        call()
        torch.cuda.synchronize()
        graphs.append(torch.cuda.CUDAGraph())
        with torch.cuda.graph(graphs[-1]):
            for _ in range(repeats):
                call()
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    for _ in range(replays):
        for i, g in enumerate(graphs):
            a.record()
            g.replay()
            b.record()
            torch.cuda.synchronize()
            best[i] = min(best[i], a.elapsed_time(b))
    return best


def decode(n, d, s, norm, code, K, make=None, packed=True):
    """A call that decodes K messages into a sum, and the payload bits per coordinate behind the scales."""
    make = make or (lambda w: I.gaussian_device(n, 1.0, seed=w))
    sent = [Q.encode_alloc(make(w), d, s, norm, code, 7, 0, w)[:2] for w in range(min(K, 4))]
    infos = [[int(v) for v in bits.tolist()] for _, bits in sent]
    B = O.n_buckets(n, d)
    pick = [w % len(sent) for w in range(K)]
    msgs, words = [sent[i][0] for i in pick], [sent[i][1] for i in pick]
    tables = [sent[i][0][infos[i][1]: infos[i][1] + 8 * (B + 1)].view(torch.int64) for i in pick]
    acc, status = torch.empty(n, device="cuda"), Q.new_status()

    def call():
        if packed:
            Q.qsgd_decode_accumulate_packed(msgs, words, n, d, s, code, acc, status)
        else:
            Q.qsgd_decode_accumulate(msgs, tables, n, d, s, code, acc, status)
    call.status = status
    call.bits = sum(i[0] - 32 * B for i in infos) / n / len(infos)
    return call


def test_fewer_bits_do_not_take_longer_in_the_dense_code():
    """Strings of small levels, whose symbols all have even lengths, against strings with twice the bits."""
    n, d, K = 2 ** 22, 4096, 8
    small, large = decode(n, d, 1, O.NORM_L2, O.CODE_ELIAS_DENSE, K), decode(n, d, 15, O.NORM_MAX, O.CODE_ELIAS_DENSE, K)
    assert small.bits < 0.6 * large.bits
    few, many = time_of(small, large)
    assert few < 1.2 * many
    assert int(small.status.item()) == int(large.status.item()) == 0


def test_rare_odd_symbols_do_not_take_longer_in_the_dense_code():
    """The same with a few levels of 3 and more among them: symbols of 7 bits, each of which shifts the rest."""
    n, d, K = 2 ** 22, 4096, 4
    rare = decode(n, d, 15, O.NORM_L2, O.CODE_ELIAS_DENSE, K, lambda w: I.gaussian_mixture_device(n, seed=w))
    large = decode(n, d, 15, O.NORM_MAX, O.CODE_ELIAS_DENSE, K)
    assert rare.bits < 0.6 * large.bits
    few, many = time_of(rare, large)
    assert few < 1.3 * many


def test_many_peers_of_a_small_problem_are_read_in_one_pass():
    """32 short strings a bucket against 8: more to add up, but no more latencies in a row."""
    n, d = 16 * 1024, 1024
    make = lambda w: I.gaussian_mixture_device(n, seed=w)
    eight, all32 = (decode(n, d, 1, O.NORM_L2, O.CODE_ELIAS, K, make) for K in (8, 32))
    few, many = time_of(eight, all32)
    assert many < 2.0 * few


def encode(n, d, s, norm, code):
    g, status = I.gaussian_device(n, 1.0, seed=3), Q.new_status()
    out = torch.empty(Q.qsgd_message_capacity(n, d, s, code), dtype=torch.uint8, device="cuda")
    info = torch.zeros(4, dtype=torch.int64, device="cuda")
    ws = torch.empty(Q.qsgd_workspace_bytes(n, d, s, code), dtype=torch.uint8, device="cuda")
    return lambda: Q.qsgd_encode(g, d, s, norm, code, 7, 0, 0, out, info, ws, status)


def test_dense_encode_grows_no_faster_than_its_length():
    """Small levels: 18 M coordinates against 24 M, which no rule sends through kernels meant for few."""
    less, more = time_of(*(encode(n, 4096, 1, O.NORM_L2, O.CODE_ELIAS_DENSE) for n in (18 * 2 ** 20, 24 * 2 ** 20)))
    assert less < 0.88 * more                              # 0.75 by length alone; 1.0 by tiles
