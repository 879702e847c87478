"""The dense code's stream decoder where a lane reads many buckets in a row, more than it has slots for their scales: sums bit for bit
against the oracle, and with single malformed strings in the middle of runs; and through a bucket map, with tensors off 16-byte places
that end in short buckets."""
import numpy as np
import pytest
import torch

import paper_1610_02132_b200 as Q
from oracle import oracle as O
from paper_1610_02132_b200 import inputs as I
from parity_util import decode_parity, encode_parity
from test_gpu_elias_decoders import worker
from test_gpu_elias_dense_streams import gradient
from test_gpu_policy import numel, run_case

pytestmark = pytest.mark.gpu

L2, MAX, DENSE = O.NORM_L2, O.NORM_MAX, O.CODE_ELIAS_DENSE


# runs of 26, 11, 4, 15 and 7 buckets where an SM has 13 warps for them (148 SMs)
@pytest.mark.parametrize("B,missing,d,s,norm,K", [(200000, 5, 32, 15, MAX, 8), (21000, 63, 64, 15, L2, 17), (60000, 9, 96, 32, MAX, 5),
                                                  (30000, 100, 160, 7, L2, 32), (400000, 1, 32, 15, MAX, 1)])
def test_sums_of_well_formed_messages(B, missing, d, s, norm, K):
    n = B * d - missing
    sent = [encode_parity(gradient(n, d, w), d, s, norm, DENSE, 7, 3, w) for w in range(min(K, 3))]
    msgs, infos = [sent[k % 3][0] for k in range(K)], [sent[k % 3][1] for k in range(K)]
    decode_parity(msgs, infos, n, d, s, DENSE, eta=0.05, x0=I.gaussian(n, 1.0, seed=9))
    words = [torch.tensor(i, dtype=torch.int64, device="cuda") for i in infos]
    acc, status = torch.empty(n, device="cuda"), Q.new_status()
    assert worker(lambda: Q.qsgd_decode_accumulate_packed(msgs, words, n, d, s, DENSE, acc, status)) == "decode_elias_dense"


@pytest.mark.parametrize("B,d,s,K", [(200000, 32, 15, 8), (21000, 64, 15, 17)])
def test_malformed_strings_in_the_middle_of_runs(B, d, s, K):
    n = B * d
    good, info = O.encode(gradient(n, d, 0), d, s, MAX, DENSE, 7, 0, 0)
    table = O.message_table(good, info, n, d)
    bad = np.arange(3, B, 1000)                            # at other places of their runs, one run apart and more
    ones, short, swapped = good.copy(), table.copy(), table.copy()
    for b in bad:                                          # ones behind the scale
        for t in range(int(table[b]) + 32, int(table[b]) + 56):
            ones[4 * (t // 32) + 3 - (t % 32) // 8] |= 1 << (7 - t % 8)
    short[bad + 1] -= 1                                    # ends a bit early, and the next one starts with it
    swapped[bad], swapped[bad + 1] = table[bad + 1], table[bad]
    ref = O.decode_accumulate([good] * K, [table] * K, n, d, s, DENSE)[1].view(np.uint32)
    words = torch.tensor(info, dtype=torch.int64, device="cuda")
    for msg, tab, hit in ((ones, table, (0,)), (good, short, (0, 1)), (good, swapped, (-1, 0, 1))):
        bufs = []
        for m, t in ((msg, tab), (good, table)):
            m = m.copy()
            m[info[1]: info[1] + t.nbytes] = t.view(np.uint8)
            bufs.append(torch.from_numpy(np.concatenate([m, np.zeros(64, np.uint8)])).cuda())
        acc, status = torch.full((n + 256,), 7.0, device="cuda"), Q.new_status()
        Q.qsgd_decode_accumulate_packed([bufs[1]] * (K - 1) + [bufs[0]], [words] * K, n, d, s, DENSE, acc[:n], status)
        assert bool((acc[n:] == 7.0).all()) and int(status.item()) != 0
        same = (acc[:n].cpu().numpy().view(np.uint32) == ref).reshape(B, d).all(axis=1)
        for h in hit:
            same[bad + h] = True
        assert same.all()


# values across the lanes and from shared memory, eight coordinates at a time and four
@pytest.mark.parametrize("tensor,count,d,s,norm,K", [(10007, 60, 32, 15, MAX, 8), (10007, 60, 64, 32, L2, 12), (10002, 60, 96, 15, L2, 17),
                                                     (98003, 40, 512, 64, MAX, 6)])
def test_buckets_through_a_map(tensor, count, d, s, norm, K):
    sizes = [tensor + 3 * i for i in range(count)]
    sizes[1::7] = [11] * len(sizes[1::7])                  # raw ones between them
    assert worker(lambda: run_case(sizes, d, s, norm, DENSE, K=K)) == "decode_elias_dense"


def test_resnet152_shapes():
    sizes = [numel(sh) for sh in I.resnet152_shapes()]
    assert worker(lambda: run_case(sizes, 512, 15, L2, DENSE, K=2)) == "decode_elias_dense"
