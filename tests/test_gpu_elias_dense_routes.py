"""The dense code's two decoders on both sides of the lines between them: the kernel that did the work, and its sums bit for bit
against the other's, which the same messages reach in pieces."""
import pytest
import torch

import paper_1610_02132_b200 as Q
from oracle import oracle as O
from paper_1610_02132_b200 import inputs as I
from test_gpu_elias_decoders import worker

pytestmark = pytest.mark.gpu

TEAMS, STREAMS = "decode_elias_teams", "decode_elias_dense"


@pytest.mark.parametrize("decoder,B,missing,d,s,K", [
    # few levels in short buckets: measured slower by streams
    (TEAMS, 13000, 1, 32, 1, 5), (TEAMS, 6000, 31, 32, 3, 8), (TEAMS, 60000, 7, 32, 7, 1), (STREAMS, 55000, 7, 32, 7, 8),
    (TEAMS, 130000, 0, 64, 3, 1), (STREAMS, 60000, 0, 64, 3, 1), (TEAMS, 14000, 95, 96, 3, 8), (STREAMS, 9000, 95, 96, 3, 8),
    (STREAMS, 36000, 3, 96, 1, 8), (TEAMS, 150000, 1, 160, 3, 1), (STREAMS, 60000, 1, 160, 3, 1), (TEAMS, 70000, 0, 256, 1, 1),
    # more levels: by the number of strings alone
    (STREAMS, 6000, 31, 32, 8, 8), (STREAMS, 60000, 1, 32, 15, 1), (TEAMS, 2000, 1, 32, 15, 8)])
def test_decoder(decoder, B, missing, d, s, K):
    n = B * d - missing
    sent = [Q.encode_alloc(I.gaussian_device(n, 1.0, seed=w), d, s, O.NORM_L2, O.CODE_ELIAS_DENSE, 7, 0, w)[:2] for w in range(min(K, 2))]
    msgs, infos = [sent[k % 2][0] for k in range(K)] if K > 1 else [sent[0][0]], [sent[k % 2][1] for k in range(K)] if K > 1 else [sent[0][1]]
    acc, status = torch.full((n + 64,), 7.0, device="cuda"), Q.new_status()
    assert worker(lambda: Q.qsgd_decode_accumulate_packed(msgs, infos, n, d, s, O.CODE_ELIAS_DENSE, acc[:n], status)) == decoder
    # the same strings as messages of 2000 buckets, which teams read whatever their kind: tables moved in front
    parts = 2000
    ref, tables = torch.empty(n, device="cuda"), [m[int(i[1]): int(i[1]) + 8 * (B + 1)].view(torch.int64) for m, i in zip(msgs, infos)]
    for b in range(0, B, parts):
        here = slice(b * d, min((b + parts) * d, n))
        cut = [t[b: b + parts + 1].clone() for t in tables]
        Q.qsgd_decode_accumulate(msgs, cut, here.stop - here.start, d, s, O.CODE_ELIAS_DENSE, ref[here], status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    assert torch.equal(acc[:n].view(torch.int32), ref.view(torch.int32)) and bool((acc[n:] == 7.0).all())
