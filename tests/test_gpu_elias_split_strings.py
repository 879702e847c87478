"""A few long strings, each read by several warps of a CTA: bit for bit against the oracle, also where readers that start out of
step stay so; and malformed strings: flagged, the kernel returns, nothing written out of bounds, the other buckets right."""
import numpy as np
import pytest
import torch

import paper_1610_02132_b200 as Q
from oracle import oracle as O
from paper_1610_02132_b200 import inputs as I
from parity_util import decode_parity, encode_parity

pytestmark = pytest.mark.gpu

L2, MAX, ELIAS, DENSE = O.NORM_L2, O.NORM_MAX, O.CODE_ELIAS, O.CODE_ELIAS_DENSE
# (buckets, missing, d, s, norm, code, K): two warps a string, and four
SHAPES = [(1, 0, 4096, 64, L2, DENSE, 8), (3, 5, 4096, 15, MAX, ELIAS, 16), (2, 2047, 2048, 15, L2, DENSE, 4), (5, 1, 2080, 100, MAX, ELIAS, 3),
          (2, 77, 4096, 255, MAX, ELIAS, 2), (3, 4000, 4096, 255, MAX, DENSE, 8), (1, 1, 4096, 200, L2, DENSE, 1), (4, 0, 4064, 255, L2, ELIAS, 5)]


@pytest.mark.parametrize("B,missing,d,s,norm,code,K", SHAPES)
@pytest.mark.parametrize("flat", [False, True])
def test_well_formed(B, missing, d, s, norm, code, K, flat):
    n = B * d - missing
    msgs, infos = [], []
    for w in range(K):
        g = np.full(n, float(w % 2), np.float32) if flat else I.gaussian(n, 1.0, seed=50 + w)
        if flat:
            g[::d] = 1.0 + w                              # one symbol over and over: readers never fall into step
        m, info = encode_parity(g, d, s, norm, code, 7, 3, w)
        msgs.append(m)
        infos.append(info)
    decode_parity(msgs, infos, n, d, s, code, eta=0.05, x0=I.gaussian(n, 1.0, seed=9))


@pytest.mark.parametrize("B,missing,d,s,norm,code,K", SHAPES)
def test_malformed(B, missing, d, s, norm, code, K):
    n = B * d - missing
    good, info = O.encode(I.gaussian(n, 1.0, seed=3), d, s, norm, code, 7, 0, 0)
    table = O.message_table(good, info, n, d)
    ref = O.decode_accumulate([good] * K, [table] * K, n, d, s, code)[1]
    words = torch.tensor(info, dtype=torch.int64, device="cuda")
    first, last = int(table[0]) // 8 + 8, int(table[1]) // 8 - 8          # bytes well inside the first string
    for fill in (None, 0, 255, "noise"):
        bad = good.copy()
        if fill == "noise":
            bad[first:last] = np.random.default_rng(1).integers(0, 256, last - first, dtype=np.uint8)
        elif fill is not None:
            bad[first:last] = fill
        bufs = [torch.from_numpy(np.concatenate([m, np.zeros(64, np.uint8)])).cuda() for m in (good, bad)]
        acc, status = torch.full((n + 256,), 7.0, device="cuda"), Q.new_status()
        Q.qsgd_decode_accumulate_packed([bufs[0]] * (K - 1) + [bufs[1]], [words] * K, n, d, s, code, acc[:n], status)
        assert bool((acc[n:] == 7.0).all())
        assert (int(status.item()) != 0) == (fill is not None)
        same = acc[:n].cpu().numpy().view(np.uint32) == ref.view(np.uint32)
        assert same[d if fill is not None else 0:].all()
