"""How much scratch an Elias encode asks for, and with it how far qsgd_encode_elias_static reaches (no GPU needed:
the size is refused before the device is looked for)."""
import pytest

import paper_1610_02132_b200 as Q
from oracle import oracle as O

ERR_SCRATCH = -10


def up16(x):
    return (x + 15) // 16 * 16


def scratch(n, d, s):
    """Fixed-width fields, a length per bucket, a record per lane of a bucket's team (a lane per 64 coordinates, at
    most a warp), a sum per 256 lanes, the control block."""
    B = O.n_buckets(n, d)
    lanes = 32 if d & (d - 1) else min(max(d // 64, 1), 32)
    ctas = -(-B // (8 * (32 // lanes)))
    return O.fixed_layout(n, d, s)[2] + up16(4 * B) + up16(4 * B * lanes) + up16(8 * (ctas + 1)) + 32


@pytest.mark.parametrize("d", [32, 64, 96, 128, 160, 256, 480, 512, 1024, 1056, 2048, 4064, 4096])
@pytest.mark.parametrize("s", [1, 3, 15, 255])
def test_scratch_is_no_more_than_the_layout_needs(d, s):
    last = 0
    for n in (1, d, 4096, 10 ** 5 + 1, 4096000, 4096001, 6 << 20, 20 << 20, (20 << 20) + 4096, 10 ** 8 + 7, 2 ** 28):
        need = Q.qsgd_workspace_bytes(n, d, s, O.CODE_ELIAS)
        assert need <= scratch(n, d, s)
        assert last <= need == Q.qsgd_workspace_bytes(n, d, s, O.CODE_ELIAS_DENSE)
        last = need
        tiles = -(-O.n_buckets(n, d) // (4096 // d))                       # a sum per tile fits where tiles keep theirs
        assert 8 * (tiles + 1) <= need - O.fixed_layout(n, d, s)[2] - 32


@pytest.mark.parametrize("d,s", [(32, 15), (64, 3), (256, 255), (512, 15), (1024, 1), (2048, 3), (4096, 1), (4096, 255)])
def test_reach_of_the_built_in_scratch(d, s):
    most, step = 1, 2 ** 27
    while step:                                            # the largest n that the layout fits 32 MiB with
        if scratch(most + step, d, s) <= Q.qsgd_static_scratch_bytes():
            most += step
        else:
            step //= 2
    L = Q.binding.lib()

    def call(n):
        return L.qsgd_encode_elias_static(16, n, d, s, O.NORM_L2, O.CODE_ELIAS, 7, 0, 0, 16, 2 ** 40, 16, 16, None)
    import torch
    if not torch.cuda.is_available():                      # with a GPU the call would go on to launch
        assert call(most) != ERR_SCRATCH
    assert call(most + 4096) == ERR_SCRATCH
