"""Parity with the CPU oracle where the last round of tiles is between half and
three quarters full, so that each SM takes one whole tile and at most one
quarter or half of another (two CTAs per SM on 152 SMs: 152 < r <= 228 of 304):
at both edges of the two ranges, with and without full rounds before it, with
the scores in the workspace, and with a mask planned on the host (more than 32
utterances) and on the device (padding after the parts).  Each call is made
three times on one workspace, since the CTAs flip the SMs' bits."""
import numpy as np
import pytest

import synth
from test_parity_gpu import assert_same, oracle_out, run_gpu

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ip():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_30846_gb300 as mod
    mod.load()
    return mod


@pytest.fixture(scope="module")
def orc():
    import oracle
    oracle.build()
    return oracle


def check(ip, orc, B, H, T, lengths=None):
    lay = synth.draw(B, H, T, 128, seed=900 + B + T, p_mode="random", masked=lengths is not None, lengths=lengths)
    c = ip.layer_constants(lay.scales)
    want = oracle_out(orc, lay, c, lengths)
    for _ in range(3):
        assert_same(run_gpu(ip, lay, c, lengths), want)


# r = N mod 304 with N = B H ceil(T / 64)
@pytest.mark.parametrize("B,H,T", [
    (19, 8, 64),     # 152: halves
    (9, 17, 64),     # 153: one tile in quarters
    (19, 10, 50),    # 190: the most quarters
    (1, 191, 33),    # 191: halves
    (19, 6, 100),    # 228: the most halves
    (1, 229, 64),    # 229: whole tiles
    (29, 8, 100),    # 304 + 160
    (48, 8, 66),     # 2 x 304 + 160
    (3, 8, 400),     # 168, scores in the workspace
    (9, 8, 400),     # 304 + 200, the same
])
def test_last_round(ip, orc, B, H, T):
    check(ip, orc, B, H, T)


@pytest.mark.parametrize("B,H,T,lengths", [
    (48, 8, 66, [66, 1, 65, 64] * 12),                                # the host's plan, padding among the items
    (12, 16, 130, [1, 64] * 5 + [0, 0]),                              # 160 live tiles, 416 of padding
    (12, 16, 130, [130] * 8 + [128, 65, 33, 0]),                      # 464 live tiles: 304 + 160
    (12, 16, 130, [130] * 10 + [100, 0]),                             # 512 live tiles: 304 + 208
])
def test_last_round_masked(ip, orc, B, H, T, lengths):
    check(ip, orc, B, H, T, np.array(lengths, np.int32))
