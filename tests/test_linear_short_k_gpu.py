"""Parity of the linear layer with the CPU oracle for one to four stages of K,
where groups of warps go without a stage and the host's choice of a tile shape
follows the number of tiles rather than the stages: both sides of the lines
between the shapes, with one tile per SM and with several."""
import numpy as np
import pytest

from guard import Guarded

import synth

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


# N = 2048: 32 x 32 tiles up to 128 frames, 64 x 64 from 129, 64 x 128 from 257 at
# K = 128 and 256; 32 x 64 from 257 to 288, 64 x 64 from 289, 64 x 128 from 897 at 384
# and 512 (64 x 64 again from 1217 to 1472)
@pytest.mark.parametrize("T,K", [(31, 128), (128, 256), (129, 128), (130, 512), (256, 256), (257, 128), (258, 384),
                                 (288, 512), (289, 512), (700, 384), (900, 512), (1217, 512), (1473, 384), (1601, 256)])
def test_short_k(ip, orc, T, K):
    N = 2048
    c = synth.linear(1, T, K, N, seed=5000 + T + K)
    m, s = orc.linear_constants(c.s_x, c.s_w, c.s_y_per_channel())
    d = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    want = orc.linear(c.x, c.w, c.bias, m, s)
    g, ws = Guarded(want.shape, torch.int8), torch.zeros(256, dtype=torch.uint8, device="cuda")
    got = ip.linear_i8(d(c.x), d(c.w), d(c.bias), d(m), d(s), out=g.view, workspace=ws)
    assert ip.status(ws) == 0
    g.check()
    bad = int((got.cpu().numpy() != want).sum())
    assert bad == 0, f"{bad} of {want.size} differ"
