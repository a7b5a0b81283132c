"""Parity of the INT16 Swish of the depthwise kernel with the CPU oracle on
nearly every INT16 value, at the shifts where the kernel changes the way it
splits the 78-bit product (s >= 17: 32-bit words, below: bit 31), with
multipliers that make exact ties."""
import numpy as np
import pytest

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


@pytest.mark.parametrize("s", [0, 1, 16, 17, 31])
@pytest.mark.parametrize("m", [1, 2 ** 30, 2 ** 31 - 1])
@pytest.mark.parametrize("q_c,q_one", [(1, 1), (256, 65536), (728, 703818), (46340, 2 ** 31 - 1)])
def test_every_value(ip, orc, s, m, q_c, q_one):
    # acc = 2 (256 (c - 128) + x), halved onto the INT16 grid: z = 256 (c - 128) + x
    C, T = 256, 255
    x = np.broadcast_to(np.arange(-127, 128, dtype=np.int8)[None, :, None], (1, T, C)).copy()
    w = np.full((C, 1), 2, np.int8)
    bias = (2 * 256 * (np.arange(C) - 128)).astype(np.int32)
    mc = np.full(C, 2 ** 30, np.int32)
    sc = np.zeros(C, np.int32)
    d = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    want = orc.swish16(orc.dwconv(x, w, bias, mc, sc), orc.Swish16Params(q_c, q_one, m, s))
    got = ip.dwconv_swish_i8(d(x), d(w), d(bias), d(mc), d(sc), (q_c, q_one, m, s)).cpu().numpy()
    bad = int((got != want).sum())
    assert bad == 0, f"{bad} of {want.size} differ"
