"""Parity of the depthwise kernel with the CPU oracle on both sides of every line
between the forms of its arithmetic: Swish constants that just fit and just miss
each form (clip point and 1 of the polynomial, shift, multiplier at which the
negative lobe reaches -127), and biases at and beyond the bound of the fast form
in some of a thread's four channels, for every kernel size."""
import numpy as np
import pytest

from guard import Guarded

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


def lobe(q_c, s):
    """The largest multiplier at which the most negative output stays at -127."""
    return min((127 << (31 + s)) // (4 * q_c ** 3 // 27 + 1), 2 ** 31 - 1)


CONSTANTS = [                                                   # q_c, q_one, m, s
    (32767, 2 ** 30 - 1, lobe(32767, 30), 30), (32767, 2 ** 30, lobe(32767, 30), 30),
    (32767, 2 ** 30 - 1, lobe(32767, 30) + 1, 30), (32768, 2 ** 30, lobe(32768, 31), 31),
    (32768, 2 ** 30, lobe(32768, 31) + 1, 31), (46340, 2 ** 31 - 1, lobe(46340, 17), 17),
    (46340, 2 ** 31 - 1, lobe(46340, 17) + 1, 17), (46340, 2 ** 31 - 1, lobe(46340, 16), 16),
    (1, 1, 2 ** 31 - 1, 17), (1, 2 ** 30 - 1, 2 ** 31 - 1, 17), (1, 2 ** 31 - 1, 2 ** 31 - 1, 17), (1, 2 ** 31 - 1, 5, 17), (10000, 2 ** 31 - 1, lobe(10000, 25), 25),
]


@pytest.mark.parametrize("K", [1, 3, 5, 7, 9, 11, 13, 15])
@pytest.mark.parametrize("i", range(len(CONSTANTS)))
def test_forms(ip, orc, K, i):
    B, T, C = 2, 61, 260
    rng = np.random.default_rng(100 * K + i)
    x = rng.integers(-128, 128, size=(B, T, C)).astype(np.int8)
    w = rng.integers(-128, 128, size=(C, K)).astype(np.int8)
    m = rng.integers(2 ** 30, 2 ** 31, size=C).astype(np.int32)
    s = rng.integers(0, 4, size=C).astype(np.int32)
    bias = rng.integers(-2000, 2000, size=C).astype(np.int32)
    # half the threads: one channel with a bias near its bound and a shift that
    # keeps the INT16 value in range
    edge = np.array([2 ** 30 - 2 ** 20, 2 ** 30 - 2 ** 20 + 1, 2 ** 30 - 1])
    at = np.arange(0, C, 8) + rng.integers(0, 4, size=len(range(0, C, 8)))
    at = at[at < C]
    bias[at] = rng.choice(edge, size=at.size) * rng.choice([-1, 1], size=at.size)
    s[at] = rng.choice([0, 14, 15, 20, 30, 31], size=at.size)
    m[at[::3]] = 2 ** 31 - 1
    q = CONSTANTS[i]
    want = orc.swish16(orc.dwconv(x, w, bias, m, s), orc.Swish16Params(*q))
    d = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    g, ws = Guarded(want.shape, torch.int8), torch.zeros(256, dtype=torch.uint8, device="cuda")
    got = ip.dwconv_swish_i8(d(x), d(w), d(bias), d(m), d(s), q, out=g.view, workspace=ws)
    assert ip.status(ws) == 0
    g.check()
    bad = int((got.cpu().numpy() != want).sum())
    assert bad == 0, f"{bad} of {want.size} differ"


# C = 512: the frames of a channel block are dealt four (eight from 3041 on) to a CTA
# as ten CTAs per SM would take them; from 609 to 1064 CTAs (912 from K = 13 on) run as
# seven (six) per SM: 1217 to 2128 frames, and 3041 to 4256 (to 1824 and 3648)
@pytest.mark.parametrize("K", [1, 3, 5, 7, 9, 11, 13, 15])
@pytest.mark.parametrize("B,T", [(4, 304), (1, 1217), (4, 456), (1, 1825), (7, 304), (1, 2129), (1, 3041), (3, 1216), (1, 3649), (8, 532),
                                 (1, 4257)])
def test_ctas_per_sm(ip, orc, K, B, T):
    C = 512
    rng = np.random.default_rng(B * T + K)
    x = rng.integers(-127, 128, size=(B, T, C)).astype(np.int8)
    w = rng.integers(-127, 128, size=(C, K)).astype(np.int8)
    m = rng.integers(2 ** 30, 2 ** 31, size=C).astype(np.int32)
    s = rng.integers(0, 4, size=C).astype(np.int32)
    bias = rng.integers(-2000, 2000, size=C).astype(np.int32)
    q = orc.swish16_params(10 / 32767, 4 / 127)
    want = orc.swish16(orc.dwconv(x, w, bias, m, s), q)
    d = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    g, ws = Guarded(want.shape, torch.int8), torch.zeros(256, dtype=torch.uint8, device="cuda")
    got = ip.dwconv_swish_i8(d(x), d(w), d(bias), d(m), d(s), (q.q_c, q.q_one, q.m, q.s), out=g.view, workspace=ws)
    assert ip.status(ws) == 0
    g.check()
    bad = int((got.cpu().numpy() != want).sum())
    assert bad == 0, f"{bad} of {want.size} differ"
