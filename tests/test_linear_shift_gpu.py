"""Parity of the linear epilogues with the CPU oracle where all, some and none of
the channels a warp finishes have a shift of zero (a shift of one and more is
taken from the product's high word), with multipliers and biases at the ends of
their domain, for each tile shape."""
import numpy as np
import pytest

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


@pytest.mark.parametrize("T", [32, 127, 256, 1505])   # the four shapes at N = 2048
@pytest.mark.parametrize("kind", ["none", "ones", "one_zero", "some", "zeros"])
def test_shifts(ip, orc, T, kind):
    K, N = 1152, 2048
    c = synth.linear(1, T, K, N, seed=77 + T)
    rng = np.random.default_rng(T)
    s = rng.integers(1, 32, size=N).astype(np.int32)
    if kind == "ones":
        s[:] = 1
    elif kind == "one_zero":
        s[N // 2 + 5] = 0
    elif kind == "some":
        s[::64] = 0
    elif kind == "zeros":
        s[:] = 0
    m = np.where(s < 4, rng.integers(0, 2 ** 24, size=N), rng.integers(2 ** 30, 2 ** 31, size=N)).astype(np.int32)
    m[::97] = 2 ** 31 - 1
    bias = c.bias.copy()
    bias[::31] = 2 ** 30 - 1
    bias[1::31] = -(2 ** 30 - 1)
    d = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    want = orc.linear(c.x, c.w, bias, m, s)
    got = ip.linear_i8(d(c.x), d(c.w), d(bias), d(m), d(s)).cpu().numpy()
    bad = int((got != want).sum())
    assert bad == 0, f"{bad} of {want.size} differ"
