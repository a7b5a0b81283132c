"""Parity of the linear epilogues with the CPU oracle where the rounding term
carries the product over 2^62: shift 31, the largest multiplier and a bias at
the end of its domain with a sum of the same sign, in tiles that hold a channel
with shift zero as well, for each tile shape and output form."""
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


def _d(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


# with K = 1152 and N = 2048 the host picks tiles of 32 x 32, 32 x 64 (353 to 448
# frames), 64 x 64 (609 to 896) and 64 x 128, more than one per SM; nine stages of
# K, so that slots of the ring are refilled
@pytest.mark.parametrize("T", [96, 400, 700, 1601])
def test_rounding_term_at_shift_31(ip, orc, T):
    K, N = 1152, 2048
    c = synth.linear(1, T, K, N, seed=31 + T)
    n = np.arange(N)
    x, w = np.abs(c.x), np.abs(c.w)
    w[n % 4 == 1] *= -1
    bias = np.where(n % 4 == 1, -(2 ** 30 - 1), 2 ** 30 - 1).astype(np.int32)
    m = np.full(N, 2 ** 31 - 1, np.int32)
    s = np.full(N, 31, np.int32)
    s[n % 8 == 2] = 30
    s[n % 32 == 7] = 0
    bias[n % 32 == 7] = 0
    m[n % 32 == 7] = 2 ** 20
    z = orc.linear(x, w, bias, m, s)
    assert (z[..., n % 4 == 0] == 1).all() and set(np.unique(z[..., n % 4 == 1])) <= {-1, 0}
    xd, wd, bd, md, sd = (_d(a) for a in (x, w, bias, m, s))
    ws = torch.zeros(256, dtype=torch.uint8, device="cuda")

    def same(want, call):
        g = Guarded(want.shape, torch.int8)
        got = call(out=g.view, workspace=ws)
        assert ip.status(ws) == 0
        g.check()
        bad = int((got.cpu().numpy() != want).sum())
        assert bad == 0, f"{bad} of {want.size} differ"

    same(z, lambda **kw: ip.linear_i8(xd, wd, bd, md, sd, **kw))
    heads = np.ascontiguousarray(z.reshape(1, T, 2, N // 256, 128).transpose(2, 0, 3, 1, 4))
    same(heads, lambda **kw: ip.linear_i8(xd, wd, bd, md, sd, y_layout=ip.HEADS, groups=2, **kw))
    xh = _d(x.reshape(1, T, K // 128, 128).transpose(0, 2, 1, 3))
    same(heads, lambda **kw: ip.linear_i8(xh, wd, bd, md, sd, x_layout=ip.HEADS, y_layout=ip.HEADS, groups=2, **kw))
    # output grids fine enough that 1 and -1 stay apart behind the gates
    s_z = 0.04
    sw, gl = orc.swish_params(s_z, s_z / 50), orc.glu_params(s_z, s_z, s_z / 50)
    same(orc.swish(z, sw), lambda **kw: ip.linear_swish_i8(xd, wd, bd, md, sd, (sw.q_c, sw.q_one, sw.m, sw.s), **kw))
    same(orc.glu(np.concatenate([z[..., 0::2], z[..., 1::2]], -1), gl),
         lambda **kw: ip.linear_glu_i8(xd, wd, bd, md, sd, (gl.q_c, gl.q_one, gl.m, gl.s), **kw))
    rp = orc.residual_params(s_z, s_z, 1.25 * s_z, 1.0)
    res = np.random.default_rng(T).integers(-127, 128, size=(1, T, N)).astype(np.int8)
    same(orc.residual(res, z, *rp), lambda **kw: ip.linear_residual_i8(xd, wd, bd, md, sd, _d(res), *rp, **kw))
