"""Parity of the linear kernel's four tile shapes and their epilogues with the
CPU oracle, bit for bit, at the edges of their tiles: one frame, full tiles, a
remainder of one row, utterances that cross a tile, fewer stages of K than
groups of warps, and stage counts that leave the groups unequal shares."""
import numpy as np
import pytest

from guard import Guarded

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

# (B, T, K): with N = 2048 the host picks 32 x 32 tiles for up to 128 frames at
# K = 128, 64 x 64 from 129, 32 x 64 from 257 and 64 x 128 from 289; 32 x 64 from 225
# and 64 x 128 from 1505 at K = 1152
SIZES = [(1, 1, 128), (2, 32, 1152), (5, 13, 128), (1, 127, 384), (3, 43, 128), (1, 256, 384), (17, 17, 128),
         (2, 192, 128), (8, 190, 1152), (1, 257, 128), (2, 200, 384), (15, 17, 1152)]


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


@pytest.mark.parametrize("B,T,K", SIZES)
def test_tile_shapes_and_epilogues(ip, orc, B, T, K):
    N = 2048
    c = synth.linear(B, T, K, N, seed=1000 + B * T + K)
    m, s = orc.linear_constants(c.s_x, c.s_w, c.s_y_per_channel())
    x, w, bias, md, sd = (_d(a) for a in (c.x, c.w, c.bias, m, s))
    ws = torch.zeros(256, dtype=torch.uint8, device="cuda")
    z = orc.linear(c.x, c.w, c.bias, m, s)
    s_z = float(c.s_y[0])
    sw = orc.swish_params(s_z, s_z)
    gl = orc.glu_params(s_z, s_z, s_z)
    rp = orc.residual_params(s_z, s_z, 1.6 * s_z, 0.5)
    res = np.random.default_rng(B * T).integers(-127, 128, size=(B, T, N)).astype(np.int8)

    def same(want, call):
        g = Guarded(want.shape, torch.int8)
        got = call(out=g.view, workspace=ws)
        assert ip.status(ws) == 0
        g.check()
        bad = int((got.cpu().numpy() != want).sum())
        assert bad == 0, f"{bad} of {want.size} differ"

    same(z, lambda **kw: ip.linear_i8(x, w, bias, md, sd, **kw))
    heads = np.ascontiguousarray(z.reshape(B, T, 2, N // 256, 128).transpose(2, 0, 3, 1, 4))
    same(heads, lambda **kw: ip.linear_i8(x, w, bias, md, sd, y_layout=ip.HEADS, groups=2, **kw))
    xh = _d(c.x.reshape(B, T, K // 128, 128).transpose(0, 2, 1, 3))
    same(z, lambda **kw: ip.linear_i8(xh, w, bias, md, sd, x_layout=ip.HEADS, **kw))
    same(heads, lambda **kw: ip.linear_i8(xh, w, bias, md, sd, x_layout=ip.HEADS, y_layout=ip.HEADS, groups=2, **kw))
    same(orc.swish(z, sw), lambda **kw: ip.linear_swish_i8(x, w, bias, md, sd, (sw.q_c, sw.q_one, sw.m, sw.s), **kw))
    same(orc.glu(np.concatenate([z[..., 0::2], z[..., 1::2]], -1), gl),
         lambda **kw: ip.linear_glu_i8(x, w, bias, md, sd, (gl.q_c, gl.q_one, gl.m, gl.s), **kw))
    same(orc.residual(res, z, *rp), lambda **kw: ip.linear_residual_i8(x, w, bias, md, sd, _d(res), *rp, **kw))
