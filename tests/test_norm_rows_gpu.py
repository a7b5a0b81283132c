"""Parity of the LayerNorm's two kernels with the CPU oracle on both sides of
the row count where the call changes from one to the other: one CTA per row up
to 256 rows, batches of rows above.  The same rows (random, constant, extreme
and nearly constant ones) with constants that take both requantisation shifts."""
import numpy as np
import pytest

from test_norm_gpu import _d, assert_same, case

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


@pytest.mark.parametrize("d", [512, 1024, 1536, 2048])
@pytest.mark.parametrize("rows,e31", [(2, True), (255, False), (256, True), (257, True), (258, False)])
def test_both_kernels(ip, orc, d, rows, e31):
    x, gamma, beta, s_x, s_y, eps = case(rows, d, seed=20 + d + rows)
    x[0] = -127
    x[rows // 2] = np.where(np.arange(d) % 2 == 0, 127, -127)
    x[-1] = np.where(np.arange(d) == d - 1, 1, 0)
    c = orc.layernorm_constants(s_x, gamma, beta, s_y, eps)
    M, B, E = c.M.copy(), c.B.copy(), c.E.copy()
    if e31:
        ch = np.arange(0, d, 61)
        sh = E[ch] - 31
        M[ch] >>= sh
        B[ch] >>= sh
        E[ch] = 31
    E[5], B[5] = 62, 0
    ws = torch.zeros(256, dtype=torch.uint8, device="cuda")
    xd = _d(x)
    got = ip.layernorm_i8(xd, _d(M), _d(B), _d(E), c.eps_c, workspace=ws)
    want = orc.layernorm(x, orc.NormConstants(M=M, B=B, E=E, eps_c=c.eps_c))
    assert ip.status(ws) == 0
    assert_same(got.cpu().numpy(), want)
    ip.layernorm_i8(xd, _d(M), _d(B), _d(E), c.eps_c, out=xd, workspace=ws)   # in place
    assert_same(xd.cpu().numpy(), want)


@pytest.mark.parametrize("rows", [256, 257])
def test_constant_out_of_domain_is_reported(ip, orc, rows):
    x, gamma, beta, s_x, s_y, eps = case(rows, 1024, seed=9)
    c = orc.layernorm_constants(s_x, gamma, beta, s_y, eps)
    B = c.B.copy()
    B[1000] = 2 ** 60
    ws = torch.zeros(256, dtype=torch.uint8, device="cuda")
    ip.layernorm_i8(_d(x), _d(c.M), _d(B), _d(c.E), c.eps_c, workspace=ws)
    assert ip.status(ws) == -7
