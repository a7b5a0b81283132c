"""Attention calls that follow one another on one workspace without a status call
between them, so that each finds the counters and the bits of the SMs as the call
before left them: last rounds with whole tiles beside quarters and halves (which
flip the bits), planned on the host and on the device, and calls without such a
round, from bits that are clear, set and mixed.  Every output is compared with the
CPU oracle."""
import numpy as np
import pytest

import synth
from test_parity_gpu import assert_same, oracle_out

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


# N mod 304 tiles: 190 (quarters), 228 (halves), 304 + 160, 464 live tiles of a masked
# batch, and without such a round 12, 304 and 229
CALLS = [(19, 10, 50, None), (2, 3, 100, None), (19, 6, 100, None), (38, 8, 64, None), (29, 8, 100, None),
         (12, 16, 130, [130] * 8 + [128, 65, 33, 0]), (1, 229, 64, None)]


@pytest.fixture(scope="module")
def calls(ip, orc):
    d = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    made = []
    for B, H, T, lengths in CALLS:
        lens = None if lengths is None else np.array(lengths, np.int32)
        lay = synth.draw(B, H, T, 128, seed=4000 + B + T, p_mode="random", masked=lens is not None, lengths=lens)
        c = ip.layer_constants(lay.scales)
        args = [d(getattr(lay, n)) for n in ("q", "k", "v", "p", "u", "vb")]
        made.append((args, c, None if lens is None else d(lens), oracle_out(orc, lay, c, lens)))
    return made


@pytest.mark.parametrize("fill", [0x00, 0xff, 0xa5])
def test_calls_in_a_row(ip, calls, fill):
    ws = torch.zeros(256, dtype=torch.uint8, device="cuda")
    ws[192:224] = fill   # the bits of the SMs: any value is valid
    outs = []
    for _ in range(3):
        for args, c, lens, _ in calls:
            outs.append(ip.relpos_mhsa_i8(*args, c, lengths=lens, workspace=ws))
    torch.cuda.synchronize()
    words = ws.view(torch.int32).cpu().numpy()
    assert (words[:48] == 0).all()   # no error, and every counter back at zero
    for i, got in enumerate(outs):
        assert_same(got.cpu().numpy(), calls[i % len(calls)][3])
