"""Parity of masked batches with the CPU oracle where the live tiles are planned
on the device: utterances with no frames, one frame, whole tiles and all of T;
live tile counts that leave the last round whole, in halves and in quarters;
more padding than work; one utterance per lane (32) and one more (the host's
plan)."""
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


def lengths_of(kind, B, T, rng):
    if kind == "mixed":
        fixed = [0, 1, 63, 64, 65, T - 1, T, 128]
        return np.array([min(T, fixed[b % len(fixed)]) for b in range(B)], np.int32)
    if kind == "short":       # most of the batch is padding
        return np.array([T] + [int(v) for v in rng.integers(0, 40, size=B - 1)], np.int32)
    if kind == "full":
        return np.full(B, T, np.int32)
    if kind == "none":
        return np.zeros(B, np.int32)
    return rng.integers(T // 2, T, size=B, endpoint=True).astype(np.int32)


@pytest.mark.parametrize("kind", ["mixed", "short", "full", "none", "half"])
@pytest.mark.parametrize("B,H,T", [(9, 5, 129), (12, 8, 200), (32, 3, 250), (33, 3, 130), (3, 16, 450)])
def test_masked_batches(ip, orc, kind, B, H, T):
    rng = np.random.default_rng(B * T)
    lay = synth.draw(B, H, T, 128, seed=700 + B + T, p_mode="random", masked=True,
                     lengths=lengths_of(kind, B, T, rng))
    c = ip.layer_constants(lay.scales)
    assert_same(run_gpu(ip, lay, c, lay.lengths), oracle_out(orc, lay, c, lay.lengths))
