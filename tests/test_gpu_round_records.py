"""The records of a run of rounds against the state they leave: emitted tokens,
positions and the C_trace window (full-model max-probabilities of the rows each
round kept, behind the prompt's), greedy and sampled."""
import numpy as np
import pytest

from parity import has_gpu, prompt
from synth.workloads import TINY

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not has_gpu(), reason="needs a CUDA GPU")]


@pytest.mark.parametrize("temperature", [0.0, 0.8])
@pytest.mark.parametrize("k", [1, 4, 16])
def test_records_match_the_state(temperature, k):
    from paper_2606_03113_gb300.runtime import DeviceModel, Engine
    eng = Engine(DeviceModel(TINY.shape), 256)
    ids = prompt(TINY)
    eng.set_static(3, k, temperature=temperature, sample_seed=11)
    first = eng.prefill(ids)
    _, p0, window = eng.read_state()
    toks, nr, _ = eng.generate(120)
    tr = eng.traces(nr)
    x, pos, got = eng.read_state()
    eng.close()
    want = list(window)
    seq = [first]
    for r in tr:
        assert r["x"] == seq[-1] and r["pos"] == p0 + len(seq) - 1
        assert r["n_emit"] == r["a"] + 1
        seq += list(r["emitted"][:r["n_emit"]])
        want += list(r["verify_pmax"][:r["a"] + 1])
    assert seq[1:] == [int(t) for t in toks] and x == seq[-1] and pos == p0 + len(seq) - 1
    assert len(want) > 64 and len(got) == 64
    assert np.array_equal(np.float32(got), np.float32(want[-64:]))
