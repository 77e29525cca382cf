"""Prompt products whose K is split over blocks (fewer tiles than SMs): a model
with a 4432-wide FFN (70 64-column stages, the last one partial, in uneven parts)
behind 200 columns, at prompt lengths on both sides of the token tiles, twice
each (the tiles' tickets are left as they were found), against the oracle; and
the logits of a prompt's last rows where trace_T asks for more rows than one
head launch takes (33)."""
import numpy as np
import pytest

import oracle
from parity import has_gpu, prompt, rel_err
from synth.workloads import LLAMA3_8B, scaled_down

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not has_gpu(), reason="needs a CUDA GPU")]

W = scaled_down(LLAMA3_8B, 2, 200, 2, 1, 4432, 1026, 140, 8, name="8b-split")


@pytest.fixture(scope="module")
def model():
    from paper_2606_03113_gb300.runtime import DeviceModel, Engine
    eng = Engine(DeviceModel(W.shape), W.max_seq)
    yield eng, oracle.Model(W.shape)
    eng.close()


@pytest.mark.parametrize("n", [17, 33, 40, 64, 65, 130])
def test_split_products(model, n):
    # the bounds of the prompt test: one bf16 rounding step of a key or value
    eng, om = model
    s = W.shape
    ids = prompt(W, n + 1)
    sess = om.session(W.max_seq)
    sess.prefill(ids[:n])
    h = om.session(W.max_seq).forward(ids, 0, 0, s.n_layers)
    seen = []
    for T in (20, 20, 64):
        eng.set_policy(0, trace_T=T)
        eng.prefill(ids[:n])
        _, pos, tr = eng.read_state()
        ref = [om.exit_head(h[r])[1]["pmax"] for r in range(max(0, n - T), n)]
        assert pos == n and len(tr) == len(ref) and rel_err(tr, ref) < 2e-2
        g = eng.read_kv(1, 1, 0, 0, n)
        r = np.array([[sess.kv(1, 1, 0, p, i) for i in range(s.head_dim)] for p in range(n)])
        assert rel_err(g, r) < 8e-3
        z, _ = eng.forward_exit(ids[n:], n, s.n_layers)
        assert rel_err(z[0], om.exit_head(h[n])[0]) < 2e-2
        seen.append((g, z, tr))
    assert np.array_equal(seen[0][0], seen[1][0]) and np.array_equal(seen[0][1], seen[1][1])
    assert list(seen[0][2]) == list(seen[1][2])
