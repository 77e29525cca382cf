"""Prompt chunks (bf16): KV rows, the C_trace window and the next logits at
prompt lengths on both sides of the token tiles' edges (32, 64, 128 rows), on
a model whose widths end inside a tile (d = 648, FFN 1712) with grouped
queries, against the oracle."""
import numpy as np
import pytest

import oracle
from parity import has_gpu, prompt, rel_err
from synth.workloads import LLAMA3_8B, scaled_down

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not has_gpu(), reason="needs a CUDA GPU")]

W = scaled_down(LLAMA3_8B, 2, 648, 6, 2, 1712, 2048, 260, 8, name="8b-ragged")


@pytest.fixture(scope="module")
def ragged():
    from paper_2606_03113_gb300.runtime import DeviceModel, Engine
    eng = Engine(DeviceModel(W.shape), W.max_seq)
    yield eng, oracle.Model(W.shape)
    eng.close()


@pytest.mark.parametrize("n", [16, 17, 31, 33, 64, 65, 128, 129, 257])
def test_prompt_at_tile_edges(ragged, n):
    # bf16 keys and values: one rounding is 2^-9 of a value, and a different
    # order of sums moves a value by at most one rounding step, so rows agree
    # within 2^-8 of the largest value (4e-3), doubled for the rows behind it
    eng, om = ragged
    s = W.shape
    ids = prompt(W, n + 1)
    eng.set_ar()
    eng.prefill(ids[:n])
    sess = om.session(W.max_seq)
    sess.prefill(ids[:n])
    for layer in range(s.n_layers):
        for kind in (0, 1):
            for head in range(s.n_kv_heads):
                g = eng.read_kv(layer, kind, head, 0, n)
                ref = np.array([[sess.kv(layer, kind, head, p, i) for i in range(s.head_dim)]
                                for p in range(n)])
                assert rel_err(g, ref) < 8e-3, (layer, kind, head)
    h = om.session(W.max_seq).forward(ids, 0, 0, s.n_layers)
    _, pos, tr = eng.read_state()
    ref = [om.exit_head(h[r])[1]["pmax"] for r in range(max(0, n - 20), n)]
    assert pos == n and len(tr) == len(ref) and rel_err(tr, ref) < 2e-2
    z, _ = eng.forward_exit(ids[n:], n, s.n_layers)
    assert rel_err(z[0], om.exit_head(h[n])[0]) < 2e-2
