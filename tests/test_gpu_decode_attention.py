"""Decode attention of bf16 models: logits of 1 to 17 rows at positions on both
sides of the 64- and 128-key splits, without and with grouped queries, against
the oracle; and the same rows one at a time, bit for bit."""
import numpy as np
import pytest

import oracle
from parity import has_gpu, prompt, rel_err
from synth.workloads import LLAMA3_8B, scaled_down

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not has_gpu(), reason="needs a CUDA GPU")]

# heads, KV heads, cache length: 64 keys per split where KV heads x splits is
# at most three per SM, else 128
SHAPES = {"split64": (16, 2, 320), "split128": (16, 16, 2048)}
W = {k: scaled_down(LLAMA3_8B, 1, 256, hq, hkv, 256, 512, 150, 8, name="attn-" + k)
     for k, (hq, hkv, _) in SHAPES.items()}


@pytest.fixture(scope="module", params=list(SHAPES))
def model(request):
    from paper_2606_03113_gb300.runtime import DeviceModel, Engine
    w = W[request.param]
    eng = Engine(DeviceModel(w.shape), SHAPES[request.param][2])
    om = oracle.Model(w.shape)
    ids = prompt(w, 290)
    h = om.session(320).forward(ids, 0, 0, 1)
    yield eng, om, ids, h
    eng.close()


@pytest.mark.parametrize("pos0,M", [(1, 1), (47, 17), (48, 17), (63, 1), (63, 2), (64, 1), (120, 8),
                                    (127, 2), (128, 17), (250, 17), (272, 17)])
def test_rows_at_split_edges(model, pos0, M):
    # one layer, bf16 KV: the bound of the prompt test (a rounding step of a
    # key or value is 2^-8 of it, doubled)
    eng, om, ids, h = model
    eng.set_ar()
    eng.prefill(ids[:pos0])
    z, st = eng.forward_exit(ids[pos0:pos0 + M], pos0, 1)
    for m in range(M):
        assert rel_err(z[m], om.exit_head(h[pos0 + m])[0]) < 8e-3, m
    eng.prefill(ids[:pos0])
    for m in range(M):
        z1, st1 = eng.forward_exit(ids[pos0 + m:pos0 + m + 1], pos0 + m, 1)
        assert np.array_equal(z1[0], z[m]) and st1[0] == st[m]
