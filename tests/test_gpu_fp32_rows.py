"""fp32 decoder at widths around the row kernels' chunks (512 columns, float4
loads, four warps of row pairs, four input rows at a time), against the
oracle; and the same rows one at a time, bit for bit."""
import numpy as np
import pytest

import oracle
from parity import has_gpu, prompt, rel_err
from synth.workloads import TINY, scaled_down

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not has_gpu(), reason="needs a CUDA GPU")]


@pytest.mark.parametrize("d,heads,kv,ffn,V", [(32, 1, 1, 16, 6), (136, 3, 1, 528, 130),
                                              (512, 8, 2, 1040, 514), (520, 4, 4, 1536, 1026)])
def test_rows_at_chunk_edges(d, heads, kv, ffn, V):
    from paper_2606_03113_gb300.runtime import DeviceModel, Engine
    w = scaled_down(TINY, 2, d, heads, kv, ffn, V, 40, 8, name="f32-rows", head_dim=64)
    eng, om = Engine(DeviceModel(w.shape), 64), oracle.Model(w.shape)
    ids = prompt(w, 40)
    h = om.session(64).forward(ids, 0, 0, 2)
    eng.set_ar()
    for M in (1, 4, 5, 8, 9, 17):
        eng.prefill(ids[:20])
        z, _ = eng.forward_exit(ids[20:20 + M], 20, 2, topk=min(5, V))
        for m in range(M):
            # the fp32 bound of the parity tests (1e-4 of the largest logit)
            assert rel_err(z[m], om.exit_head(h[20 + m], topk=min(5, V))[0]) < 1e-4, (M, m)
        eng.prefill(ids[:20])
        for m in range(M):
            z1, _ = eng.forward_exit(ids[20 + m:21 + m], 20 + m, 2, topk=min(5, V))
            assert np.array_equal(z1[0], z[m]), (M, m)
    eng.close()
