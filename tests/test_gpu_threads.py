"""Two contexts on two host threads: calls with different numbers of rows (and of
different model shapes) interleave freely and change nothing of each other.
Both contexts launch on one stream, so their kernels run one after the other."""
import threading

import numpy as np
import pytest

from parity import has_gpu, prompt
from synth.workloads import LLAMA3_8B, TINY, scaled_down

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not has_gpu(), reason="needs a CUDA GPU")]

BF16 = scaled_down(LLAMA3_8B, 8, 256, 8, 2, 256, 512, 40, 8, name="8b-thr")
F32 = [scaled_down(TINY, 8, 128, 1, 1, 128, 512, 40, 8, head_dim=hd, name=f"tiny-thr{hd}")
       for hd in (128, 256)]


@pytest.mark.parametrize("models", [[(BF16, 1), (BF16, 17)], [(F32[0], 1), (F32[1], 17)]],
                         ids=["bf16", "f32"])
def test_contexts_on_two_threads(models):
    from paper_2606_03113_gb300.runtime import DeviceModel, Engine
    jobs = []
    for w, M in models:
        eng = Engine(DeviceModel(w.shape), 64)
        eng.set_ar()
        ids = prompt(w)
        eng.prefill(ids[:9])
        ref, _ = eng.forward_exit(ids[9:9 + M], 9, w.shape.n_layers)
        jobs.append((eng, ids[9:9 + M], w.shape.n_layers, ref))
    errors = []

    def work(eng, rows, L, ref):
        try:
            for _ in range(400):
                z, _ = eng.forward_exit(rows, 9, L)
                assert np.array_equal(z, ref)
        except Exception as e:  # reported by the main thread
            errors.append(repr(e))

    ts = [threading.Thread(target=work, args=j) for j in jobs]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    for j in jobs:
        j[0].close()
    assert not errors
