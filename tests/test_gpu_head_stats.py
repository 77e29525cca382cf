"""Exit-head statistics (§3.1.1) at vocabulary sizes around the chunks of the
statistics kernel (2048 logits; 256 chunks before a block takes several),
against float64 sums over the logits that the same call returns."""
import numpy as np
import pytest

from parity import has_gpu
from synth.workloads import TINY, scaled_down

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not has_gpu(), reason="needs a CUDA GPU")]


@pytest.mark.parametrize("V", [2, 10, 2046, 2048, 2050, 4098, 600002])
def test_head_statistics_at_chunk_edges(V):
    from paper_2606_03113_gb300.runtime import DeviceModel, Engine
    w = scaled_down(TINY, 1, 64, 1, 1, 64, V, 8, 4, name="tiny-v")
    eng = Engine(DeviceModel(w.shape), 64)
    k = min(5, V)
    ids = np.arange(17, dtype=np.int32) % V
    eng.set_ar()
    eng.prefill(ids[:2])
    z, st = eng.forward_exit(ids, 2, 1, topk=k)
    again = eng.forward_exit(ids[:3], 2, 1, topk=k)[1]
    eng.close()
    for m in range(17):
        x = z[m].astype(np.float64)
        s = st[m]
        order = np.lexsort((np.arange(V), -z[m]))[:8]  # larger first, then lower ids
        assert s["argmax"] == order[0]
        assert s["top_idx"][:len(order)] == list(order)
        assert s["top_logit"][:len(order)] == [float(z[m][i]) for i in order]
        lse = np.log(np.exp(x - x.max()).sum()) + x.max()
        p = np.exp(x - lse)
        # fp32 sums of positive terms in chunks of 8 per thread and trees: a
        # few 2^-24 each; the log-sum-exp of up to 13 adds 13 x 2^-24
        assert abs(s["lse"] - lse) < 1e-5
        assert abs(s["entropy"] - (p * (lse - x)).sum()) < 2e-5
        assert abs(s["conf_k"] - (lse - x[order[:k]]).mean()) < 1e-5
        assert abs(s["pmax"] - p.max()) < 1e-6 * p.max() + 1e-7
    # the same statistics whatever the number of rows
    assert again == st[:3]
