"""Draws from hand-set logits: rows whose logits are not finite.

The model's layers add nothing (wo = w_down = 0), every embedding is a row of
ones and eps is 0, so the normed row is ones and a logit is the sum of its
LM-head row: the first column holds the logits, the others are zero."""
import dataclasses

import numpy as np
import pytest

from parity import has_gpu
from synth.workloads import TINY, scaled_down
from paper_2606_03113_gb300 import ssd as S

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not has_gpu(), reason="needs a CUDA GPU")]


def engine(V, z):
    """Engine of a one-layer model whose logits are z at every position."""
    import torch
    from paper_2606_03113_gb300.runtime import DeviceModel, Engine
    w = scaled_down(TINY, 1, 64, 1, 1, 64, V, 8, 24, name="tiny-set")
    dm = DeviceModel(dataclasses.replace(w.shape, rms_eps=0.0))
    dm.embed.fill_(1.0)
    dm.layers[0]["wo"].zero_()
    dm.layers[0]["w_down"].zero_()
    dm.lm_head.zero_()
    dm.lm_head[:, 0] = torch.from_numpy(np.asarray(z, dtype=np.float32)).cuda()
    torch.cuda.synchronize()
    return dm, Engine(dm, 128)


@pytest.mark.parametrize("V", [1024, 8192])
@pytest.mark.parametrize("bad", [np.inf, np.nan])
def test_rows_without_a_finite_sum_are_refused(V, bad):
    dm, eng = engine(V, np.linspace(-1, 1, V))
    try:
        # an LM-head row whose product overflows (or is not a number)
        dm.lm_head[37] = 3e38 if np.isinf(bad) else bad
        ids = np.arange(5, dtype=np.int32)
        z, st = eng.forward_exit(ids, 0, 1)
        assert np.array_equal(z[0][37], np.float32(bad), equal_nan=True)
        if np.isinf(bad):
            assert st[0]["argmax"] == 37 and st[0]["zmax"] == np.inf
            assert np.isnan(st[0]["lse"]) and np.isnan(st[0]["entropy"])
        smp = dict(temperature=0.6, sample_seed=3)
        for policy in (lambda: eng.set_ar(**smp), lambda: eng.set_static(1, 3, **smp)):
            policy()
            with pytest.raises(S.SsdError) as e:  # the draw after the prompt
                eng.prefill(ids)
            assert e.value.status == S.SSD_ERR_DEVICE_FLAG
            eng.set_ar()
            eng.prefill(ids)
            policy()
            with pytest.raises(S.SsdError) as e:  # a round's drafts and last draw
                eng.step(4)
            assert e.value.status == S.SSD_ERR_DEVICE_FLAG
        # the context works on with finite rows
        dm.lm_head[37] = 0
        policy()
        eng.prefill(ids)
        assert len(eng.generate(8)[0]) == 8
    finally:
        eng.close()
