"""Draws from hand-set logits: weights of exactly zero with u S in the rounding
gap between two threads' runs, and rows whose logits are not finite.

The model's layers add nothing (wo = w_down = 0), every embedding is a row of
ones and eps is 0, so the normed row is ones and a logit is the sum of its
LM-head row: the first column holds the logits, the others are zero."""
import dataclasses

import numpy as np
import pytest

import synth
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


def test_token_of_zero_weight_is_never_drawn():
    # Token 1 has weight 1; the first token of each 8-token run has weight 0,
    # the others 0.9 x 2^-25, which a running sum above 1 cannot take up (half
    # its last place is 2^-24) but the sums of runs and chunks do.  Every u S
    # above 1 then lies between the end of a run's sequential sum and the prefix
    # that the next run starts from.
    V = 32768
    z = np.full(V, np.log(0.9 * 2.0 ** -25), dtype=np.float32)
    z[::8] = -200.0
    z[1] = 0.0
    wgt = np.exp(z.astype(np.float64))
    wgt[::8] = 0.0
    cdf = np.cumsum(wgt) / wgt.sum()
    ids = np.arange(5, dtype=np.int32)
    above = [(s, u) for s in range(40000)
             for u in [float(synth.sample_uniforms(s, len(ids) - 1, 2, 1)[0])] if u > cdf[7]][:12]
    assert len(above) == 12
    dm, eng = engine(V, z)
    try:
        zg, _ = eng.forward_exit(ids, 0, 1)
        assert np.array_equal(zg[0], z)
        for seed, u in above:
            eng.set_ar(temperature=1.0, sample_seed=seed)
            t = eng.prefill(ids)
            assert z[t] > -200.0, (seed, u, t)
            # fp32 sums of at most 8 + 256 + 16 terms, all below 2: 2^-23 each
            assert abs(cdf[t] - u) < 280 * 2.0 ** -23
    finally:
        eng.close()


@pytest.mark.parametrize("n", [1, 5, 16, 17, 40])
def test_draw_after_the_prompt_reads_its_last_row(n):
    # the last token's row gives 2048 tokens equal weights, so that u decides; the
    # rows before it (of opposite sign) would give them none
    V = 4096
    z = np.zeros(V)
    z[V // 2:] = -200.0
    dm, eng = engine(V, z)
    try:
        dm.embed[1:] = -1.0
        ids = np.array([1] * (n - 1) + [0], dtype=np.int32)
        for seed in range(4):
            eng.set_ar(temperature=0.7, sample_seed=seed)
            t = eng.prefill(ids)
            u = float(synth.sample_uniforms(seed, n - 1, 2, 1)[0])
            assert t == int(u * 2048)  # sums of ones up to 2048 are exact in fp32
    finally:
        eng.close()


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
