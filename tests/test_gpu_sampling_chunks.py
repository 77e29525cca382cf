"""Draws, acceptance tests and residual draws at vocabulary sizes around the
sampling kernels' chunks (2048 tokens; 4096 beyond 524288), recomputed in
float64 from the logits that the engine returns for the same rows."""
import numpy as np
import pytest

import oracle
import synth
from parity import has_gpu, prompt
from synth.workloads import TINY, scaled_down

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not has_gpu(), reason="needs a CUDA GPU")]

TEMP, SEED = 0.6, 9
# fp32 sums of positive weights: at most 16 terms per thread, then trees of 256
# threads and 256 chunks (16 + 5 + 8 + 5 + 8 additions of 2^-24 each), and
# weights within 2^-20 (z / T of up to 16 with one rounding each)
TOL = 2.0 ** -18


@pytest.mark.parametrize("V", [2, 2046, 2048, 2050, 4098, 530002])
def test_draws_at_chunk_edges(V):
    from paper_2606_03113_gb300.runtime import DeviceModel, Engine
    w = scaled_down(TINY, 2, 64, 1, 1, 64, V, 8, 24, name="tiny-v")
    eng = Engine(DeviceModel(w.shape), 64)
    eng.set_static(1, 3, temperature=TEMP, sample_seed=SEED)
    ids = [int(i) for i in prompt(w)]
    first = eng.prefill(np.array(ids, dtype=np.int32))
    toks, nr, _ = eng.generate(w.gen_len)
    seq = ids + [first] + [int(t) for t in toks]
    rounds = eng.traces(nr)
    compared = 0

    def same(weights, u, token):
        nonlocal compared
        t, margin = oracle.draw(weights, u)
        if margin > TOL:
            compared += 1
            assert t == token

    z, _ = eng.forward_exit(np.array(ids[-1:], dtype=np.int32), len(ids) - 1, 2)
    same(oracle.tempered(z[0], TEMP), synth.sample_uniforms(SEED, len(ids) - 1, 2, 1)[0], first)
    for r in rounds:
        pos, k, a = r["pos"], r["k"], r["a"]
        rows = np.array([seq[pos]] + list(r["drafts"][:k]), dtype=np.int32)
        zq = eng.forward_exit(rows[:k], pos, 1)[0] if k else []
        zp, _ = eng.forward_exit(rows, pos, 2)
        p = [oracle.tempered(x, TEMP) for x in zp]
        q = [oracle.tempered(x, TEMP) for x in zq]
        ud, ua = synth.sample_uniforms(SEED, pos, 0, 16), synth.sample_uniforms(SEED, pos, 1, 16)
        for i in range(k):
            same(q[i], ud[i], rows[i + 1])
        for i in range(min(a + 1, k)):
            d = rows[i + 1]
            margin = p[i][d] - ua[i] * q[i][d]
            if abs(margin) > TOL * max(p[i][d], ua[i] * q[i][d]):
                compared += 1
                assert (margin > 0) == (i < a)
        u = synth.sample_uniforms(SEED, pos, 2, 1)[0]
        if a == k:
            same(p[k], u, r["emitted"][a])
        else:
            res = np.maximum(p[a] - q[a], 0)
            # differences of the two: errors relative to the residual's mass
            if res.sum() > 1e-2:
                t, margin = oracle.draw(res, u)
                if margin > TOL / res.sum():
                    compared += 1
                    assert t == r["emitted"][a]
    eng.close()
    assert compared >= 2 * len(rounds)
