"""A prompt's KV rows (bf16, more than 16 rows) do not depend on what follows
them: prompts of every plan (token tiles of 32, 64 and 128 rows, K of a product
split over blocks or not, one chunk or several) agree bit for bit on their
common rows, and so does ssd_resume.  fp32 rows do not depend on the way they
came either: decoding and resuming leave the same."""
import numpy as np
import pytest

from parity import has_gpu, prompt
from synth.workloads import LLAMA3_8B, TINY, scaled_down

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not has_gpu(), reason="needs a CUDA GPU")]

# products of 28 to 70 64-column stages; few row tiles (K split up to eight
# ways in short prompts) and many (never split)
W = {"narrow": scaled_down(LLAMA3_8B, 3, 1800, 2, 1, 4432, 1026, 1400, 8, name="8b-narrow"),
     "wide": scaled_down(LLAMA3_8B, 2, 4096, 8, 2, 2048, 1026, 300, 8, name="8b-wide")}


@pytest.mark.parametrize("name", list(W))
def test_rows_do_not_depend_on_the_prompts_length(name):
    from paper_2606_03113_gb300.runtime import DeviceModel, Engine
    w = W[name]
    s = w.shape
    eng = Engine(DeviceModel(s), w.prompt_len + 8)
    eng.set_ar()
    ids = prompt(w)

    def rows(n):
        return np.array([[eng.read_kv(l, kind, 0, 0, n) for kind in (0, 1)]
                         for l in range(s.n_layers)])

    eng.prefill(ids)
    ref = rows(len(ids))
    for n in (17, 32, 33, 65, 93, 129, 200, 300, 700, 1290):
        if n >= len(ids):
            break
        eng.prefill(ids[:n])
        assert np.array_equal(rows(n), ref[:, :, :n]), n
        eng.resume(ids[:n + 1])
        assert np.array_equal(rows(n), ref[:, :, :n]), n
    eng.close()


@pytest.mark.parametrize("n", [3, 16, 33])
def test_fp32_rows_are_the_same_after_resuming(n):
    from paper_2606_03113_gb300.runtime import DeviceModel, Engine
    w = TINY
    eng = Engine(DeviceModel(w.shape), 160)
    eng.set_static(2, 4)
    ids = prompt(w, 33)[:n]
    seq = list(ids) + [eng.prefill(ids)]
    seq += [int(t) for t in eng.generate(80)[0]]
    _, pos, _ = eng.read_state()

    def rows():
        return np.array([[eng.read_kv(l, kind, h, 0, pos) for kind in (0, 1)
                          for h in range(w.shape.n_kv_heads)] for l in range(w.shape.n_layers)])

    ref = rows()
    eng.resume(seq)
    assert pos == len(seq) - 1 and np.array_equal(rows(), ref)
    eng.close()
