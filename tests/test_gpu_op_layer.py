"""ssd_op_layer: each kernel reads the residual rows under its own norm, whatever
pass or kernel wrote them last.  Layers run kernel by kernel give the KV rows
and the logits of a teacher-forced pass bit for bit."""
import numpy as np
import pytest

from parity import has_gpu, prompt
from synth.workloads import LLAMA3_8B, TINY, scaled_down

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not has_gpu(), reason="needs a CUDA GPU")]

W = {"bf16": scaled_down(LLAMA3_8B, 3, 256, 4, 2, 512, 512, 24, 8, name="8b-op"),
     "f32": scaled_down(TINY, 3, 128, 2, 2, 256, 512, 24, 8, name="tiny-op")}


@pytest.fixture(scope="module", params=list(W))
def model(request):
    import torch
    from paper_2606_03113_gb300.runtime import DeviceModel, Engine
    w = W[request.param]
    dm = DeviceModel(w.shape)
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    for t in [dm.final_norm] + [l[k] for l in dm.layers for k in ("attn_norm", "ffn_norm")]:
        t.normal_(1.0, 0.3, generator=g)  # each norm its own weights
    torch.cuda.synchronize()
    eng = Engine(dm, 64)
    eng.set_ar()
    yield w, eng
    eng.close()


def kv(eng, w, layer, p0, M):
    return np.array([[eng.read_kv(layer, kind, h, p0, M) for h in range(w.shape.n_kv_heads)]
                     for kind in (0, 1)])


@pytest.mark.parametrize("M", [1, 3, 17])
def test_kernels_read_the_rows_under_their_own_norm(model, M):
    w, eng = model
    ids, p0 = prompt(w), 5
    rows = ids[p0:p0 + M]

    def start(l_exit):
        eng.prefill(ids[:p0])
        return eng.forward_exit(rows, p0, l_exit)[0]

    ref = [None, start(1), start(2), start(3)]
    want = [kv(eng, w, l, p0, M) for l in range(3)]
    # QKV behind an exit at layer 1 (whose rows are under the final norm)
    start(1)
    eng.op_layer(0, 1, M, p0)
    assert np.array_equal(kv(eng, w, 1, p0, M), want[1])
    # the rest of layer 1; gate/up after another kernel's norm has been asked for
    for k in (1, 2):
        eng.op_layer(k, 1, M, p0)
    eng.op_layer(0, 0, M, p0 + 20)
    for k in (3, 4):
        eng.op_layer(k, 1, M, p0)
    eng.op_layer(0, 2, M, p0)
    assert np.array_equal(kv(eng, w, 2, p0, M), want[2])
    # exit head behind layer 2, whose rows are under layer 3's norm: the logits lie
    # where the last call's lie in the workspace
    z = start(1)
    eng.stream.synchronize()
    off = (-eng.workspace.data_ptr()) % 256
    words = eng.workspace[off:off + (eng.workspace.numel() - off) // 4 * 4].view(torch_f32())
    hits = find_row(words, z[0])
    assert len(hits) == 1
    for k in range(5):
        eng.op_layer(k, 1, M, p0)
    eng.op_layer(5, 0, M, p0)
    eng.stream.synchronize()
    got = words[hits[0]:hits[0] + z.size].cpu().numpy().reshape(z.shape)
    assert np.array_equal(got, ref[2])


def torch_f32():
    import torch
    return torch.float32


def find_row(words, row):
    """Offsets of `row` in the float32 tensor `words`."""
    import torch
    c = torch.nonzero(words == float(row[0])).flatten()
    r = torch.from_numpy(row).to(words.device)
    return [int(i) for i in c if int(i) + len(r) <= len(words) and
            torch.equal(words[int(i):int(i) + len(r)], r)]
