"""The work that the engine's users have it do, as cases that can be timed and compared.

Three kinds of call, on the five decoder shapes of synth/workloads.py (the four bf16 ones at their
real widths, vocabularies and context lengths, mostly with fewer layers; the fp32 one whole):

- "exit": ssd_forward_exit on a prefilled sequence: one row is a draft step (or an autoregressive
  step) that ends at an exit layer, 2 to 17 rows are a verification pass of a drafted run;
- "prefill": ssd_prefill of a prompt, then the logits of its last tokens through ssd_forward_exit,
  which read every KV row that the prefill wrote, and the C_trace window it left;
- "generate": ssd_prefill and ssd_generate under a policy, then the last tokens' logits.

Weights are random, made here in torch, and scaled as a trained decoder's are: unit-variance
projections, residual branches that together weigh about as much as the embedding, and an LM head
that predicts a fixed successor of the current token with probability 0.9 or more, at the early exits
too (LayerSkip-trained checkpoints have their drafts accepted at such rates; with plain random weights
a next token is a near-tie, and no two implementations decode the same text).
"""
from __future__ import annotations

import math
from dataclasses import replace

import numpy as np
import torch

import synth
from paper_2606_03113_gb300 import ssd as S
from paper_2606_03113_gb300.runtime import Engine
from synth.workloads import LLAMA2_7B, LLAMA2_13B, LLAMA2_70B, LLAMA3_8B, TINY

FAMILIES = {"tiny": TINY, "7b": LLAMA2_7B, "8b": LLAMA3_8B, "13b": LLAMA2_13B, "70b": LLAMA2_70B}
PEAK_LOGIT = 14.0  # of the successor token, against others' 0 +- 0.2 to 1.4
SAMPLE_SEED = 7
TAIL = 4  # tokens whose logits a prefill or generate case returns


def listed():
    return [
        # the smallest call there is: a verification pass over five rows of the fp32 decoder,
        # where launches and latency are everything
        dict(name="tiny-verify5", kind="exit", family="tiny", layers=4, ctx=40, rows=5, exit=4),
        # a whole short answer of the fp32 decoder under the LEDE policy
        dict(name="tiny-lede", kind="generate", family="tiny", layers=4, ctx=32, new=64,
             policy="lede", l=0, k=4, temp=0.0),
        # a draft (or autoregressive) step in the middle of an answer
        dict(name="7b-draft", kind="exit", family="7b", layers=4, ctx=640, rows=1, exit=4),
        # the static baseline's verification of one draft, at the 13B shape's long context
        dict(name="13b-verify2", kind="exit", family="13b", layers=4, ctx=2176, rows=2, exit=4),
        # grouped queries and the large vocabulary: verification of a full run of 12 drafts
        dict(name="8b-verify13", kind="exit", family="8b", layers=4, ctx=1100, rows=13, exit=4),
        # the widest matrices: a draft step that leaves at an inner layer, and the largest
        # verification pass (16 drafts)
        dict(name="70b-draft", kind="exit", family="70b", layers=2, ctx=1031, rows=1, exit=1),
        dict(name="70b-verify17", kind="exit", family="70b", layers=2, ctx=1024, rows=17, exit=2),
        # prompts: short and ragged, the usual one, and the longest
        dict(name="8b-prompt93", kind="prefill", family="8b", layers=4, ctx=93),
        dict(name="7b-prompt512", kind="prefill", family="7b", layers=4, ctx=512),
        dict(name="13b-prompt2047", kind="prefill", family="13b", layers=4, ctx=2047),
        # speculative sampling over the large vocabulary
        dict(name="8b-sampled", kind="generate", family="8b", layers=4, ctx=48, new=48,
             policy="static", l=2, k=4, temp=0.6),
        # a whole answer of a full-depth model: the LEDE walk over all seven candidates
        dict(name="7b-lede", kind="generate", family="7b", layers=32, ctx=64, new=48,
             policy="lede-walk", l=0, k=12, temp=0.0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    family = rng.choice(["tiny", "7b", "7b", "8b", "8b", "13b", "13b", "70b"])
    w = FAMILIES[family]
    layers = w.shape.n_layers if family == "tiny" else rng.randint(2, 3 if family == "70b" else 6)
    longest = 100 if family == "tiny" else 2300
    kind = rng.choice(["exit", "exit", "prefill", "generate"])
    if kind == "exit":
        rows = rng.choice([1, 1, rng.randint(2, 8), rng.randint(2, w.kmax + 1)])
        return dict(kind=kind, family=family, layers=layers, ctx=_log_int(rng, 4, longest),
                    rows=rows, exit=rng.randint(1, layers))
    if kind == "prefill":
        return dict(kind=kind, family=family, layers=layers, ctx=_log_int(rng, 12, longest))
    policy = rng.choice(["ar", "static", "lede", "lede-walk", "threshold"])
    return dict(kind=kind, family=family, layers=layers, ctx=_log_int(rng, 8, longest // 2),
                new=rng.randint(16, 48), policy=policy, l=rng.randint(1, layers - 1),
                k=rng.randint(1, w.kmax), temp=rng.choice([0.0, 0.0, 0.6]))


# ----------------------------------------------------------------- inputs

def _shape(case):
    s = FAMILIES[case["family"]].shape
    return replace(s, n_layers=case["layers"])


class Weights:
    """A program's own checkpoint, as the engine takes it: per-layer matrices, norms, embedding
    and LM head on the device."""

    def __init__(self, shape, seed):
        self.shape = shape
        self.device = torch.device("cuda:0")
        dt = torch.bfloat16 if shape.dtype == "bf16" else torch.float32
        self.dtype_code = S.SSD_DTYPE_BF16 if shape.dtype == "bf16" else S.SSD_DTYPE_F32
        g = torch.Generator(device=self.device)
        g.manual_seed(seed)

        def normal(*dims, std, mean=0.0):
            return torch.empty(dims, dtype=dt, device=self.device).normal_(mean, std, generator=g)

        d, f, v, L = shape.d_model, shape.ffn_dim, shape.vocab, shape.n_layers
        qd = shape.n_heads * shape.head_dim
        branch = 1.0 / math.sqrt(2 * L)
        self.embed = normal(v, d, std=1.0)
        self.final_norm = normal(d, std=0.1, mean=1.0)
        self.layers = [dict(attn_norm=normal(d, std=0.1, mean=1.0),
                            wqkv=normal(shape.qkv_rows, d, std=1.28 / math.sqrt(d)),
                            wo=normal(d, qd, std=1.28 * branch / math.sqrt(qd)),
                            ffn_norm=normal(d, std=0.1, mean=1.0),
                            w_gate_up=normal(2 * f, d, std=1.28 / math.sqrt(d)),
                            w_down=normal(d, f, std=2.1 * branch / math.sqrt(f)))
                       for _ in range(L)]
        # lm_head row of v's successor: v's embedding, scaled so that its logit is PEAK_LOGIT
        succ = torch.randperm(v, generator=g, device=self.device)
        self.lm_head = torch.empty_like(self.embed)
        self.lm_head[succ] = self.embed * (PEAK_LOGIT / (0.6 * d))


def _ids(case, seed, n):
    rng = np.random.default_rng(seed)
    return rng.integers(0, FAMILIES[case["family"]].shape.vocab, n).astype(np.int32)


def _set_policy(eng, case):
    w = FAMILIES[case["family"]]
    opt = dict(temperature=case["temp"], sample_seed=SAMPLE_SEED) if case["temp"] else {}
    L = case["layers"]
    if case["policy"] == "ar":
        eng.set_ar(**opt)
    elif case["policy"] == "static":
        eng.set_static(case["l"], case["k"], **opt)
    elif case["policy"] == "threshold":
        eng.set_threshold(case["l"], 0.5, case["k"], **opt)
    else:
        cand = sorted({max(1, min(L - 1, round(c * L / w.shape.n_layers))) for c in w.candidates})
        qp = synth.qnet_hidden_params(3, w.qnet_hidden)
        if case["policy"] == "lede-walk":
            # always "continue": every candidate is visited and one token drafted, which is what
            # the Q-network trained on the benchmark's workload does
            qp = np.zeros_like(qp)
            qp[-2] = 1.0
        eng.set_lede(w, qp, kmax=case["k"], cand=cand, **opt)


def prepare(case, seed):
    shape = _shape(case)
    rows = case.get("rows", TAIL)
    need = case["ctx"] + case.get("new", 0) + rows + FAMILIES[case["family"]].kmax + 2
    eng = Engine(Weights(shape, seed), (need + 63) // 64 * 64)
    ids = _ids(case, seed, case["ctx"] + rows)
    if case["kind"] == "generate":
        _set_policy(eng, case)
    else:
        eng.set_ar()
    if case["kind"] == "exit":
        eng.prefill(ids[:case["ctx"]])
    return dict(case=case, eng=eng, ids=ids)


def _logits(eng, ids, pos0, l_exit):
    z, st = eng.forward_exit(ids, pos0, l_exit)
    return dict(logits=z, argmax=np.array([s["argmax"] for s in st]),
                stats=np.array([[s[k] for k in ("lse", "entropy", "conf_k", "pmax")] for s in st]))


def run(state):
    case, eng, ids = state["case"], state["eng"], state["ids"]
    n = case["ctx"]
    if case["kind"] == "exit":
        return _logits(eng, ids[n:n + case["rows"]], n, case["exit"])
    if case["kind"] == "prefill":
        first = eng.prefill(ids[:n - TAIL])
        _, _, trace = eng.read_state()
        return dict(_logits(eng, ids[n - TAIL:n], n - TAIL, case["layers"]), first=first,
                    trace=trace)
    first = eng.prefill(ids[:n])
    tokens, _, _ = eng.generate(case["new"])
    seq = np.concatenate([ids[:n], [first], tokens]).astype(np.int32)
    return dict(_logits(eng, seq[-TAIL:], len(seq) - TAIL, case["layers"]), first=first,
                tokens=tokens)


# ---------------------------------------------------- what a pass cannot do without

def _span(case, layers, rows, ctx, heads=1):
    """Bytes and operations of `rows` rows through `layers` layers after ctx rows of context."""
    s = _shape(case)
    e = s.elt_bytes
    nbytes = layers * (s.layer_weight_bytes() + (ctx + rows) * s.kv_bytes_per_pos_layer())
    keys = rows * ctx + rows * (rows + 1) / 2
    flops = 2 * layers * (rows * s.layer_weight_elems() + 2 * keys * s.n_heads * s.head_dim)
    if heads:
        nbytes += s.lm_head_bytes() + heads * 4 * s.vocab
        flops += 2 * heads * s.vocab * s.d_model
    return nbytes + rows * s.d_model * e, flops


def work(case):
    L, n = case["layers"], case["ctx"]
    if case["kind"] == "exit":
        parts = [_span(case, case["exit"], case["rows"], n, case["rows"])]
    elif case["kind"] == "prefill":
        parts = [_span(case, L, n - TAIL, 0, min(20, n - TAIL)), _span(case, L, TAIL, n - TAIL, TAIL)]
    else:
        # the prompt, then rounds in which every draft is accepted
        l = case["l"] or max(1, L - 4 if case["policy"] == "lede-walk" else L // 8)
        k = {"ar": 0, "lede-walk": 1}.get(case["policy"], case["k"])
        rounds = -(-case["new"] // (k + 1))
        mid = n + case["new"] // 2
        parts = [_span(case, L, n, 0, min(20, n))] + rounds * [_span(case, L, k + 1, mid, k + 1)]
        parts += rounds * k * [_span(case, l, 1, mid, 1)] + [_span(case, L, TAIL, mid, TAIL)]
    return dict(bytes=sum(b for b, _ in parts), flops=sum(f for _, f in parts))


def tolerance(case):
    if case["family"] == "tiny":
        return {"rel": 1e-5}
    return {"rel": 8e-3}


# --------------------------------------------------------- the same in 64 bits

class _Exact:
    """The decoder in fp64 torch, one sequence, keys and values kept unrounded."""

    def __init__(self, case, seed):
        self.s = _shape(case)
        self.w = Weights(self.s, seed)
        self.kv = {}

    def norm(self, x, g):
        return x / torch.sqrt((x * x).mean(-1, keepdim=True) + self.s.rms_eps) * g.double()

    def forward(self, ids, pos0, layers):
        s, dev = self.s, self.w.device
        M, hd, Hq, Hk = len(ids), s.head_dim, s.n_heads, s.n_kv_heads
        h = self.w.embed[torch.as_tensor(np.asarray(ids), device=dev).long()].double()
        pos = torch.arange(pos0, pos0 + M, device=dev, dtype=torch.float64)
        half = torch.arange(hd // 2, device=dev, dtype=torch.float64)
        ang = pos[:, None] * (s.rope_theta ** (-2 * half / hd))[None]
        cos, sin = ang.cos()[:, None], ang.sin()[:, None]

        def rope(x):
            a, b = x[..., :hd // 2], x[..., hd // 2:]
            return torch.cat([a * cos - b * sin, b * cos + a * sin], -1)

        for l in range(layers):
            w = self.w.layers[l]
            qkv = self.norm(h, w["attn_norm"]) @ w["wqkv"].double().T
            q, k, v = (t.view(M, -1, hd) for t in qkv.split([Hq * hd, Hk * hd, Hk * hd], 1))
            q, k = rope(q), rope(k)
            if pos0:
                ko, vo = self.kv[l]
                k, v = torch.cat([ko[:pos0], k]), torch.cat([vo[:pos0], v])
            self.kv[l] = (k, v)
            att = torch.empty(M, Hq, hd, dtype=torch.float64, device=dev)
            seen = torch.arange(pos0 + M, device=dev)[None] <= pos.long()[:, None]
            for g in range(Hk):
                qs = slice(g * (Hq // Hk), (g + 1) * (Hq // Hk))
                z = torch.einsum("mhd,nd->hmn", q[:, qs], k[:, g]) / math.sqrt(hd)
                p = z.masked_fill(~seen, -math.inf).softmax(-1)
                att[:, qs] = torch.einsum("hmn,nd->mhd", p, v[:, g])
            h = h + att.reshape(M, -1) @ w["wo"].double().T
            gu = self.norm(h, w["ffn_norm"]) @ w["w_gate_up"].double().T
            act = torch.nn.functional.silu(gu[:, :s.ffn_dim]) * gu[:, s.ffn_dim:]
            h = h + act @ w["w_down"].double().T
        return h

    def head(self, h):
        z = self.norm(h, self.w.final_norm) @ self.w.lm_head.double().T
        lse = z.logsumexp(-1)
        lp = z - lse[:, None]
        stats = torch.stack([lse, -(lp.exp() * lp).sum(-1), -lp.topk(5).values.mean(-1),
                             lp.max(-1).values.exp()], -1)
        return z, z.argmax(-1), stats


def exact(case, seed):
    rows = case.get("rows", TAIL)
    n, L = case["ctx"], case["layers"]
    ids = _ids(case, seed, n + rows)
    m = _Exact(case, seed)

    def tail(ids_, pos0, layers):
        z, top, stats = m.head(m.forward(ids_, pos0, layers))
        return dict(logits=z.cpu().numpy(), argmax=top.cpu().numpy(), stats=stats.cpu().numpy())

    if case["kind"] == "exit":
        m.forward(ids[:n], 0, case["exit"])
        return tail(ids[n:n + rows], n, case["exit"])
    if case["kind"] == "prefill":
        _, top, stats = m.head(m.forward(ids[:n - TAIL], 0, L)[-20:])
        return dict(tail(ids[n - TAIL:n], n - TAIL, L), first=int(top[-1]),
                    trace=stats[:, 3].cpu().numpy())
    # greedy; at temperature 0.6 the successor's probability leaves about 1e-5 to all others
    seq = list(ids[:n])
    h = m.forward(seq, 0, L)
    for i in range(case["new"] + 1):
        seq.append(int(m.head(h[-1:])[1][0]))
        if i < case["new"]:
            h = m.forward(seq[-1:], len(seq) - 1, L)
    return dict(tail(seq[-TAIL:], len(seq) - TAIL, L), first=seq[n],
                tokens=np.array(seq[n + 1:], dtype=np.int32))
