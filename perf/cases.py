"""The work that is timed: what a program that uses this package has it do, through
the calls that such a program makes, from one draft row to a whole prompt.

Kinds of case (the "kind" of a case):

* linear   op_linear: a bf16 projection at the row counts of a draft pass, a verify
           pass, a tree pass and a batched pass;
* int4     op_linear_int4: a group-wise INT4 projection at decode row counts;
* sample   op_sample: one categorical draw (or argmax) per row of logits;
* step     Engine.step for one or a few requests: the draft's proposals, the
           target's verify pass, acceptance and commit, results read by the host;
* verify   Engine.verify_step for a batch of requests with contexts of their own;
* prefill  Engine.prefill: a prompt through the target into its KV cache.

Weights are N(0, 0.02^2) with norm gains around 1, cached keys and values N(0, 1),
prompts uniform-random ids: random stand-ins of the shapes in seeded_inputs.SHAPES.
Sequences that are decoded are put in place by writing the KV cache, the tokens and
the sequence state, as a program that restores a saved request does.
"""
import dataclasses
import math

import numpy as np
import torch

import paper_2608_10362_gb300 as pkg
from paper_2608_10362_gb300 import _lib
from seeded_inputs import SHAPES

DEV = "cuda"


def listed():
    return [
        # one row through the QKV projection of the 160M draft: the smallest call
        dict(name="linear_draft_qkv", kind="linear", rows=1, n=2304, k=768),
        # the O projection of a 7B target at the K + 1 = 5 rows of a verify pass
        dict(name="linear_verify_o", kind="linear", rows=5, n=4096, k=4096),
        # an LM head of odd size at the 21 rows of a draft tree
        dict(name="linear_tree_lm_head", kind="linear", rows=21, n=32003, k=4096),
        # gate/up of an 8B target at 16 requests x 9 rows
        dict(name="linear_batched_gate_up", kind="linear", rows=144, n=28672, k=4096),
        # the INT4 targets' QKV and down projections at one verify pass's rows and at eight
        dict(name="int4_verify_qkv", kind="int4", rows=5, n=12288, k=4096),
        dict(name="int4_down_8rows", kind="int4", rows=8, n=4096, k=11008),
        # one draft token
        dict(name="sample_one", kind="sample", rows=1, vocab=32000, temp=1.0),
        # every row of a batched pass at a 128K vocabulary
        dict(name="sample_batch", kind="sample", rows=144, vocab=128256, temp=1.0),
        # a decoding step of the 1.1B target with the 68M draft (edge-class pair)
        dict(name="step_edge", kind="step", target="target_1b1", layers=22, draft="draft_68m", batch=1, K=5, ctx=512),
        # a decoding step of the 7B target with the 160M draft: the headline workload
        dict(name="step_7b", kind="step", target="target_7b", layers=32, draft="draft_160m", batch=1, K=4, ctx=2048),
        # 16 requests of 512 to 4096 tokens verified together (8B target, K = 8)
        dict(name="verify_8b_batched", kind="verify", target="target_8b", layers=32, batch=16, K=8, ctx_lo=512,
             ctx_hi=4096),
        # a 2048-token prompt through the 7B target
        dict(name="prefill_7b", kind="prefill", target="target_7b", layers=32, n=2048),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["linear", "linear", "linear", "int4", "int4", "sample", "sample", "step", "verify", "prefill"])
    if kind == "linear":
        return dict(kind=kind, rows=_log(rng, 1, 256), n=_log(rng, 256, 32768), k=8 * _log(rng, 16, 1408))
    if kind == "int4":
        rows, k = rng.randint(1, 16), 128 * _log(rng, 2, 86)
        while rows * (2 * k + 64) + k > 180000:   # the rows have to fit in shared memory
            k -= 128
        return dict(kind=kind, rows=rows, n=_log(rng, 64, 22016), k=k)
    if kind == "sample":
        return dict(kind=kind, rows=_log(rng, 1, 256), vocab=_log(rng, 2000, 131072), temp=rng.choice([0.0, 0.7, 1.0]))
    # whole models: a few layers of the large shapes, so that a case is put up quickly
    target = rng.choice(["draft_160m", "target_1b1", "target_7b", "target_8b"])
    layers = rng.randint(2, 8)
    if kind == "step":
        target = rng.choice(["draft_160m", "target_1b1", "target_7b"])   # the drafts have their vocabulary
        return dict(kind=kind, target=target, layers=layers, draft=rng.choice(["draft_68m", "draft_160m"]),
                    batch=rng.randint(1, 4), K=rng.randint(1, 8), ctx=_log(rng, 64, 3000))
    if kind == "verify":
        lo = _log(rng, 32, 1024)
        return dict(kind=kind, target=target, layers=layers, batch=_log(rng, 1, 16), K=rng.randint(1, 8), ctx_lo=lo,
                    ctx_hi=lo + _log(rng, 1, 3000))
    return dict(kind=kind, target=target, layers=layers, n=_log(rng, 4, 2048))


# ------------------------------------------------------------------ inputs
def _gen(*key):
    return torch.Generator(device=DEV).manual_seed(hash(key) & 0x7FFFFFFFFFFF)


def _randn(key, shape, std=1.0):
    """N(0, std^2) in bf16."""
    return torch.empty(shape, dtype=torch.bfloat16, device=DEV).normal_(0.0, std, generator=_gen(*key))


def _shape(name, layers=None):
    s = SHAPES[name]
    return s if layers is None else dataclasses.replace(s, n_layers=layers)


_STREAM = {"tok_emb": 1, "lm_head": 2, "attn_norm": 3, "ffn_norm": 4, "final_norm": 5, "wq": 6, "wk": 7, "wv": 8,
           "wo": 9, "w_gate": 10, "w_up": 11, "w_down": 12}


def _weight(s, seed, who, name, layer=-1):
    """One bf16 weight tensor: a function of the seed and of its place in the model."""
    d, f = s.d_model, s.d_ffn
    shape = {"tok_emb": (s.vocab, d), "lm_head": (s.vocab, d), "attn_norm": (d,), "ffn_norm": (d,),
             "final_norm": (d,), "wq": (s.q_dim, d), "wk": (s.kv_dim, d), "wv": (s.kv_dim, d), "wo": (d, s.q_dim),
             "w_gate": (f, d), "w_up": (f, d), "w_down": (d, f)}[name]
    key = (seed, who, _STREAM[name], layer)
    if name.endswith("norm"):
        return (1.0 + 0.1 * torch.randn(shape, device=DEV, generator=_gen(*key))).to(torch.bfloat16)
    return _randn(key, shape, 0.02)


def _weights(s, seed, who):
    yield "tok_emb", -1, _weight(s, seed, who, "tok_emb")
    for layer in range(s.n_layers):
        for name in ("attn_norm", "wq", "wk", "wv", "wo", "ffn_norm", "w_gate", "w_up", "w_down"):
            yield name, layer, _weight(s, seed, who, name, layer)
    yield "final_norm", -1, _weight(s, seed, who, "final_norm")
    if not s.tied:
        yield "lm_head", -1, _weight(s, seed, who, "lm_head")


def _kv_view(raw, s, batch, max_seq):
    """The bytes of a KV cache as bf16 [layer][K|V][request][kv head][position][hd]."""
    return raw.view(torch.bfloat16).view(s.n_layers, 2, batch, s.n_kv_heads, max_seq, s.head_dim)


def _fill_kv(raw, seed, who):
    raw.view(torch.bfloat16).normal_(0.0, 1.0, generator=_gen(seed, who, 77))


def _contexts(case, seed):
    """Committed tokens of each request."""
    if case["kind"] == "step":
        return [case["ctx"]] * case["batch"]
    lo, hi = case["ctx_lo"], case["ctx_hi"]
    # the lengths belong to the case and not to the seed: its work is the same for every seed
    r = np.random.default_rng([11, case["batch"], lo, hi])
    return [int(v) for v in r.integers(lo, hi + 1, size=case["batch"])]


def _max_seq(case):
    if case["kind"] == "step":
        return case["ctx"] + 4096       # room for the tokens that are generated
    if case["kind"] == "verify":
        return case["ctx_hi"] + 2 * (case["K"] + 1)
    return case["n"] + 64


def _tokens(case, seed, vocab):
    r = np.random.default_rng([seed, 3])
    B, n = (1, case["n"]) if case["kind"] == "prefill" else (case["batch"], _max_seq(case))
    return r.integers(0, vocab, size=(B, n)).astype(np.int32)


def _draft_tokens(case, seed, vocab):
    return np.random.default_rng([seed, 4]).integers(0, vocab, size=(case["batch"], case["K"])).astype(np.int32)


# ------------------------------------------------------------------ prepare / run
@dataclasses.dataclass
class State:
    case: dict
    x: torch.Tensor = None
    w: torch.Tensor = None
    scratch: torch.Tensor = None
    u: torch.Tensor = None
    eng: object = None
    prompt: np.ndarray = None


def _linear_inputs(case, seed):
    return _randn((seed, 1), (case["rows"], case["k"])), _randn((seed, 2), (case["n"], case["k"]), 0.02)


def _int4_inputs(case, seed):
    n, k, g = case["n"], case["k"], _gen(seed, 5)
    q = torch.randint(0, 256, (n, k // 2), dtype=torch.uint8, device=DEV, generator=g)
    s = (torch.rand(n, k // 128, device=DEV, generator=g) * 0.006 + 0.002).to(torch.bfloat16)
    z = torch.randint(0, 16, (n, k // 128), dtype=torch.uint8, device=DEV, generator=g)
    return _randn((seed, 1), (case["rows"], k)), q, s, z


def _sample_inputs(case, seed):
    g = _gen(seed, 6)
    z = torch.randn(case["rows"], case["vocab"], device=DEV, generator=g) * 3.0
    u = (2 * torch.randint(0, 1 << 23, (case["rows"],), device=DEV, generator=g) + 1).double() * 2.0 ** -24
    return z, u.float()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "linear":
        x, w = _linear_inputs(case, seed)
        # the split-K scratch that a program keeps for its projections
        return State(case, x=x, w=w, scratch=torch.zeros(64 << 20, dtype=torch.uint8, device=DEV))
    if kind == "int4":
        x, q, s, z = _int4_inputs(case, seed)
        return State(case, x=x, w=pkg.int4_pack(q, s, z))
    if kind == "sample":
        z, u = _sample_inputs(case, seed)
        return State(case, x=z, u=u)
    t = _shape(case["target"], case["layers"])
    max_seq = _max_seq(case)
    if kind == "prefill":
        eng = pkg.Engine(t, _weights(t, seed, 1), max_batch=1, max_seq=max_seq, max_k=4, max_drafts=0)
        return State(case, eng=eng, prompt=_tokens(case, seed, t.vocab)[0])
    B, K = case["batch"], case["K"]
    if kind == "step":
        d = _shape(case["draft"])
        eng = pkg.Engine(t, _weights(t, seed, 1), max_batch=B, max_seq=max_seq, max_k=K, max_drafts=1,
                         draft_shape_max=d, draft_budget_bytes=pkg.weights_bytes(d) + (1 << 20))
        eng.register_draft(0, d, _weights(d, seed, 2))
        eng.load_draft_async(0)
        eng.set_active_draft(0)
        _fill_kv(eng.drafts[0][2], seed, 2)
    else:
        eng = pkg.Engine(t, _weights(t, seed, 1), max_batch=B, max_seq=max_seq, max_k=K, max_drafts=0)
    _fill_kv(eng.kv, seed, 1)
    torch.cuda.synchronize()
    st = np.zeros((B, 4), dtype=np.int32)
    st[:, 0] = _contexts(case, seed)
    st[:, 1] = st[:, 3] = st[:, 0] - 1
    eng.write_buffer(_lib.BUF_TOKENS, _tokens(case, seed, t.vocab))
    eng.write_buffer(_lib.BUF_SEQ_STATE, st)
    if kind == "verify":
        eng.write_buffer(_lib.BUF_DRAFT_TOKENS, _draft_tokens(case, seed, t.vocab))
    eng.set_batch(B)
    return State(case, eng=eng)


def run(state):
    case, kind = state.case, state.case["kind"]
    if kind == "linear":
        return pkg.op_linear(state.x, state.w, state.scratch)
    if kind == "int4":
        return pkg.op_linear_int4(state.x, state.w, case["n"])
    if kind == "sample":
        return pkg.op_sample(state.x, case["temp"], state.u)
    eng = state.eng
    if kind == "prefill":
        eng.prefill(0, state.prompt, seed=1)
        s = eng.shape
        return _kv_view(eng.kv, s, 1, eng.max_seq)[:, :, 0, :, :case["n"] - 1]
    B, K = case["batch"], case["K"]
    if kind == "step":
        # greedy decoding; the program reads the step's outcome before the next
        eng.step(K, 0.0, eng.results_host)
        eng.sync()
        return {"results": eng.results_host, "logits": eng.target_logits(B, K)}
    eng.verify_step(K)
    kv = _kv_view(eng.kv, eng.shape, B, eng.max_seq)
    return {"logits": eng.target_logits(B, K),
            "kv": [kv[:, :, b, :, L - 1:L + K] for b, L in enumerate(_contexts(case, 0))]}


# ------------------------------------------------------------------ what a pass needs
def _model_bytes(s, head):
    per = (s.q_dim + 2 * s.kv_dim) * s.d_model + s.d_model * s.q_dim + 3 * s.d_ffn * s.d_model + 2 * s.d_model
    return 2 * (s.n_layers * per + (s.d_model + s.vocab * s.d_model if head else 0))


def _model_flops(s, rows, keys, head_rows):
    """rows rows through the layers, `keys` (row, key) pairs of attention, head_rows rows of logits."""
    per = (s.q_dim + 2 * s.kv_dim) * s.d_model + s.d_model * s.q_dim + 3 * s.d_ffn * s.d_model
    return 2 * rows * s.n_layers * per + 4 * keys * s.n_layers * s.q_dim + 2 * head_rows * s.vocab * s.d_model


def _pass_work(s, ctxs, R):
    """A pass over R new rows per request, the request's context before them."""
    kv = 2 * 2 * s.n_layers * s.kv_dim
    rows = R * len(ctxs)
    keys = sum(R * c + R * (R + 1) // 2 for c in ctxs)
    return (_model_bytes(s, True) + kv * (sum(ctxs) + rows) + 2 * rows * s.d_model + 4 * rows * s.vocab,
            _model_flops(s, rows, keys, rows))


def work(case):
    kind = case["kind"]
    if kind == "linear":
        r, n, k = case["rows"], case["n"], case["k"]
        return {"bytes": 2 * n * k + 2 * r * k + 4 * r * n, "flops": 2 * r * n * k}
    if kind == "int4":
        r, n, k = case["rows"], case["n"], case["k"]
        return {"bytes": n * k // 2 + 3 * n * (k // 128) + 2 * r * k + 4 * r * n, "flops": 2 * r * n * k}
    if kind == "sample":
        return {"bytes": 4 * case["rows"] * case["vocab"], "flops": 2 * case["rows"] * case["vocab"]}
    t = _shape(case["target"], case["layers"])
    if kind == "prefill":
        n = case["n"] - 1
        return {"bytes": _model_bytes(t, False) + n * (2 * t.d_model + 4 * t.n_layers * t.kv_dim),
                "flops": _model_flops(t, n, n * (n + 1) // 2, 0)}
    ctxs = [c - 1 for c in _contexts(case, 0)]
    b, f = _pass_work(t, ctxs, case["K"] + 1)
    if kind == "step":
        d = _shape(case["draft"])
        for j in range(case["K"]):
            db, df = _pass_work(d, [c + j for c in ctxs], 1)
            b, f = b + db, f + df
    return {"bytes": b, "flops": f}


def tolerance(case):
    """About four times the distance from exact() that was measured."""
    kind = case["kind"]
    if kind == "linear":
        return {"rel": 4e-5}         # 32-bit sums of exact products: 4e-6 at k = 4096, 1.1e-5 at the longest sums
    if kind == "int4":
        return {"rel": 4e-6}         # as above: 0.5e-6 to 0.9e-6
    if kind == "sample":
        return {"rel": 0.0, "differ": 0.01}   # u within a rounding of a boundary between two ids
    if kind == "step":
        return {"rel": 6e-4}         # logits: 3e-5 to 1.5e-4 (keys and values rounded to bf16 on the way)
    if kind == "verify":
        return {"rel": 2.5e-3}       # new keys and values in bf16: up to 6e-4
    return {"rel": 1e-2}             # bf16 keys and values, each layer's from the last's: 1.7e-3 after a few layers


# ------------------------------------------------------------------ 64-bit values
def _rms(h, gain, eps):
    return h * torch.rsqrt((h * h).mean(-1, keepdim=True) + eps) * gain.double()


def _rope(x, pos, base):
    """x [rows][heads][hd], rotated on the pairs (i, i + hd/2)."""
    half = x.shape[-1] // 2
    inv = base ** (-2.0 * torch.arange(half, dtype=torch.float64, device=DEV) / x.shape[-1])
    ang = pos.double()[:, None] * inv[None]
    c, s = ang.cos()[:, None], ang.sin()[:, None]
    a, b = x[..., :half], x[..., half:]
    return torch.cat([a * c - b * s, a * s + b * c], -1)


def _forward64(s, seed, who, toks, starts, kv, head=True):
    """Rows toks[g][i] of request g at positions starts[g] + i against the bf16 cache
    kv, which takes the rows' keys and values.  Logits [g][i][vocab]."""
    W = lambda name, layer=-1: _weight(s, seed, who, name, layer)
    G, R = toks.shape
    h = W("tok_emb")[torch.as_tensor(toks.reshape(-1).astype(np.int64), device=DEV)].double()
    pos = torch.cat([torch.arange(st, st + R, device=DEV) for st in starts])
    gs = s.n_heads // s.n_kv_heads
    for l in range(s.n_layers):
        x = _rms(h, W("attn_norm", l), s.norm_eps)
        q = _rope((x @ W("wq", l).double().T).view(-1, s.n_heads, s.head_dim), pos, s.rope_base)
        k = _rope((x @ W("wk", l).double().T).view(-1, s.n_kv_heads, s.head_dim), pos, s.rope_base)
        v = (x @ W("wv", l).double().T).view(-1, s.n_kv_heads, s.head_dim)
        outs = []
        for g, st in enumerate(starts):
            sl = slice(g * R, (g + 1) * R)
            kv[l, 0, g, :, st:st + R] = k[sl].transpose(0, 1).to(torch.bfloat16)
            kv[l, 1, g, :, st:st + R] = v[sl].transpose(0, 1).to(torch.bfloat16)
            keys, vals = kv[l, 0, g, :, :st + R].double(), kv[l, 1, g, :, :st + R].double()
            qg = q[sl].view(R, s.n_kv_heads, gs, s.head_dim).permute(1, 2, 0, 3)           # [kvh][gs][R][hd]
            sc = qg @ keys[:, None].transpose(-1, -2) / math.sqrt(s.head_dim)
            seen = torch.arange(st + R, device=DEV)[None] <= torch.arange(st, st + R, device=DEV)[:, None]
            p = sc.masked_fill(~seen, -math.inf).softmax(-1)
            outs.append((p @ vals[:, None]).permute(2, 0, 1, 3).reshape(R, -1))
        h = h + torch.cat(outs) @ W("wo", l).double().T
        x = _rms(h, W("ffn_norm", l), s.norm_eps)
        a = torch.nn.functional.silu(x @ W("w_gate", l).double().T) * (x @ W("w_up", l).double().T)
        h = h + a @ W("w_down", l).double().T
    if not head:
        return None
    lm = W("tok_emb" if s.tied else "lm_head")
    return (_rms(h, W("final_norm"), s.norm_eps) @ lm.double().T).view(G, R, -1)


def exact(case, seed):
    kind = case["kind"]
    if kind == "linear":
        x, w = _linear_inputs(case, seed)
        return x.double() @ w.double().T
    if kind == "int4":
        x, q, s, z = _int4_inputs(case, seed)
        codes = torch.stack([q & 15, q >> 4], -1).view(case["n"], -1).double()
        rep = lambda t: t.double().repeat_interleave(128, 1)
        return x.double() @ ((codes - rep(z)) * rep(s)).T
    if kind == "sample":
        return None          # whole numbers: a draw has no value in more bits
    if work(case)["flops"] > 8e12:
        return None          # 64-bit products of this size take too long
    t = _shape(case["target"], case["layers"])
    max_seq = _max_seq(case)
    B = 1 if kind == "prefill" else case["batch"]
    kv = torch.zeros(pkg.kv_bytes(t, B, max_seq), dtype=torch.uint8, device=DEV)
    toks = _tokens(case, seed, t.vocab)
    if kind == "prefill":
        n = case["n"] - 1
        kv = _kv_view(kv, t, 1, max_seq)
        for at in range(0, n, 512):
            _forward64(t, seed, 1, toks[:, at:min(n, at + 512)], [at], kv, head=False)
        return kv[:, :, 0, :, :n].double()
    _fill_kv(kv, seed, 1)
    kv = _kv_view(kv, t, B, max_seq)
    ctxs = _contexts(case, seed)
    first = np.stack([toks[b, c - 1:c] for b, c in enumerate(ctxs)])     # the last committed token
    if kind == "verify":
        rows = np.concatenate([first, _draft_tokens(case, seed, t.vocab)], 1)
        logits = _forward64(t, seed, 1, rows, [c - 1 for c in ctxs], kv)
        K = case["K"]
        return {"logits": logits, "kv": [kv[:, :, b, :, c - 1:c + K].double() for b, c in enumerate(ctxs)]}
    d = _shape(case["draft"])
    dkv = torch.zeros(pkg.kv_bytes(d, B, max_seq), dtype=torch.uint8, device=DEV)
    _fill_kv(dkv, seed, 2)
    dkv = _kv_view(dkv, d, B, max_seq)
    rows = first
    for j in range(case["K"]):
        z = _forward64(d, seed, 2, rows[:, -1:], [c - 1 + j for c in ctxs], dkv)
        rows = np.concatenate([rows, z.argmax(-1).cpu().numpy().astype(np.int32)], 1)
    return {"results": None, "logits": _forward64(t, seed, 1, rows, [c - 1 for c in ctxs], kv)}
