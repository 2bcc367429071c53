"""End-to-end parity of the draft-then-verify step on the GPU against the oracle,
in lock step (tests/lockstep.py), on the tiny pair: every launch mode at T = 0
and T = 1, a batch of four requests, the greedy stream against greedy
target-only decoding, and prompt edge cases."""
import numpy as np
import pytest
import torch

from lockstep import LOGIT_TOL, RECORDS, LockstepReport, check_step
from oracle.llama import LlamaOracle
from oracle.speculative import SpecDecoder, argmax_first, greedy_generate
from seeded_inputs import SHAPES, gen_prompt, gen_weights

pytestmark = pytest.mark.gpu


def _run_lockstep(eng, target_o, draft_o, prompt, K, T, seed, steps):
    eng.prefill(0, prompt, seed=seed)
    sd = SpecDecoder(target_o, draft_o, prompt, len(prompt) + steps * (K + 1) + 4)
    rep = LockstepReport()
    for step in range(steps):
        eng.step(K, T, eng.results_host)
        check_step(eng, sd, K, T, seed, step, rep)
    return rep, sd


# (CUDA graphs, launch mode): per-op launches with and without graphs, and the
# persistent pass kernel
MODES = [(False, "per_op"), (True, "per_op"), (True, "pass"), (False, "pass")]


def _engine(t, wt, d, wd, graphs, launch, max_batch=1, draft_kernel="auto"):
    from paper_2608_10362_gb300 import Engine
    eng = Engine(t, wt, max_batch=max_batch, max_seq=512, max_k=8, max_drafts=1,
                 draft_shape_max=d, draft_budget_bytes=32 << 20, use_graphs=graphs,
                 launch_mode=launch, draft_kernel=draft_kernel)
    eng.register_draft(0, d, wd)
    eng.load_draft_async(0)
    eng.set_active_draft(0)
    return eng


@pytest.fixture(scope="module")
def tiny():
    t, d = SHAPES["tiny_target"], SHAPES["tiny_draft"]
    wt, wd = gen_weights(t, 0), gen_weights(d, 1)
    engines = {mode: _engine(t, wt, d, wd, *mode) for mode in MODES}
    yield engines, LlamaOracle(t, wt), LlamaOracle(d, wd), (t, wt, d, wd)
    for e in engines.values():
        e.close()


@pytest.mark.parametrize("mode", MODES, ids=lambda m: f"graphs{int(m[0])}-{m[1]}")
@pytest.mark.parametrize("T", [0.0, 1.0])
def test_tiny_pair_lockstep(tiny, T, mode):
    engines, to, do, _ = tiny
    eng = engines[mode]
    prompt = gen_prompt(7, 128, 2048)
    rep, sd = _run_lockstep(eng, to, do, prompt, 4, T, seed=3, steps=16)
    line = rep.record(f"tiny T={T} graphs={int(mode[0])} {mode[1]}")
    assert rep.band_flags == 0, line
    assert list(eng.committed_tokens(0)) == sd.tokens


@pytest.mark.parametrize("B", [1, 4])
@pytest.mark.parametrize("T", [0.0, 1.0])
def test_tiny_pair_lockstep_fused_draft_kernel(tiny, T, B):
    """The draft step as one launch (draft_kernel "fused"), one and four requests."""
    from paper_2608_10362_gb300 import _lib
    _, to, do, (t, wt, d, wd) = tiny
    eng = _engine(t, wt, d, wd, True, "per_op", max_batch=B, draft_kernel="fused")
    prompts = [gen_prompt(27 + b, 100 + 9 * b, 2048) for b in range(B)]
    sds = []
    for b, p in enumerate(prompts):
        eng.prefill(b, p, seed=5 + b)
        sds.append(SpecDecoder(to, do, p, 256))
    eng.set_batch(B)
    rep = LockstepReport()
    for step in range(6):
        eng.step(4, T, eng.results_host)
        for b in range(B):
            check_step(eng, sds[b], 4, T, 5 + b, step, rep, req=b, batch=B)
    assert eng.info(_lib.INFO_DRAFT_FUSED) == 1
    line = rep.record(f"tiny fused draft kernel T={T} B={B}")
    eng.close()
    assert rep.band_flags == 0, line


def test_tiny_pair_lockstep_per_op_draft_path(tiny):
    """The draft step through the per-op kernels (the path larger drafts take),
    T = 1."""
    _, to, do, (t, wt, d, wd) = tiny
    eng = _engine(t, wt, d, wd, True, "per_op", draft_kernel="per_op")
    prompt = gen_prompt(17, 128, 2048)
    rep, sd = _run_lockstep(eng, to, do, prompt, 4, 1.0, seed=13, steps=12)
    line = rep.record("tiny T=1.0 per-op draft kernels")
    eng.close()
    assert rep.band_flags == 0, line


@pytest.mark.parametrize("T", [0.0, 1.0])
@pytest.mark.parametrize("launch", ["per_op", "pass"])
def test_tiny_pair_lockstep_batch4(tiny, T, launch):
    """Four requests stepped together (per-request lengths, Philox keys and
    KV caches): draft step, verify pass and acceptance at B = 4."""
    _, to, do, (t, wt, d, wd) = tiny
    B, K, steps = 4, 4, 8
    eng = _engine(t, wt, d, wd, True, launch, max_batch=B)
    lens = [128, 61, 130, 97]
    seeds = [21, 22, 23, 24]
    sds = []
    for b in range(B):
        prompt = gen_prompt(40 + b, lens[b], 2048)
        eng.prefill(b, prompt, seed=seeds[b])
        sds.append(SpecDecoder(to, do, prompt, len(prompt) + steps * (K + 1) + 4))
    eng.set_batch(B)
    rep = LockstepReport()
    for step in range(steps):
        eng.step(K, T, eng.results_host)
        bits = eng.sync()
        for b in range(B):
            check_step(eng, sds[b], K, T, seeds[b], step, rep, req=b, batch=B, bits=bits)
        res = eng.results_host.numpy()[:B * (K + 2)].reshape(B, K + 2)
        for b in range(B):      # the pinned result rows agree with the committed tokens
            n = int(res[b, 0])
            assert list(res[b, 1:n + 2]) == sds[b].tokens[-(n + 1):]
    line = rep.record(f"tiny B=4 T={T} {launch}")
    for b in range(B):
        assert list(eng.committed_tokens(b)) == sds[b].tokens
    eng.close()
    assert rep.band_flags == 0, line


def test_tiny_greedy_stream_equals_oracle_target_greedy(tiny):
    """Greedy speculative output == greedy target-only output, token for token,
    over the whole stream.  A divergence is allowed only where the oracle's two
    candidates are closer than the logit tolerance (0.03 max|z|); it is
    counted, the GPU is resynchronised to the oracle's token (prefill of the
    prompt plus the oracle's tokens so far) and the comparison continues."""
    engines, to, do, _ = tiny
    eng = engines[(True, "per_op")]
    n_new = 40
    flagged = []
    for seed in (8, 9, 10):
        prompt = [int(x) for x in gen_prompt(seed, 128, 2048)]
        ref = greedy_generate(to, prompt, n_new)
        i = 0
        while i < n_new:
            ctx = prompt + ref[:i]
            eng.prefill(0, ctx, seed=0)
            while int(eng.seq_state()[0, 0]) < len(ctx) + (n_new - i):
                eng.step(4, 0.0, eng.results_host)
                assert eng.sync() == 0
            got = [int(t) for t in eng.committed_tokens(0)[len(ctx):len(ctx) + n_new - i]]
            j = next((k for k in range(len(got)) if got[k] != ref[i + k]), None)
            if j is None:
                break
            pos = i + j
            z = to.forward(to.new_cache(len(prompt) + pos + 1), prompt + ref[:pos])[-1]
            gap = float(z[ref[pos]] - z[got[j]])
            assert ref[pos] == argmax_first(z)
            assert 0 <= gap < LOGIT_TOL * np.abs(z).max(), (seed, pos, gap)
            flagged.append((seed, pos, f"{gap / np.abs(z).max():.2e}"))
            i = pos + 1                        # resync on the oracle's token
    RECORDS.append(f"tiny greedy streams (3 x {n_new} tokens): tolerance-flags {len(flagged)} "
                   f"{flagged}")


def test_tiny_prompt_edge_cases(tiny):
    """Prompt of one token (nothing to prefill) and a prompt crossing the
    128-row prefill chunk boundary by one."""
    engines, to, do, _ = tiny
    eng = engines[(False, "per_op")]
    for n in (1, 129):
        prompt = gen_prompt(9 + n, n, 2048)
        rep, sd = _run_lockstep(eng, to, do, prompt, 3, 1.0, seed=5, steps=4)
        rep.record(f"tiny prompt length {n}")
        assert rep.steps == 4
        assert rep.band_flags == 0


@pytest.mark.parametrize("B,K", [(1, 1), (2, 3), (1, 8), (3, 3), (2, 8), (3, 10), (8, 15), (9, 14), (10, 15), (16, 15)])
def test_verify_pass_row_counts(B, K):
    """One verify pass at 2, 8, 9, 12, 18, 33, 128, 135, 160 and 256 rows (up to 8: the
    small GEMM; above: the CTA-pair GEMM's operand layouts, two planes side by side up
    to 128 rows, one after the other above), requests of different lengths: every
    request's logits, keys and values against the oracle at the step tests' tolerance."""
    from oracle.llama import LlamaOracle
    from paper_2608_10362_gb300 import Engine, _lib
    from seeded_inputs import SHAPES, gen_prompt, gen_weights
    t = SHAPES["tiny_target"]
    wt = gen_weights(t, 0)
    oracle = LlamaOracle(t, wt, keep_f64=True)
    eng = Engine(t, wt, max_batch=B, max_seq=96, max_k=K, max_drafts=0, use_graphs=False)
    try:
        prompts = [gen_prompt(40 + b, 3 + 5 * (b % 7), t.vocab) for b in range(B)]
        for b, p in enumerate(prompts):
            eng.prefill(b, p, seed=b)
        x = np.stack([gen_prompt(80 + b, K, t.vocab) for b in range(B)]).astype(np.int32)
        eng.set_batch(B)
        eng.write_buffer(_lib.BUF_DRAFT_TOKENS, x)
        eng.verify_step(K)
        assert eng.sync() == 0
        z = eng.target_logits(B, K)
        kv = eng.kv.view(torch.bfloat16).view(t.n_layers, 2, B, t.n_kv_heads, 96, t.head_dim).float().cpu().numpy()
        for b, p in enumerate(prompts):
            cache = oracle.new_cache(96)
            rows = np.concatenate([p, x[b]])
            ref = oracle.forward(cache, rows)[-(K + 1):]
            assert np.abs(z[b] - ref).max() <= 1e-3 * np.abs(ref).max()
            n = len(rows)
            for side, cached in enumerate((cache.k, cache.v)):   # [layer][pos][head][hd]
                kv_ref = np.stack([np.asarray(cached[l])[:n] for l in range(t.n_layers)])
                got = kv[:, side, b, :, :n].transpose(0, 2, 1, 3)
                # bf16 values: at most one rounding step apart
                assert np.abs(got - kv_ref).max() <= 2.0 ** -7 * np.abs(kv_ref).max()
    finally:
        eng.close()


_MANY = [(2, 2, 64, 1), (16, 2, 64, 3), (16, 2, 64, 4), (16, 2, 64, 7), (16, 2, 64, 8), (16, 2, 64, 15), (1, 1, 128, 8),
         (4, 1, 128, 8), (12, 1, 128, 10)]
_LENS = [(3,), (120, 128, 129), (258, 265, 266), (1100, 30)]
_WIDE = [((32, 16, 64, 4), (3, 500, 130, 1000, 64, 257)), ((16, 16, 128, 8), (3, 500, 130, 1000, 64, 257)),
         ((128, 16, 64, 8), (5, 700, 5, 5, 130, 5)), ((32, 16, 64, 4), (90, 90, 90, 90, 90, 90))]


@pytest.mark.parametrize("H,Hkv,hd,K,lens", [(*m, l) for l in _LENS for m in _MANY] + [(*m, l) for m, l in _WIDE])
def test_attention_of_many_vectors(H, Hkv, hd, K, lens):
    """Verify passes of 2 to 132 query vectors per KV head (the tcgen05 attention kernel's
    four, two and one copies of the vectors and a second row block; every head size), with
    contexts around a tile of 128 keys, in one tile and in many (clusters of one to eight
    CTAs, some without keys; 96 units: one CTA each): logits against the oracle at the step tests' tolerance.  The
    prompts' prefill runs row blocks of up to 128 vectors, and last passes of 1, 8 and 9
    rows."""
    from paper_2608_10362_gb300 import Engine, _lib
    from seeded_inputs import ModelShape
    t = ModelShape(1, 256, H, Hkv, hd, 256, 512)
    wt = gen_weights(t, 3)
    oracle = LlamaOracle(t, wt, keep_f64=True)
    B, S = len(lens), max(lens) + 32
    eng = Engine(t, wt, max_batch=B, max_seq=S, max_k=K, max_drafts=0, use_graphs=False)
    try:
        prompts = [gen_prompt(60 + b, n, t.vocab) for b, n in enumerate(lens)]
        for b, p in enumerate(prompts):
            eng.prefill(b, p, seed=b)
        x = np.stack([gen_prompt(90 + b, K, t.vocab) for b in range(B)]).astype(np.int32)
        eng.set_batch(B)
        eng.write_buffer(_lib.BUF_DRAFT_TOKENS, x)
        eng.verify_step(K)
        assert eng.sync() == 0
        z = eng.target_logits(B, K)
        for b, p in enumerate(prompts):
            ref = oracle.forward(oracle.new_cache(S), np.concatenate([p, x[b]]))[-(K + 1):]
            assert np.abs(z[b] - ref).max() <= 1e-3 * np.abs(ref).max()
    finally:
        eng.close()


@pytest.mark.parametrize("rows", [144, 256])
def test_prefill_is_as_exact_in_large_passes(rows):
    """Values that one prefill pass of 144 or 256 rows leaves in the cache, against the
    64-bit ones rounded to bf16: the share that differs is proportional to the error of
    the projection's sums before they are rounded, and no larger than a pass of 128
    rows leaves (1.5 times: about 90 of 131072 values differ there, so chance is 1.1 to
    1.3; sums of both planes in one accumulator give 2).  Stream-K ranges of 16.8 k
    tiles of 64: most CTA pairs work on two row tiles."""
    from paper_2608_10362_gb300 import Engine
    from seeded_inputs import ModelShape
    t = ModelShape(1, 4096, 24, 8, 128, 256, 1000)
    g = torch.Generator(device="cuda").manual_seed(31)
    normal = lambda *shape: torch.randn(shape, device="cuda", generator=g)
    d, f, q, kv = t.d_model, t.d_ffn, t.q_dim, t.kv_dim
    w = {"tok_emb": normal(t.vocab, d) * 0.02, "attn_norm": 1 + 0.1 * normal(d), "wq": normal(q, d) * 0.02,
         "wk": normal(kv, d) * 0.02, "wv": normal(kv, d) * 0.02, "wo": normal(d, q) * 0.02,
         "ffn_norm": 1 + 0.1 * normal(d), "w_gate": normal(f, d) * 0.02, "w_up": normal(f, d) * 0.02,
         "w_down": normal(d, f) * 0.02, "final_norm": 1 + 0.1 * normal(d), "lm_head": normal(t.vocab, d) * 0.02}
    w = {name: v.to(torch.bfloat16) for name, v in w.items()}
    model = ("tok_emb", "final_norm", "lm_head")
    eng = Engine(t, [(name, -1 if name in model else 0, v) for name, v in w.items()], max_batch=1, max_seq=300,
                 max_k=4, max_drafts=0, use_graphs=False)
    try:
        def share(n):
            prompt = gen_prompt(n, n + 1, t.vocab)     # the last token is the next pass's
            eng.prefill(0, prompt, seed=1)
            assert eng.sync() == 0
            got = eng.kv.view(torch.bfloat16).view(2, t.n_kv_heads, 300, t.head_dim)[1, :, :n].transpose(0, 1)
            h = w["tok_emb"][torch.as_tensor(prompt[:n].astype(np.int64), device="cuda")].double()
            x = h * torch.rsqrt((h * h).mean(-1, keepdim=True) + t.norm_eps) * w["attn_norm"].double()
            ref = (x @ w["wv"].double().T).view(n, t.n_kv_heads, t.head_dim)
            assert (got.double() - ref).abs().max() <= 2.0 ** -8 * ref.abs().max()
            return (got != ref.to(torch.bfloat16)).double().mean().item()
        assert 0 < share(rows) <= 1.5 * share(128)
    finally:
        eng.close()
