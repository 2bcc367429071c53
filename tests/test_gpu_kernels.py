"""Kernel-level parity on the GPU (through the C ABI): the weight-streaming GEMM,
the categorical sampler, and the acceptance / resample / commit kernel fed with
synthetic logits, against the oracle's definitions."""
import ctypes as C

import numpy as np
import pytest
import torch

from oracle.philox import step_uniforms
from oracle.speculative import accept, draft_token, softmax_t
from seeded_inputs import SHAPES, bf16_round, gen_logits, gen_weights

pytestmark = pytest.mark.gpu


def _bf16_pair(seed, rows, n_out, k):
    rng = np.random.default_rng([seed, rows, n_out, k])
    x = bf16_round(rng.standard_normal((rows, k), dtype=np.float32))
    w = bf16_round((rng.standard_normal((n_out, k), dtype=np.float32) * 0.02).astype(np.float32))
    return x, w


@pytest.mark.parametrize("rows,n_out,k", [
    (1, 256, 128), (5, 768, 256), (9, 688, 256), (16, 256, 688), (17, 2048, 2048),
    (6, 2560, 2048), (144, 1024, 4096), (128, 384, 352), (2, 640, 768), (256, 256, 256),
    # up to 16 rows: one row tile, k of less than one, one and more than four k tiles, k not
    # whole tiles, many row tiles per CTA, ranges that end inside a row tile
    (16, 1, 8), (3, 128, 64), (9, 129, 328), (16, 300, 320), (1, 128, 4096), (7, 40000, 72), (8, 2560, 2048),
    (13, 5000, 1000),
    # CTA pairs (from 161 rows): odd row tiles, one tile, ragged n and k, many tiles per pair
    (161, 129, 8), (161, 128, 64), (176, 300, 72), (193, 385, 4104), (255, 20001, 328), (256, 1, 1000),
])
def test_linear_matches_fp64_matmul(rows, n_out, k):
    from paper_2608_10362_gb300 import op_linear
    x, w = _bf16_pair(1, rows, n_out, k)
    xt = torch.from_numpy(x).to(torch.bfloat16).cuda()
    wt = torch.from_numpy(w).to(torch.bfloat16).cuda()
    scratch = torch.zeros(64 << 20, dtype=torch.uint8, device="cuda")
    y = op_linear(xt, wt, scratch).cpu().numpy().astype(np.float64)
    ref = x.astype(np.float64) @ w.astype(np.float64).T
    bound = np.abs(x).astype(np.float64) @ np.abs(w).astype(np.float64).T
    err = np.abs(y - ref)
    assert np.all(err <= 1e-4 * bound + 1e-6), (err.max(), np.unravel_index(err.argmax(), err.shape))
    # a second launch reuses the same scratch: counters must have been reset
    y2 = op_linear(xt, wt, scratch).cpu().numpy().astype(np.float64)
    np.testing.assert_array_equal(y, y2)      # deterministic split-K reduction


def test_linear_calls_of_all_row_counts_share_one_scratch():
    """One scratch, zeroed once, for calls of every row count and size in turn, as a
    program keeps it for its projections.  The calls of up to 16 rows are of sizes
    whose split row tiles no cluster holds (12, 48 and 24 row tiles of 47 k tiles), so
    that they count arrivals in the scratch; the others leave partial sums in it.  y is
    full of NaN before each call: a row tile that no CTA finishes shows."""
    from paper_2608_10362_gb300 import _lib
    lib = _lib.load()
    sizes = [(5, 1500, 3000), (32, 12288, 4096), (5, 1500, 3000), (200, 12288, 4096), (16, 6100, 3000),
             (256, 300, 4096), (1, 3000, 3000), (17, 40000, 1000), (5, 1500, 3000), (16, 40000, 72), (5, 6100, 3000)]
    need = C.c_size_t()
    nbytes = 0
    for rows, n_out, k in sizes:
        assert lib.memspec_op_linear_scratch_bytes(rows, n_out, k, C.byref(need)) == 0
        nbytes = max(nbytes, need.value)
    scratch = torch.zeros(nbytes + 256, dtype=torch.uint8, device="cuda")
    base = (scratch.data_ptr() + 255) // 256 * 256
    g = torch.Generator(device="cuda").manual_seed(8)
    for rows, n_out, k in sizes:
        x = torch.randn(rows, k, device="cuda", generator=g).to(torch.bfloat16)
        w = (torch.randn(n_out, k, device="cuda", generator=g) * 0.02).to(torch.bfloat16)
        y = torch.full((rows, n_out), float("nan"), device="cuda")
        st = lib.memspec_op_linear(x.data_ptr(), w.data_ptr(), y.data_ptr(), rows, n_out, k, base, nbytes, None,
                                   torch.cuda.current_stream().cuda_stream)
        assert st == 0, lib.memspec_op_last_error()
        x, w = x.double(), w.double()
        bad = ~((y.double() - x @ w.T).abs() <= 1e-4 * (x.abs() @ w.abs().T) + 1e-6)   # true for NaN
        assert not bad.any(), (rows, n_out, k, int(bad.sum()))


def test_linear_refuses_a_scratch_that_is_too_small():
    """The call is given what the scratch holds from its first 256-byte boundary on."""
    from paper_2608_10362_gb300 import MemSpecError, _lib, op_linear
    need = C.c_size_t()
    assert _lib.load().memspec_op_linear_scratch_bytes(32, 256, 64, C.byref(need)) == 0
    x = torch.ones(32, 64, dtype=torch.bfloat16, device="cuda")
    w = torch.ones(256, 64, dtype=torch.bfloat16, device="cuda")
    buf = torch.zeros(need.value + 512, dtype=torch.uint8, device="cuda")
    assert buf.data_ptr() % 256 == 0
    assert (op_linear(x, w, buf[:need.value]) == 64).all()
    assert (op_linear(x, w, buf[1:256 + need.value]) == 64).all()
    for small in (buf[:need.value - 1], buf[1:need.value + 255], buf[1:9]):
        with pytest.raises(MemSpecError):
            op_linear(x, w, small)


@pytest.mark.parametrize("n_out,k", [(12288, 4096), (4096, 11008), (32000, 4096)])
def test_linear_full_7b_shapes_sampled(n_out, k):
    from paper_2608_10362_gb300 import op_linear
    rows = 5
    x, w = _bf16_pair(2, rows, n_out, k)
    y = op_linear(torch.from_numpy(x).to(torch.bfloat16).cuda(),
                  torch.from_numpy(w).to(torch.bfloat16).cuda()).cpu().numpy()
    cols = np.unique(np.concatenate([np.random.default_rng(3).integers(0, n_out, 512),
                                     np.arange(n_out - 130, n_out), np.arange(0, 130)]))
    ref = x.astype(np.float64) @ w[cols].astype(np.float64).T
    bound = np.abs(x).astype(np.float64) @ np.abs(w[cols]).astype(np.float64).T
    assert np.all(np.abs(y[:, cols] - ref) <= 1e-4 * bound + 1e-6)


def _pack_reference(a, b=None):
    """Packed-tile bytes (as bf16 bit patterns) written out from the documented
    format: 128-row (pairs: 64 + 64) x 64-column tiles, row-major tiles in
    (row tile, k tile) order, 16-byte chunk c of row r stored at c ^ (r % 8)."""
    n, k = a.shape
    rows = 64 if b is not None else 128
    RT, KT = -(-n // rows), -(-k // 64)
    bits = lambda x: (np.ascontiguousarray(x, dtype=np.float32).view(np.uint32) >> 16).astype(np.uint16)
    out = np.zeros((RT, KT, 128, 64), dtype=np.uint16)
    for rt in range(RT):
        for kt in range(KT):
            tile = np.zeros((128, 64), dtype=np.uint16)
            for r in range(128):
                if b is not None:
                    src, row = (a, rt * 64 + r) if r < 64 else (b, rt * 64 + r - 64)
                else:
                    src, row = a, rt * 128 + r
                if row >= n:
                    continue
                cols = src[row, kt * 64:kt * 64 + 64]
                vals = np.zeros(64, dtype=np.uint16)
                vals[:len(cols)] = bits(cols)
                for c in range(8):
                    pos = c ^ (r % 8)
                    tile[r, pos * 8:pos * 8 + 8] = vals[c * 8:c * 8 + 8]
            out[rt, kt] = tile
    return out.reshape(-1)


@pytest.mark.parametrize("n,k,pair", [(300, 200, False), (130, 136, True), (128, 64, False),
                                      (256, 8, True)])
def test_pack_matrix_matches_documented_layout(n, k, pair):
    from paper_2608_10362_gb300 import pack_matrix
    rng = np.random.default_rng(n * 7 + k)
    a = bf16_round(rng.standard_normal((n, k), dtype=np.float32))
    b = bf16_round(rng.standard_normal((n, k), dtype=np.float32)) if pair else None
    ref = _pack_reference(a, b)
    dst = torch.full((ref.size * 2,), 0xAB, dtype=torch.uint8, device="cuda")   # non-zero fill
    ta = torch.from_numpy(a).to(torch.bfloat16).cuda()
    tb = torch.from_numpy(b).to(torch.bfloat16).cuda() if pair else None
    pack_matrix(ta, dst, tb)
    torch.cuda.synchronize()
    got = dst.cpu().numpy().view(np.uint16)
    assert np.array_equal(got, ref)


def test_calls_back_to_back_see_their_predecessors_output():
    """op_linear over rows of every kernel, each reading weights and activations that
    the work before it writes, its output drawn from by op_sample, and INT4 layers right
    after their packing: nothing waits on the host, one scratch.  The launches may start
    before their predecessors end; the outputs have to be those of the final inputs."""
    from paper_2608_10362_gb300 import int4_pack, op_linear, op_linear_int4, op_sample
    V, k, rounds = 5000, 3000, 3
    g = torch.Generator(device="cuda").manual_seed(12)
    normal = lambda *s: torch.randn(s, device="cuda", generator=g)
    all_rows = (5, 16, 17, 144, 160, 161, 256)
    ws = [(normal(V, k) * 0.02).to(torch.bfloat16) for _ in range(2)]
    xs = {r: [normal(r, k).to(torch.bfloat16) for _ in range(2)] for r in all_rows}
    u = {r: torch.rand(r, device="cuda", generator=g).clamp(1e-6, 1 - 1e-6) for r in all_rows}
    codes = [torch.randint(0, 256, (V, 2048 // 2), dtype=torch.uint8, device="cuda", generator=g) for _ in range(2)]
    scales = torch.full((V, 16), 0.005, dtype=torch.bfloat16, device="cuda")
    zeros = torch.full((V, 16), 8, dtype=torch.uint8, device="cuda")
    x4 = normal(5, 2048).to(torch.bfloat16)
    w = torch.empty_like(ws[0])
    x = {r: torch.empty_like(xs[r][0]) for r in all_rows}
    scratch = torch.zeros(64 << 20, dtype=torch.uint8, device="cuda")
    got = []
    for i in range(rounds):
        for r in all_rows:
            torch.add(ws[i % 2], 0, out=w)
            torch.add(xs[r][i % 2], 0, out=x[r])
            y = op_linear(x[r], w, scratch)
            t = op_sample(y, 0.9, u[r])
            got.append((r, i % 2, y, t, op_sample(y, 0.0)))
        y4 = op_linear_int4(x4, int4_pack(codes[i % 2], scales, zeros), V)
        got.append((0, i % 2, y4, op_sample(y4, 0.9, u[5]), op_sample(y4, 0.0)))
    torch.cuda.synchronize()
    for r, i, y, t, greedy in got:
        if r:
            a, b = xs[r][i].double(), ws[i].double()
            bound = 1e-4 * (a.abs() @ b.abs().T) + 1e-6
        else:   # sums of 128 terms x (128 + q), the zero point's (128 + 8) x beside them
            a, s = x4.double(), scales[0, 0].double()
            b = (torch.stack([codes[i] & 15, codes[i] >> 4], -1).view(V, -1).double() - 8) * s
            bound = 2.0 ** -24 * (128 * (256 + 15 + 8) * s * a.abs().sum(1, keepdim=True) + 8 * (a.abs() @ b.abs().T))
        assert ((y.double() - a @ b.T).abs() <= bound).all(), (r, i)
        assert torch.equal(greedy, y.argmax(1).int()) and torch.equal(t, op_sample(y, 0.9, u[r or 5])), (r, i)


@pytest.mark.parametrize("T", [0.0, 1.0, 0.8])
@pytest.mark.parametrize("vocab", [2048, 32000, 128256, 97])
def test_sampler_matches_inverse_cdf(T, vocab):
    from paper_2608_10362_gb300 import op_sample
    rows = 24
    z = gen_logits(11, rows, vocab, scale=1.3)
    z[3, :] = 0.0                        # all-equal row: argmax tie -> id 0
    z[4, vocab // 2] = 40.0              # one dominant id
    rng = np.random.default_rng(5)
    u = ((2 * (rng.integers(0, 1 << 23, rows)) + 1) * 2.0 ** -24).astype(np.float32)
    u[5], u[6] = 2.0 ** -24, 1 - 2.0 ** -24
    out = op_sample(torch.from_numpy(z).cuda(), T, torch.from_numpy(u).cuda()).cpu().numpy()
    flags = 0
    for r in range(rows):
        expect = draft_token(z[r].astype(np.float64), T, float(u[r]))
        if out[r] == expect:
            continue
        assert T > 0, (r, out[r], expect)
        q = softmax_t(z[r], T)
        c = np.cumsum(q)
        b = c[min(out[r], expect)]
        assert abs(u[r] - b) < 1e-5, (r, out[r], expect, u[r], b)
        flags += 1
    assert flags <= 1


@pytest.mark.parametrize("rows,vocab,offset", [
    (1, 1, 0), (3, 127, 1), (2, 2048, 3), (5, 2049, 0), (1, 8191, 2), (152, 8192, 0), (1, 16384, 0),
    (77, 16385, 0), (1, 32000, 0), (500, 8001, 1), (200, 32003, 1), (2, 65537, 0), (3, 131071, 0), (2, 131072, 3),
])
def test_sampler_slices(rows, vocab, offset):
    """Vocabularies at the edges of a 128-id tile, a CTA's slice and the largest
    cluster, rows whose first logit is not 16-byte aligned (offset floats past an
    aligned address, odd vocabularies), few and many rows: every drawn id is one of the
    row's, has weight, and its share of [0, 1) holds u up to fp32 rounding (bound 1e-5:
    the sums are of at most 131072 terms in a tree, relative error below 40 * 2^-24);
    greedy: the first largest."""
    from paper_2608_10362_gb300 import op_sample
    z = gen_logits(21, rows, vocab, scale=2.0)
    z[0, vocab - 1] = 12.0               # mass at the end of the last slice
    u = ((2 * np.random.default_rng(6).integers(0, 1 << 23, rows) + 1) * 2.0 ** -24).astype(np.float32)
    u[rows - 1] = 1 - 2.0 ** -24
    buf = torch.empty(rows * vocab + offset, dtype=torch.float32, device="cuda")
    zt = buf[offset:].view(rows, vocab)
    zt.copy_(torch.from_numpy(z))
    for T in (0.0, 0.9):
        out = op_sample(zt, T, torch.from_numpy(u).cuda()).cpu().numpy()
        assert ((0 <= out) & (out < vocab)).all(), (T, out)
        for r in range(rows):
            if T == 0:
                assert out[r] == int(np.argmax(z[r])), r
                continue
            q = softmax_t(z[r], T)
            c = np.cumsum(q)
            below, upto = c[out[r]] - q[out[r]], c[out[r]]
            assert q[out[r]] > 0 and below - 1e-5 <= u[r] <= upto + 1e-5, (r, out[r], u[r], below, upto)


@pytest.mark.parametrize("copies", [1, 40])
def test_sampler_degenerate_rows(copies):
    """Rows without a proper distribution: a NaN among the logits, +inf, every
    logit -inf but one, all equal; the draw is an id of the row (the first argmax
    where the weights have no finite sum).  Few rows (slices of one round) and many
    (slices of several)."""
    from paper_2608_10362_gb300 import op_sample
    V = 32000
    z = gen_logits(22, 5, V, scale=1.0)
    z[0, 17000] = np.nan
    z[1, 29000] = np.inf
    z[2, :] = -np.inf
    z[2, 31999] = -3.0
    z[3, :] = 0.0
    u = np.full(5 * copies, 0.5, dtype=np.float32)
    zt = torch.from_numpy(np.tile(z, (copies, 1))).cuda()
    out = op_sample(zt, 1.0, torch.from_numpy(u).cuda()).cpu().numpy().reshape(copies, 5)
    assert (out == out[0]).all()
    out = out[0]
    assert out[0] == int(np.nanargmax(z[0])) and out[1] == 29000 and out[2] == 31999
    assert abs(int(out[3]) - V // 2) <= 1
    g = op_sample(zt, 0.0).cpu().numpy().reshape(copies, 5)
    assert (g == g[0]).all()
    g = g[0]
    assert g[0] == int(np.nanargmax(z[0])) and g[1] == 29000 and g[2] == 31999 and g[3] == 0


@pytest.fixture(scope="module")
def tiny_engine():
    from paper_2608_10362_gb300 import Engine
    t, d = SHAPES["tiny_target"], SHAPES["tiny_draft"]
    eng = Engine(t, gen_weights(t, 0), max_batch=4, max_seq=512, max_k=8, max_drafts=2,
                 draft_shape_max=d, draft_budget_bytes=64 << 20, use_graphs=False)
    eng.register_draft(0, d, gen_weights(d, 1))
    eng.load_draft_async(0)
    eng.set_active_draft(0)
    yield eng
    eng.close()


@pytest.mark.parametrize("T", [1.0, 0.7, 0.0])
def test_acceptance_kernel_on_synthetic_logits(tiny_engine, T):
    """accept_commit on seeded logits: n and the final token equal the oracle's
    speculative-sampling decision with the same Philox uniforms."""
    from paper_2608_10362_gb300 import _lib
    eng = tiny_engine
    V, K, B = eng.vocab, 4, 4
    eng.set_batch(B)
    flags = 0
    n_seen = set()
    for trial in range(40):
        zt = gen_logits(100 + trial, B * (K + 1), V, 2.0).reshape(B, K + 1, V)
        zd = zt[:, :K] + gen_logits(200 + trial, B * K, V, 0.6 + 0.1 * (trial % 5)).reshape(B, K, V)
        x = np.zeros((B, eng.max_k), dtype=np.int32)
        for b in range(B):
            for j in range(K):
                x[b, j] = draft_token(zd[b, j], T, (j + 0.5) / K) if T > 0 else int(np.argmax(zt[b, j]) if (b + j + trial) % 3 else np.argmax(zd[b, j]))
        L0 = 50 + trial
        state = np.zeros((eng.max_batch, 4), dtype=np.int32)
        state[:, 0], state[:, 1], state[:, 2], state[:, 3] = L0, L0 - 1, trial, L0 - 1
        eng.write_buffer(_lib.BUF_TARGET_LOGITS, zt.astype(np.float32).ravel())
        eng.write_buffer(_lib.BUF_DRAFT_LOGITS, zd.astype(np.float32).ravel())
        eng.write_buffer(_lib.BUF_DRAFT_TOKENS, x[:B].ravel())
        eng.write_buffer(_lib.BUF_SEQ_STATE, state)
        eng.accept_commit(K, T, eng.results_host)
        assert eng.sync() == 0
        res = eng.results_host.numpy()[:B * (K + 2)].reshape(B, K + 2)
        dbg = eng.accept_debug(B, K)
        st = eng.seq_state()
        for b in range(B):
            # no request was prefilled: seeds are zero, so the uniforms are seed 0's
            u_d, u_a, u_f = step_uniforms(0, b, trial, K)
            ro = accept(zt[b].astype(np.float64), zd[b].astype(np.float64), x[b, :K], T, u_a, u_f)
            n = int(res[b, 0])
            y = int(res[b, n + 1])
            n_seen.add(n)
            if T > 0:
                np.testing.assert_allclose(dbg[b, :n], ro.p_of_x[:n], rtol=1e-4)
                np.testing.assert_allclose(dbg[b, K:K + n], ro.q_of_x[:n], rtol=1e-4)
            if n != ro.n_accepted:
                i = min(n, ro.n_accepted)
                assert T > 0 and abs(u_a[i] - ro.p_of_x[i] / ro.q_of_x[i]) < 1e-3, (trial, b, n, ro)
                flags += 1
                continue
            if y != ro.token:
                assert T > 0, (trial, b, y, ro.token)
                if n < K:
                    w = np.maximum(softmax_t(zt[b, n], T) - softmax_t(zd[b, n], T), 0)
                else:
                    w = softmax_t(zt[b, n], T)
                c = np.cumsum(w) / w.sum()
                assert abs(u_f - c[min(y, ro.token)]) < 1e-4, (trial, b, y, ro.token)
                flags += 1
            assert list(res[b, 1:n + 1]) == list(x[b, :n])
            assert st[b, 0] == L0 + n + 1 and st[b, 1] == L0 + n and st[b, 2] == trial + 1
            assert st[b, 3] == L0 + min(n, K - 1)
    assert flags <= 2
    assert len(n_seen) >= 3        # several accept lengths were exercised
