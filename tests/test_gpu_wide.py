"""Split tiles of wide token tiles, and query tiles cut from a K/V head's whole group, at the sizes
where their bookkeeping can go wrong, against the same sums in 64 bits; and windows of such tiles
through whole layers, with bf16 weights against the oracle, with 4-bit ones against 64 bits."""
import numpy as np
import pytest

import dllm_inputs as I
import oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2606_13740_gb300 as p
    p.lib()
    return p


def _bf16(g, *shape, sigma=1.0):
    return (torch.randn(*shape, generator=g, dtype=torch.float32) * sigma).to(torch.bfloat16).cuda()


# (M, N, K, grid): one tile of 31 parts; more parts than chunks; two parts (one finisher); three (two
# finishers, uneven chunks); two chunks; several token tiles; whole tiles beside split ones; a grid
# that cuts no tile; one part per k-block
@pytest.mark.parametrize("M,N,K,grid", [
    (128, 250, 18944, 0), (128, 64, 18944, 0), (1024, 251, 4096, 0), (12288, 256, 1024, 0), (256, 96, 640, 5),
    (384, 33, 1088, 0), (4096, 96, 4096, 0), (640, 515, 2048, 0), (24576, 65, 512, 0), (512, 200, 640, 4),
    (200, 129, 64, 0), (130, 40, 192, 0),
])
def test_wide_split_tiles(pkg, M, N, K, grid):
    g = torch.Generator().manual_seed(M + N + K)
    W, X = _bf16(g, M, K, sigma=0.05), _bf16(g, N, K)
    D = pkg.dllm_op_gemm(W, X, M, N, K, grid=grid)
    w, x = W.double(), X.double()
    # fp32 sums of exact products: rounding errors of random sign, a few 2^-24 sqrt(K) of the terms'
    # size, i.e. of the norms' product over sqrt(K) (1e-5 of that product is 160 x 2^-24)
    tol = 1e-5 * x.norm(dim=1)[:, None] * w.norm(dim=1)[None, :]
    assert bool(((D.double() - x @ w.T).abs() <= tol).all())
    assert torch.equal(D, pkg.dllm_op_gemm(W, X, M, N, K, grid=grid))


# Sizes (for s SMs) whose tiles run whole, 32 tokens and one CTA each: up to 15 k-blocks of 64 and at
# most one tile per SM, eight token tiles counted for up to 256 tokens; the last ones and the first
# past them.  small: which it is, seen by the number of CTAs.
@pytest.mark.parametrize("small,size", [
    (True, lambda s: (768, 33, 256)), (True, lambda s: (128, 1, 8)),
    (True, lambda s: (128 * (s // 8), 256, 960)), (False, lambda s: (128 * (s // 8) + 1, 256, 960)),
    (True, lambda s: (128 * (s // 8 - 1), 250, 960)), (False, lambda s: (128 * (s // 8 - 1), 250, 968)),
    (True, lambda s: (256, 32 * (s // 2), 688)), (False, lambda s: (256, 32 * (s // 2) + 1, 688)),
    (True, lambda s: (128, 32 * (s - 1), 64)), (True, lambda s: (130, 31, 960)), (False, lambda s: (130, 31, 968)),
])
def test_small_whole_tiles(pkg, small, size):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    M, N, K = size(sms)
    g = torch.Generator().manual_seed(M + N + K)
    W, X = _bf16(g, M, K, sigma=0.05), _bf16(g, N, K)
    D = pkg.dllm_op_gemm(W, X, M, N, K)
    w, x = W.double(), X.double()
    tol = 1e-5 * x.norm(dim=1)[:, None] * w.norm(dim=1)[None, :]  # as above
    assert bool(((D.double() - x @ w.T).abs() <= tol).all())
    mt, kb = (M + 127) // 128, (K + 63) // 64
    _, trace = pkg.dllm.dllm_op_gemm_trace(W, X, M, N, K, 1)
    assert (len(trace) == mt * ((N + 31) // 32)) == small
    if small:  # the sums are those of 32 rows alone, and of one k-block per CTA, bit for bit
        n = min(N, 32)
        first = pkg.dllm_op_gemm(W, X[:n].contiguous(), M, n, K)
        assert torch.equal(D[:n], first)
        if mt * kb < sms:
            assert torch.equal(first, pkg.dllm_op_gemm(W, X[:n].contiguous(), M, n, K, grid=mt * kb))


@pytest.mark.parametrize("V,N,d", [(1024, 251, 4096), (512, 96, 2048), (4096, 64, 512)])
def test_wide_head_split_tiles(pkg, V, N, d):
    g = torch.Generator().manual_seed(V + N)
    W, X = _bf16(g, V, d, sigma=0.02), _bf16(g, N, d)
    cur = torch.randint(0, V - 1, (N,), generator=g, dtype=torch.int32).cuda()
    x0, conf, tc, lg = pkg.dllm_op_lmhead(W, X, cur, V, N, d, V - 1, want_logits=True)
    ref = (X.double() @ W.double().T).cpu().numpy()
    assert np.abs(lg.cpu().numpy() - ref).max() <= 1e-4 * np.abs(ref).max()
    x0, conf, tc, cur = (t.cpu().numpy() for t in (x0, conf, tc, cur))
    for n in range(N):
        rx0, rconf, rtc, margin = O.decide(ref[n].astype(np.float32), V - 1, cur[n])
        assert margin <= 1e-3 or x0[n] == rx0
        assert abs(conf[n] - rconf) <= 1e-3 * rconf and abs(tc[n] - rtc) <= 1e-3 * rtc + 1e-12


# the group's rows end inside a tile, at its edge and one past it; one query head per K/V head; one
# K/V head; prefixes that leave some key splits empty
@pytest.mark.parametrize("B,T,H,Hkv,kv", [
    (1, 5, 28, 4, [1200]), (2, 32, 28, 4, [1024, 3]), (1, 64, 8, 4, [1500]), (1, 43, 6, 2, [1061]),
    (2, 100, 8, 1, [1300, 700]), (3, 96, 4, 4, [2000, 64, 1]), (1, 129, 4, 2, [1111]),
    # two, three, six and seven key splits
    (6, 20, 24, 24, [1100, 900, 64, 1, 1003, 500]), (3, 32, 32, 32, [1100, 64, 1]), (1, 64, 8, 8, [1030]),
    (1, 64, 8, 8, [1200]),
])
def test_group_query_tiles(pkg, B, T, H, Hkv, kv):
    g = torch.Generator().manual_seed(B * T + H)
    cap = max(kv) + T + 7
    q, k, v = _bf16(g, B, H, T, 128), _bf16(g, B, Hkv, cap, 128), _bf16(g, B, Hkv, cap, 128)
    out = pkg.dllm_op_attention(q, k, v, torch.tensor(kv, dtype=torch.int32).cuda(), B, T, H, 128, cap, max(kv), Hkv=Hkv)
    for b in range(B):
        n = kv[b] + T
        kk, vv = (t[b, :, :n].double().repeat_interleave(H // Hkv, 0) for t in (k, v))
        ref = torch.softmax(q[b].double() @ kk.transpose(1, 2) / 128 ** 0.5, -1) @ vv
        got = out.view(B, T, H, 128)[b].transpose(0, 1).double()
        assert (got - ref).norm() <= 1e-2 * ref.norm()  # bf16 probabilities and outputs
        assert (got - ref).abs().max() <= 0.05 * ref.abs().max()


def test_group_query_tiles_past_65535(pkg):
    """256 sequences of 256 query tiles each (one K/V head, 32 query heads, 1024 tokens): the first and
    the last sequence."""
    B, T, H = 256, 1024, 32
    g = torch.Generator(device="cuda").manual_seed(1)
    q, k, v = (torch.randn(*s, device="cuda", generator=g, dtype=torch.bfloat16)
               for s in ((B, H, T, 128), (B, 1, T, 128), (B, 1, T, 128)))
    out = pkg.dllm_op_attention(q, k, v, torch.zeros(B, dtype=torch.int32).cuda(), B, T, H, 128, T, 0, Hkv=1)
    for b in (0, B - 1):
        ref = torch.softmax(q[b].double() @ k[b].double().transpose(1, 2) / 128 ** 0.5, -1) @ v[b].double()
        got = out.view(B, T, H, 128)[b].transpose(0, 1).double()
        assert (got - ref).norm() <= 1e-2 * ref.norm()  # bf16 probabilities and outputs


@pytest.mark.parametrize("N", [32, 40])
def test_head_argmax_ties(pkg, N):
    """Equal largest logits in one warp's rows, in two quarters, in two tiles and beside the mask id:
    the lowest id wins; conf is exact (the tied logits are 0 or powers of two apart)."""
    V, d, mask = 384, 64, 5
    W = torch.zeros(V, d, dtype=torch.bfloat16, device="cuda")
    X = torch.zeros(N, d, dtype=torch.bfloat16, device="cuda")
    for k, ids in enumerate([(3, 9), (40, 70), (100, 300), (mask, 7, 8), (383,), (127, 128)]):
        W[list(ids), k] = 16.0
    first = [3, 40, 100, 7, 383, 127, 0]  # the last kind: every logit 0
    ties = [2, 2, 2, 2, 1, 2, V - 1]
    kind = [n % 7 for n in range(N)]
    for n, k in enumerate(kind):
        if k < 6:
            X[n, k] = 1.0
    cur = torch.zeros(N, dtype=torch.int32, device="cuda")
    x0, conf, _, _ = pkg.dllm_op_lmhead(W, X, cur, V, N, d, mask)
    rest = np.exp(-16.0)
    for n, k in enumerate(kind):
        assert int(x0[n]) == first[k]
        p = 1 / ties[k] if k == 6 else 1 / (ties[k] + (V - 1 - ties[k]) * rest)
        assert abs(float(conf[n]) - p) <= 1e-5 * p  # a sum of at most 384 exponentials in fp32


# One layer of LLaDA-8B's width under a small vocabulary
SHAPE = dict(n_layers=1, d_model=4096, n_heads=32, head_dim=128, ffn=12288, vocab=1024, mask_id=1023,
             rope_base=500000.0)


def _weights(ctx):
    """The context's embedding, projections and head in 64 bits."""
    w = {i: ctx.dllm_get_weight(0, i) for i in range(7)} | {"emb": ctx.dllm_get_weight(-1, 1), "head": ctx.dllm_get_weight(-1, 2)}
    return {k: torch.from_numpy(v.view(np.int16)).cuda().view(torch.bfloat16).double() for k, v in w.items()}


def _one_layer(w, tok, pk, pv, r=lambda t: t):
    """Logits of the window `tok` after the prefix keys and values pk, pv [P][H][hd] through one layer and the
    head, in 64 bits; r is applied where the kernels round to bf16."""
    H, hd, T, P = SHAPE["n_heads"], SHAPE["head_dim"], len(tok), pk.shape[0]
    ang = torch.arange(P, P + T, device="cuda").double()[:, None] * SHAPE["rope_base"] ** (
        -torch.arange(0, hd, 2, device="cuda").double() / hd)[None, :]
    cs, sn = ang.cos()[:, None], ang.sin()[:, None]

    def rms(x):
        return (x.square().mean(-1, keepdim=True) + 1e-5).rsqrt()

    def rope(x):
        a, b = x[..., :hd // 2], x[..., hd // 2:]
        return torch.cat([a * cs - b * sn, b * cs + a * sn], -1)

    x = w["emb"][tok]
    q, k, v = ((x @ w[i].T * rms(x)).view(T, H, hd) for i in range(3))
    q, k, v = r(rope(q)), torch.cat([pk, r(rope(k))]), torch.cat([pv, r(v)])
    p = torch.softmax(torch.einsum("thd,nhd->htn", q, k) / hd ** 0.5, -1)
    x = x + r(torch.einsum("htn,nhd->thd", r(p), v).reshape(T, H * hd)) @ w[3].T
    g, u = (r(x) @ w[i].T * rms(x) for i in (4, 5))
    x = x + r(torch.nn.functional.silu(g) * u) @ w[6].T
    return r(x) @ w["head"].T * rms(x)


@pytest.fixture(scope="module")
def q4_weights(pkg):
    ctx = pkg.Context(pkg.Config(weight_bits=4, **SHAPE))
    yield _weights(ctx)
    ctx.close()


# 4-bit weights: the expanded tiles in tensor memory with 6 and 4 stages, then in shared memory; last
# chunks of one token and whole ones
@pytest.mark.parametrize("T", [33, 64, 65, 128, 129])
def test_q4_wide_windows(pkg, q4_weights, T):
    P = 70
    ctx = pkg.Context(pkg.Config(weight_bits=4, max_ctx=P + T, max_window=T, block_len=T, **SHAPE))
    ctx.dllm_set_prefix_kv_random(pkg.Sched(), 1, P, T, 7)
    ctx.dllm_begin_block()
    tok = I.uniform_prompt(P + T, 1024, 1023, seed=T)[None]
    st = np.full((1, P + T), pkg.COMMITTED, np.uint8)
    st[0, :P] = pkg.FIXED
    tok[0, P + T // 2], st[0, P + T // 2] = 1023, pkg.MASKED
    ctx.dllm_set_state(tok, st)
    ctx.dllm_set_debug(1)
    ctx.dllm_denoise_step()
    got = torch.as_tensor(ctx.dllm_get_step_debug(logits=True)["logits"][0]).double().cuda()
    pk, pv = (torch.as_tensor(ctx.dllm_get_kv(0, i, 0, 0, P)).double().cuda().view(P, 32, 128) for i in (0, 1))
    ctx.close()
    win = torch.as_tensor(tok[0, P:]).long().cuda()
    ref = _one_layer(q4_weights, win, pk, pv)

    # Every row within 5 times what bf16 roundings do to it: the largest of 16 draws of errors of
    # random sign and up to bf16's largest relative size, 2^-9, at every place where the kernels
    # round.  The 4-bit draws' mean is not zero, so a row's state lies along one direction with the
    # sign of a sum, and in a row whose sum is close to 0 any rounding grows (to 30 %); the others,
    # a last chunk's last row among them, must stay within a thousandth or so.
    def off(z):
        return (z - ref).norm(dim=-1) / ref.norm(dim=-1)

    gen = torch.Generator(device="cuda").manual_seed(T)

    def rounding(t):
        return t * (1 + 2.0 ** -9 * (2 * torch.rand(t.shape, device="cuda", dtype=torch.float64, generator=gen) - 1))

    spread = torch.stack([off(_one_layer(q4_weights, win, pk, pv, rounding)) for _ in range(16)]).amax(0)
    assert bool((off(got) <= 5 * spread).all())
    assert float(spread.median()) <= 1e-3 and float(spread[-1]) <= 1e-2


# Windows and lookahead windows of several 32-token chunks through two layers of LLaDA-8B's width,
# without and with refresh rows (chunks of window rows, of refresh rows and of both): block length,
# prompt, tokens to generate, schedule
@pytest.fixture(scope="module")
def wide_model():
    return O.Model(O.OracleConfig(**(SHAPE | {"n_layers": 2})))


@pytest.mark.parametrize("block,P,gen,kw", [
    (33, 70, 33, {}), (129, 20, 129, {}), (251, 12, 251, {}),
    (32, 70, 96, dict(spec_blocks=2, spec_trigger=32)),
    (33, 40, 66, dict(scr_rows=8, theta_stable=2.0)), (96, 40, 192, dict(scr_rows=32, theta_stable=2.0)),
])
def test_wide_windows_teacher_forced(pkg, wide_model, block, P, gen, kw):
    from test_gpu_step import _run_teacher_forced
    kw = dict(steps_per_block=1, **kw)
    # n bf16 roundings of random sign, 2^-9 / sqrt(3) of a value each: three times what they sum to.
    # A layer has eight (q, k, v, probabilities, attention output, x, h, x), keys and values one more.
    def bound(n):
        return 3 * (n / 3) ** 0.5 * 2.0 ** -9

    def rows_off(a, b):
        return float((np.linalg.norm(a - b, axis=-1) / np.linalg.norm(b, axis=-1)).max())

    seen = {"T": set(), "rows": 0}

    def check(sess, ctx, oo, go, before, o_after, g_after):
        got, ref = ctx.dllm_get_step_debug(logits=True)["logits"][0], sess.decisions(logits=True)["logits"]
        assert rows_off(got, ref) <= bound(16)
        seen["T"].add(sess.window()["T"])
        if kw.get("scr_rows"):
            od, gd = sess.scr_decisions(), ctx.dllm_get_scr_debug()
            n = len(od["pos"])
            assert np.array_equal(gd["pos"][:n], od["pos"]) and (gd["pos"][n:] == -1).all()
            assert np.allclose(gd["conf"][:n], od["conf"], rtol=0.05)
            assert np.allclose(gd["tokconf"][:n], od["tokconf"], rtol=0.05)
            assert go["n_refreshed"] == oo["n_refreshed"]
            seen["rows"] += n
        for layer in (0, 1):  # every cached row, refreshed ones included
            for which in (0, 1):
                ref = sess.prefix_kv(layer, which)
                got = ctx.dllm_get_kv(layer, which, 0, 0, ref.shape[0])
                assert rows_off(got, ref) <= bound(8 * layer + 1)

    ctx = pkg.Context(pkg.Config(max_ctx=P + gen, max_window=max(P, 3 * block if "spec_blocks" in kw else block + 32),
                                 block_len=block, **(SHAPE | {"n_layers": 2})))
    _run_teacher_forced(wide_model, O.OracleSched(block_len=block, **kw), pkg.Sched(**kw),
                        I.uniform_prompt(P, 1024, 1023, seed=block), gen, ctx, check)
    ctx.close()
    assert max(seen["T"]) == (96 if block == 32 else block) and (seen["rows"] > 0) == ("scr_rows" in kw)
