"""Split tiles of wide token tiles, and query tiles cut from a K/V head's whole group, at the sizes
where their bookkeeping can go wrong, against the same sums in 64 bits."""
import numpy as np
import pytest

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


# the last sizes whose tiles run whole, 32 tokens and one CTA each (up to 960 columns deep, at most
# one tile per SM), and the first past them
@pytest.mark.parametrize("M,N,K", [
    (768, 33, 256), (128, 1, 8), (2432, 256, 960), (2433, 256, 960), (2432, 250, 968), (256, 2432, 688),
    (256, 2433, 688), (128, 4096, 64), (130, 31, 960), (130, 31, 968),
])
def test_small_whole_tiles(pkg, M, N, K):
    g = torch.Generator().manual_seed(M + N + K)
    W, X = _bf16(g, M, K, sigma=0.05), _bf16(g, N, K)
    D = pkg.dllm_op_gemm(W, X, M, N, K)
    w, x = W.double(), X.double()
    tol = 1e-5 * x.norm(dim=1)[:, None] * w.norm(dim=1)[None, :]  # as above
    assert bool(((D.double() - x @ w.T).abs() <= tol).all())


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


# 4-bit weights: the expanded tiles in tensor memory with 5 and 4 stages, then in shared memory
@pytest.mark.parametrize("T", [33, 64, 65, 128, 129])
def test_q4_wide_windows(pkg, T):
    from perf import cases
    case = dict(name="", kind="step", shape="llada", layers=1, B=1, P=70, T=T, masked=T // 2, bits=4, cache=True,
                vocab=1024)
    got = torch.as_tensor(cases.run(cases.prepare(case, 7))["logits"]).double().cuda()
    ref = cases.exact(case, 7)["logits"]
    assert got.shape == ref.shape
    # A layer and the head round to bf16 (2^-9) eight times in a row (embedding, q/k/v, probabilities,
    # attention output, x, h, x; the weights are exact): sqrt(8) 2^-9 = 5.5e-3 where the errors' signs
    # are random.  By the median row: the 4-bit draws' mean is not zero, so a row's state lies along
    # one direction with the sign of a sum, and a row whose sum is close to 0 amplifies any rounding.
    err = ((got - ref).norm(dim=-1) / ref.norm(dim=-1)).flatten()
    assert err.median() <= 5.5e-3
