"""What is measured: the work a user of this library has it do, through its public entry points.

Most of it is the denoising step of a context (`dllm_denoise_step`), the library's main path, over
the windows, batches, prefixes, model widths and options it is used with; then the start of a
request (`dllm_prefill`), and the single-kernel entry points: a projection, attention, the LM head.
Models keep the real widths (LLaDA-8B, Dream-7B's grouped-query shape, the tiny model of the
tests) with fewer layers: every layer runs the same kernels, and rounding differences stay
comparable.  Two of the steps have the real vocabulary; the others are blocks of layers, under a
vocabulary of 1024, so that their logits say what the layers computed and cost little to read
(the LM head has a case of its own).

A step returns its logits and counts.  Argmax ids are left out: among random-init logits the
largest two are often closer than one rounding.

Weights come from the library's own seeded draws; `exact` draws the same weights again in plain
torch and runs the model in 64 bits.
"""
import ctypes
import math

import numpy as np
import torch

from paper_2606_13740_gb300 import COMMITTED, FIXED, MASKED, Config, Context, Sched
from paper_2606_13740_gb300 import dllm

# widths of this repository's configurations and tests
SHAPES = {
    "tiny": dict(d_model=256, n_heads=4, head_dim=64, ffn=688, rope_base=10000.0, n_kv_heads=0),
    "llada": dict(d_model=4096, n_heads=32, head_dim=128, ffn=12288, rope_base=500000.0, n_kv_heads=0),
    "dream": dict(d_model=3584, n_heads=28, head_dim=128, ffn=18944, rope_base=1000000.0, n_kv_heads=4),
}
FULL_VOCAB = {"tiny": 1024, "llada": 126464, "dream": 152064}
WEIGHT_SEED = 0x11ADA8B
EPS = 1e-5


def listed():
    return [
        # The smallest step there is: the two-layer model of the tests, where launches and the host
        # count and nothing else.
        _step("tiny_step_t32", "tiny", layers=2, P=64, T=32, masked=24),
        # The benchmark's step: batch 1, one 32-token block after a 512-token prefix (weights stream).
        _step("step_b1_t32", "llada", layers=8, P=512, T=32, masked=24, vocab=126464),
        # The same with weights in the 4-bit block format, the form the paper runs.
        _step("step_b1_t32_q4", "llada", layers=8, P=512, T=32, masked=24, vocab=126464, bits=4),
        # Multi-block speculation: the block and two lookahead blocks in one window.
        _step("step_b1_t96", "llada", layers=8, P=1024, T=96, masked=72),
        # Vanilla decoding without the prefix cache: the whole 251-position sequence every step.
        _step("step_vanilla_t251", "llada", layers=8, P=123, T=128, masked=96, cache=False),
        # Batched serving: 16 sequences, 4096-token prefixes, 64 window tokens each.
        _step("step_b16_t64", "llada", layers=4, B=16, P=4096, T=64, masked=32),
        # A small batch of the grouped-query model with ragged sizes.
        _step("step_gqa_b5_t32", "dream", layers=4, B=5, P=1501, T=32, masked=20),
        # The start of a request: a 2000-token prompt through the layers, then the first step.
        _prefill("prefill_t2000", "llada", layers=4, B=1, P=2000, T=32),
        # A projection of the batched step by itself: gate/up over 1024 tokens.
        _gemm("gemm_gateup_n1024", M=24576, N=1024, K=4096),
        # Attention of a prompt over itself (the prefill's attention).
        _attn("attn_prompt_t2048", B=1, T=2048, H=32, Hkv=32, hd=128, P=0),
        # Attention of decoding windows over long, unequal prefixes, grouped-query.
        _attn("attn_gqa_b6_t96", B=6, T=96, H=28, Hkv=4, hd=128, P=3001),
        # The LM head with its decision over a small batch of windows.
        _head("lmhead_n96", V=126464, N=96, d=4096),
    ]


def _step(name, shape, layers, P, T, masked, B=1, bits=16, cache=True, vocab=1024):
    return dict(name=name, kind="step", shape=shape, layers=layers, B=B, P=P, T=T, masked=masked, bits=bits,
                cache=cache, vocab=vocab)


def _prefill(name, shape, layers, B, P, T, bits=16, vocab=1024):
    return dict(name=name, kind="prefill", shape=shape, layers=layers, B=B, P=P, T=T, bits=bits, vocab=vocab)


def _gemm(name, M, N, K):
    return dict(name=name, kind="gemm", M=M, N=N, K=K)


def _attn(name, B, T, H, Hkv, hd, P):
    return dict(name=name, kind="attn", B=B, T=T, H=H, Hkv=Hkv, hd=hd, P=P)


def _head(name, V, N, d):
    return dict(name=name, kind="head", V=V, N=N, d=d)


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _seconds(case):
    w = work(case)
    return w["bytes"] / 6.8e12 + w["flops"] / 1.9e15


def draw(rng):
    most = max(_seconds(c) for c in listed())
    while True:
        kind = rng.choice(["step", "step", "step", "step", "prefill", "prefill", "gemm", "attn", "attn", "head"])
        if kind in ("step", "prefill"):
            shape = rng.choice(["tiny", "llada", "llada", "dream"])
            layers = 2 if shape == "tiny" else rng.randint(2, 6)
        if kind == "step":
            # 4-bit weights: one sequence and its lookahead (their codes' mean is not zero, so every
            # row's hidden state grows along one direction, with the sign of a sum; in many rows
            # there is one whose sum is close to 0 and whose sign a rounding decides)
            bits = rng.choice([16, 16, 16, 4])
            T = min(256, _log(rng, 4, 300)) if bits == 16 else _log(rng, 4, 96)
            B = max(1, min(_log(rng, 1, 16), 1024 // T)) if bits == 16 else 1
            cache = bits == 4 or rng.random() < 0.85
            # the real vocabulary where the logits are few enough to read beside the step
            full = shape != "tiny" and B * T <= 64 and cache and rng.random() < 0.5
            c = _step("", shape, layers, _log(rng, 16, 4096) if cache else _log(rng, 16, 256), T,
                      rng.randint((T + 1) // 2, T), B=B if cache else 1, bits=bits, cache=cache,
                      vocab=FULL_VOCAB[shape] if full else 1024)
        elif kind == "prefill":
            P = _log(rng, 64, 2048)
            c = _prefill("", shape, layers, rng.randint(1, max(1, min(4, 2048 // P))), P, 32)
        elif kind == "gemm":
            M, K = rng.choice([(4096, 4096), (12288, 4096), (24576, 4096), (4096, 12288), (37888, 3584), (3584, 18944),
                               (768, 256), (256, 688)])
            c = _gemm("", M, _log(rng, 1, 2048), K)
        elif kind == "attn":
            H, Hkv, hd = rng.choice([(32, 32, 128), (28, 4, 128), (4, 4, 64), (16, 4, 64)])
            if rng.random() < 0.4:  # a prompt over itself
                c = _attn("", rng.randint(1, 4), _log(rng, 64, 2048), H, Hkv, hd, 0)
            else:  # windows over a prefix
                c = _attn("", _log(rng, 1, 16), _log(rng, 4, 256), H, Hkv, hd, _log(rng, 16, 4096))
        else:
            V, d = rng.choice([(126464, 4096), (152064, 3584), (1024, 256)])
            c = _head("", V, _log(rng, 1, 512), d)
        del c["name"]
        if _seconds(c) <= most:
            return c


# ------------------------------------------------------------------------------------ inputs
def _rng(seed, salt):
    return np.random.default_rng([int(seed), salt])


def _config(case):
    s = SHAPES[case["shape"]]
    n_pos = case["P"] + case["T"]
    window = case["T"] if case.get("cache", True) else n_pos
    if case["kind"] == "prefill":
        window = max(case["P"], case["T"])
    return Config(n_layers=case["layers"], max_batch=case["B"], max_ctx=n_pos, max_window=window,
                  block_len=case["T"], rms_eps=EPS, weight_seed=WEIGHT_SEED, weight_bits=case["bits"],
                  vocab=case["vocab"], mask_id=case["vocab"] - 1, **s)


def _ids(case, seed):
    """Prompt (or vanilla prefix) ids and the window's ids and states, [B][P + T]: Zipf(1.1) ids, `masked`
    of the window's positions masked, the others visible."""
    B, P, T, V = case["B"], case["P"], case["T"], case["vocab"]
    g = _rng(seed, 1)
    cdf = np.cumsum(np.arange(1, V, dtype=np.float64) ** -1.1)
    tok = np.minimum(np.searchsorted(cdf / cdf[-1], g.random((B, P + T))), V - 2).astype(np.int32)
    st = np.full((B, P + T), FIXED, np.uint8)
    st[:, P:] = COMMITTED
    for b in range(B):
        m = P + g.permutation(T)[:case.get("masked", T)]
        tok[b, m], st[b, m] = V - 1, MASKED
    return tok, st


def _sched(case):
    return Sched(steps_per_block=16, use_prefix_cache=1 if case.get("cache", True) else 0)


def prepare(case, seed):
    if case["kind"] == "step":
        # a context inside a block: the prefix cached, some of the window visible, the rest masked
        ctx, sched = Context(_config(case)), _sched(case)
        tok, st = _ids(case, seed)
        B, P, T = case["B"], case["P"], case["T"]
        if case["cache"]:
            ctx.dllm_set_prefix_kv_random(sched, B, P, T, int(seed))
            tok[:, :P] = 0
        else:
            ctx.dllm_prefill(sched, tok[:, :P], T)
        ctx.dllm_begin_block()
        ctx.dllm_set_state(tok, st)
        ctx.dllm_set_debug(1)  # keep the logits
        return {"kind": "step", "ctx": ctx}
    if case["kind"] == "prefill":
        tok, _ = _ids(case, seed)
        ctx = Context(_config(case))
        ctx.dllm_set_debug(1)  # keep the logits
        return {"kind": "prefill", "ctx": ctx, "sched": _sched(case),
                "prompt": np.ascontiguousarray(tok[:, :case["P"]]), "T": case["T"]}
    t = _op_inputs(case, seed)
    return {"kind": case["kind"], "case": dict(case), **t}


def _op_inputs(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))

    def normal(*shape, sigma=1.0):
        return torch.randn(*shape, device="cuda", generator=g, dtype=torch.float32).mul_(sigma).to(torch.bfloat16)

    if case["kind"] == "gemm":  # weights at the models' initialisation, unit-variance activations
        return {"W": normal(case["M"], case["K"], sigma=0.02), "X": normal(case["N"], case["K"])}
    if case["kind"] == "attn":  # unequal prefixes, none longer than P
        B, T, hd, P = case["B"], case["T"], case["hd"], case["P"]
        q = normal(B, case["H"], T, hd)
        k, v = normal(B, case["Hkv"], P + T, hd), normal(B, case["Hkv"], P + T, hd)
        kv = torch.randint(P // 2, P + 1, (B,), device="cuda", generator=g, dtype=torch.int32)
        kv[0] = P
        return {"q": q, "k": k, "v": v, "kv": kv}
    V, N, d = case["V"], case["N"], case["d"]
    return {"W": normal(V, d, sigma=0.02), "X": normal(N, d),
            "cur": torch.randint(0, V - 1, (N,), device="cuda", generator=g, dtype=torch.int32)}


def run(state):
    if state["kind"] in ("step", "prefill"):
        ctx = state["ctx"]
        if state["kind"] == "step":
            ctx.dllm_rewind_block()  # the block's state as prepared
        else:
            ctx.dllm_prefill(state["sched"], state["prompt"], state["T"])
            ctx.dllm_begin_block()
        o = ctx.dllm_denoise_step()
        return {"logits": ctx.dllm_get_step_debug(logits=True)["logits"], "committed": o["n_committed"],
                "masked": o["masked_after"]}
    c = state["case"]
    if state["kind"] == "gemm":
        return dllm.dllm_op_gemm(state["W"], state["X"], c["M"], c["N"], c["K"])
    if state["kind"] == "attn":
        return dllm.dllm_op_attention(state["q"], state["k"], state["v"], state["kv"], c["B"], c["T"], c["H"], c["hd"],
                                      c["P"] + c["T"], c["P"], Hkv=c["Hkv"])
    _, conf, tokconf, _ = dllm.dllm_op_lmhead(state["W"], state["X"], state["cur"], c["V"], c["N"], c["d"], c["V"] - 1)
    return {"conf": conf, "tokconf": tokconf}


# ------------------------------------------------------------------------------------ work
def _dims(shape):
    s = SHAPES[shape]
    qd = s["n_heads"] * s["head_dim"]
    kvd = (s["n_kv_heads"] or s["n_heads"]) * s["head_dim"]
    return s["d_model"], qd, kvd, s["ffn"]


def _forward_work(case, T, keys, head):
    """Layers over T rows of each sequence attending to `keys` keys, and the LM head with its logits."""
    d, qd, kvd, F = _dims(case["shape"])
    B, layers, V = case["B"], case["layers"], case["vocab"] if head else 0
    params = layers * (d * (qd + 2 * kvd) + qd * d + 3 * d * F) + V * d
    weight = 2.0 if case["bits"] == 16 else 0.5 + 2.0 / 32
    cache = layers * B * 2 * keys * kvd * 2
    return (params * weight + cache + B * T * (2.0 * d + 4.0 * V),
            2.0 * B * T * params + layers * 4.0 * B * T * keys * qd)


def work(case):
    k = case["kind"]
    if k == "step":
        keys = case["P"] + case["T"]
        b, f = _forward_work(case, case["T"] if case["cache"] else keys, keys, True)
        return {"bytes": b, "flops": f}
    if k == "prefill":
        b0, f0 = _forward_work(case, case["P"], case["P"], False)
        b1, f1 = _forward_work(case, case["T"], case["P"] + case["T"], True)
        return {"bytes": b0 + b1, "flops": f0 + f1}
    if k == "gemm":
        M, N, K = case["M"], case["N"], case["K"]
        return {"bytes": 2.0 * (M * K + N * K) + 4.0 * M * N, "flops": 2.0 * M * N * K}
    if k == "attn":
        B, T, H, Hkv, hd, P = (case[x] for x in ("B", "T", "H", "Hkv", "hd", "P"))
        keys = 0.75 * P + T  # the prefixes lie between P / 2 and P
        return {"bytes": 2.0 * (2 * B * H * T * hd + 2 * B * Hkv * keys * hd), "flops": 4.0 * B * H * T * keys * hd}
    V, N, d = case["V"], case["N"], case["d"]
    return {"bytes": 2.0 * (V * d + N * d) + 8.0 * N, "flops": 2.0 * V * N * d}


def tolerance(case):
    # about four times the distance from 64 bits (see exact), which is rounding: fp32 sums for a
    # projection (4.2e-6) and the head (1.9e-5), bf16 outputs and probabilities for attention
    # (2.3e-3), bf16 operands in every layer for models (3.6e-3 for the tiny one, 7.8e-3 to 1.3e-2
    # for 2 to 8 real layers; with 4-bit weights, whose logits one direction dominates, 3e-4)
    k = case["kind"]
    if k == "gemm":
        return {"rel": 2e-5, "max": 1e-4}
    if k == "head":
        return {"rel": 8e-5, "max": 2e-4}
    if k == "attn":
        return {"rel": 1e-2, "max": 5e-2}
    if case["shape"] == "tiny":
        return {"rel": 1.5e-2, "max": 0.1}
    return {"rel": 0.03, "max": 0.3} if case["bits"] == 16 else {"rel": 3e-3, "max": 0.1}


# ------------------------------------------------------------------------------------ 64 bits
def _i64(x):
    return ctypes.c_int64(x & 0xFFFFFFFFFFFFFFFF).value


def _shr(z, n):
    return (z >> n) & ((1 << (64 - n)) - 1)


def _mix(z):
    """SplitMix64's output function (int64 arithmetic wraps as uint64 does)."""
    z = (z ^ _shr(z, 30)) * _i64(0xBF58476D1CE4E5B9)
    z = (z ^ _shr(z, 27)) * _i64(0x94D049BB133111EB)
    return z ^ _shr(z, 31)


def _key(seed, tid):
    """Output `tid` of the stream `seed`."""
    m = 0xFFFFFFFFFFFFFFFF
    z = (seed + (tid + 1) * 0x9E3779B97F4A7C15) & m
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & m
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & m
    return z ^ (z >> 31)


def _outputs(key, n):
    """Outputs n (an int64 tensor) of the stream `key`."""
    return _mix((n + 1) * _i64(0x9E3779B97F4A7C15) + _i64(key))


def _normals(seed, tid, first, count, sigma):
    """Elements first .. first + count - 1 of a seeded tensor: Irwin-Hall(4) draws, rounded to bf16."""
    key, out = _key(seed, tid), torch.empty(count, dtype=torch.bfloat16, device="cuda")
    for a in range(0, count, 1 << 24):
        b = min(count, a + (1 << 24))
        i = torch.arange(first + a, first + b, dtype=torch.int64, device="cuda") * 4
        s = torch.zeros_like(i)
        for j in range(4):
            s += _shr(_outputs(key, i + j), 32)
        out[a:b] = ((s.double() - 8589934592.0) * float.fromhex("0x1.bb67ae8584caap-32") * sigma).float().bfloat16()
    return out


def _matrix(case, tid, rows, cols, bits=None):
    """The seeded weight matrix `tid` in 64 bits (bf16, or the 4-bit block format's values)."""
    if (bits or case["bits"]) == 16:
        return _normals(WEIGHT_SEED, tid, 0, rows * cols, 0.02).view(rows, cols).double()
    nblk = (cols + 31) // 32
    out = torch.empty(rows, cols, dtype=torch.float64, device="cuda")
    kq, ks = _key(WEIGHT_SEED, (3 << 40) + tid), _key(WEIGHT_SEED, (4 << 40) + tid)
    col = torch.arange(cols, device="cuda")
    for a in range(0, rows, 2048):
        r = torch.arange(a, min(rows, a + 2048), dtype=torch.int64, device="cuda")[:, None]
        q = _shr(_outputs(kq, r * cols + col[None, :]), 60)
        m = _shr(_outputs(ks, r * nblk + torch.arange(nblk, device="cuda")[None, :]), 59)
        d = (1 + m.double() / 128) / 256
        out[a:a + 2048] = (d[:, col // 32] * (q - 8).double()).float().bfloat16().double()
    return out


def _rms(x):
    return x * torch.rsqrt(x.square().mean(-1, keepdim=True) + EPS)


def _rope(x, pos, base):
    """Rotate-half RoPE of [B][heads][T][hd] at positions pos [T]."""
    hd = x.shape[-1]
    th = base ** (-2.0 * torch.arange(hd // 2, dtype=torch.float64, device="cuda") / hd)
    a = pos.double()[:, None] * th[None, :]
    c, s = a.cos(), a.sin()
    u, v = x[..., :hd // 2], x[..., hd // 2:]
    return torch.cat([u * c - v * s, u * s + v * c], -1)


def _attention(q, k, v):
    """[H][T][hd] over [Hkv][n][hd]."""
    g = q.shape[0] // k.shape[0]
    out = torch.empty_like(q)
    for h in range(q.shape[0]):
        p = torch.softmax(q[h] @ k[h // g].T / math.sqrt(q.shape[-1]), -1)
        out[h] = p @ v[h // g]
    return out


def _layers(case, x, pos, prefix):
    """x [B][T][d] through the layers; prefix(l) gives each layer's earlier keys and values (lists over the
    sequences of [Hkv][P][hd], or None). Returns x and every layer's own keys and values."""
    s = SHAPES[case["shape"]]
    d, qd, kvd, F = _dims(case["shape"])
    hd, B, T = s["head_dim"], x.shape[0], x.shape[1]

    def heads(y):
        return y.view(B, T, -1, hd).transpose(1, 2)

    own = []
    for l in range(case["layers"]):
        t = 16 + 8 * l
        n = _rms(x)
        q = _rope(heads(n @ _matrix(case, t, qd, d).T), pos, s["rope_base"])
        k = _rope(heads(n @ _matrix(case, t + 1, kvd, d).T), pos, s["rope_base"])
        v = heads(n @ _matrix(case, t + 2, kvd, d).T)
        own.append((k, v))
        a = torch.empty(B, T, qd, dtype=torch.float64, device="cuda")
        for b in range(B):
            pk, pv = prefix(l, b) if prefix else (k[b, :, :0], v[b, :, :0])
            o = _attention(q[b], torch.cat([pk, k[b]], 1), torch.cat([pv, v[b]], 1))
            a[b] = o.transpose(0, 1).reshape(T, qd)
        x = x + a @ _matrix(case, t + 3, d, qd).T
        n = _rms(x)
        h = torch.nn.functional.silu(n @ _matrix(case, t + 4, F, d).T) * (n @ _matrix(case, t + 5, F, d).T)
        x = x + h @ _matrix(case, t + 6, d, F).T
    return x, own


def _decide(z, cur, mask_id):
    """conf, tokconf of logits z [N][V] (the mask id excluded)."""
    m = z.clone()
    m[:, mask_id] = -math.inf
    p = torch.softmax(m, -1)
    own = p.gather(1, cur.long()[:, None])[:, 0]
    return p.max(-1).values, torch.where(cur == mask_id, torch.zeros_like(own), own)


def _exact_model(case, seed):
    d, qd, kvd, F = _dims(case["shape"])
    hd = SHAPES[case["shape"]]["head_dim"]
    B, P, T, V, Hkv, L = case["B"], case["P"], case["T"], case["vocab"], kvd // hd, case["layers"]
    tok, _ = _ids(case, seed)
    tok = torch.from_numpy(tok).cuda().long()
    emb = _normals(WEIGHT_SEED, 1, 0, V * d, 0.02).view(V, d)
    if case["kind"] == "prefill":
        tok[:, P:] = V - 1
        _, kv = _layers(case, emb[tok[:, :P]].double(), torch.arange(P, device="cuda"), None)

        def prefix(l, b):
            return kv[l][0][b], kv[l][1][b]
    elif case["cache"]:
        def prefix(l, b):
            return [_normals(int(seed), (1 << 32) + (b * L + l) * 2 + w, 0, P * kvd, 1.0).view(P, Hkv, hd)
                    .transpose(0, 1).double() for w in (0, 1)]
    else:
        prefix = None
    first = P if prefix else 0
    x, _ = _layers(case, emb[tok[:, first:]].double(), torch.arange(first, P + T, device="cuda"), prefix)
    n = _rms(x).view(-1, d)
    z = torch.empty(n.shape[0], V, dtype=torch.float64, device="cuda")
    if case["bits"] == 16:
        w = _normals(WEIGHT_SEED, 2, 0, V * d, 0.02).view(V, d)
    else:
        w = _matrix(case, 2, V, d)
    for a in range(0, V, 16384):
        z[:, a:a + 16384] = n @ w[a:a + 16384].double().T
    return {"logits": z.view(B, -1, V), "committed": None, "masked": None}


def exact(case, seed):
    if case["kind"] in ("step", "prefill"):
        return _exact_model(case, seed)
    t = _op_inputs(case, seed)
    if case["kind"] == "gemm":
        return t["X"].double() @ t["W"].double().T
    if case["kind"] == "attn":
        B, T, H, hd = case["B"], case["T"], case["H"], case["hd"]
        out = torch.empty(B, T, H * hd, dtype=torch.float64, device="cuda")
        for b in range(B):
            n = int(t["kv"][b]) + T
            o = _attention(t["q"][b].double(), t["k"][b, :, :n].double(), t["v"][b, :, :n].double())
            out[b] = o.transpose(0, 1).reshape(T, H * hd)
        return out.view(B * T, H * hd)
    z = torch.cat([t["X"].double() @ t["W"][a:a + 16384].double().T for a in range(0, case["V"], 16384)], 1)
    conf, tokconf = _decide(z, t["cur"], case["V"] - 1)
    return {"conf": conf, "tokconf": tokconf}
