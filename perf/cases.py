"""The work that users of nc24 have it do, as cases that can be timed and compared.

A case is a call, or a short run of calls, of the public binding
(``paper_2602_19626_gb300.nc24`` and ``.autograd``):

* ``step``    a program with its own entropy coder: open streams, one
              nc_step_probe and nc_update_bias per token, read the adaptive
              state, close;
* ``decode``  nc_decode of a container (the decompressor);
* ``encode``  nc_encode of host tokens into a container (the compressor), a
              file cut into chunks where ``file`` is set;
* ``probe``   nc_encode_probe: the batched compressor's device half, with the
              logits and distributions of one token of every stream;
* ``gemm``    nc_gemm_tc, one projection over a batch of rows;
* ``cdf``     nc_probs_to_cdf, the quantiser over rows of probabilities;
* ``mixnll``  forward and backward of the mixed-distribution loss under
              autograd, one training step's loss and gradients.

Model sizes are the two the package's tests and benchmark run: the
135M-parameter shape ("full") and a four-layer one ("small").  Weights are
random-init N(0, 0.02) as a BF16 checkpoint holds them; tokens are Zipf(1.1)
ids with recurring phrases, so that the N-gram contexts fill as in text.
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_2602_19626_gb300 import nc24
from paper_2602_19626_gb300.autograd import mixed_nll

SHAPES = {
    "full": SimpleNamespace(n_layers=30, d_model=576, n_heads=9, n_kv_heads=3, d_ffn=1536, vocab=49152,
                            ctx_len=2048, slide=512, rope_theta=1e5, rms_eps=1e-5),
    "small": SimpleNamespace(n_layers=4, d_model=256, n_heads=4, n_kv_heads=2, d_ffn=688, vocab=49152,
                             ctx_len=512, slide=128, rope_theta=1e5, rms_eps=1e-5),
}
D_HEAD = 64
WARMUP, ALPHA, ETA, W_LLM, ORDER = 100, 1e-3, 1.0, 0.85, 3      # the library's defaults


def listed():
    return [
        # the smallest call in use: a few tokens of one stream of the small
        # FP32 model, through a caller's own coder; launches and host calls
        dict(name="step_small_fp32", kind="step", shape="small", fmt="fp32", path="gemv", n=1, steps=16),
        # one stream of the full model with the library's default
        # configuration (BF16 weights, GEMV path), token by token
        dict(name="step_one_bf16", kind="step", shape="full", fmt="bf16", path="gemv", n=1, steps=24),
        # a server stepping an odd number of streams together on the
        # tensor-core path
        dict(name="step_batch_tc", kind="step", shape="full", fmt="bf16", path="tc", n=37, steps=6),
        # decompression of one stream: one dependent step per token
        dict(name="decode_one_tc", kind="decode", shape="full", fmt="bf16", path="tc", n=1, lo=300, hi=300,
             coder="arith"),
        # decompression of a batch of ragged FP8 streams, rANS coder
        dict(name="decode_batch_fp8", kind="decode", shape="full", fmt="fp8", path="tc", n=48, lo=20, hi=160,
             coder="rans"),
        # compression of one long stream (the benchmark's headline workload),
        # host tokens in, container bytes out
        dict(name="encode_one_tc", kind="encode", shape="full", fmt="bf16", path="tc", n=1, lo=8192, hi=8192,
             rows=4096, rule="paper", skip=False, coder="arith", file=False),
        # one file as the eight chunks of a container, with the differentiable
        # (mixed-NLL) update rule
        dict(name="encode_file_nll", kind="encode", shape="full", fmt="bf16", path="tc", n=8, lo=12000, hi=12000,
             rows=4096, rule="mixed_nll", skip=False, coder="arith", file=True),
        # batched compression of ragged BF16 streams: the throughput workload
        dict(name="probe_batch_bf16", kind="probe", shape="full", fmt="bf16", path="tc", n=96, lo=128, hi=2048,
             rows=4096, at=150),
        # many short FP8 streams: the precision workload
        dict(name="probe_batch_fp8", kind="probe", shape="full", fmt="fp8", path="tc", n=320, lo=96, hi=320,
             rows=4096, at=70),
        # the largest projection, the tied LM head, over a prefill forward's rows
        dict(name="gemm_bf16", kind="gemm", fp8=False, M=49152, K=576, N=1024),
        # the quantiser over a batch of rows of a caller's probabilities
        dict(name="cdf_rows", kind="cdf", n=256, V=49152),
        # one training step of the bias head and mixer weights
        dict(name="mixnll_train", kind="mixnll", n=512, V=49152, tau=1.0),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["step", "step", "decode", "decode", "encode", "encode", "probe", "probe", "gemm", "cdf", "mixnll"])
    if kind == "gemm":
        fp8 = rng.random() < 0.4
        K = 16 * _log_int(rng, 4, 192)
        return dict(kind=kind, fp8=fp8, M=_log_int(rng, 33, 4097), K=K, N=_log_int(rng, 1, 4096))
    if kind == "cdf":
        return dict(kind=kind, n=_log_int(rng, 1, 256), V=_log_int(rng, 257, 50001))
    if kind == "mixnll":
        return dict(kind=kind, n=_log_int(rng, 1, 512), V=_log_int(rng, 257, 50001), tau=rng.choice([1.0, 0.8]))
    path, fmt = rng.choice([("gemv", "fp32"), ("gemv", "bf16"), ("tc", "bf16"), ("tc", "bf16"), ("tc", "fp8")])
    shape = "small" if rng.random() < 0.25 else "full"
    base = dict(kind=kind, shape=shape, fmt=fmt, path=path)
    if kind == "step":
        return dict(base, n=_log_int(rng, 1, 48 if path == "tc" else 6), steps=rng.randint(3, 16))
    if kind == "decode":
        n = _log_int(rng, 1, 48 if path == "tc" else 4)
        hi = _log_int(rng, 17, 120)
        return dict(base, n=n, lo=max(1, hi // 5), hi=hi, coder=rng.choice(["arith", "rans"]))
    if path == "gemv":                      # CUDA-core projections: small batches only
        n, hi = _log_int(rng, 1, 3), _log_int(rng, 30, 300)
    else:
        n = _log_int(rng, 1, 96)
        hi = min(_log_int(rng, 60, 4000), max(60, 60000 // n))
    if kind == "encode":
        return dict(base, n=n, lo=max(1, hi // 4), hi=hi, rows=rng.choice([512, 1024, 4096]),
                    rule=rng.choice(["paper", "mixed_nll"]), skip=rng.random() < 0.3,
                    coder=rng.choice(["arith", "rans"]), file=False)
    return dict(base, n=n, lo=max(1, hi // 4), hi=hi, rows=rng.choice([512, 1024, 4096]),
                at=rng.randint(3, min(140, hi - 1)))


# ------------------------------------------------------------------- inputs

def _tensors(s):
    """(name, shape) in the order of nc_ctx_create's weight buffer."""
    d, F, kv = s.d_model, s.d_ffn, s.n_kv_heads * D_HEAD
    yield "embed", (s.vocab, d)
    for l in range(s.n_layers):
        yield f"{l}.g1", (d,)
        yield f"{l}.q", (d, d)
        yield f"{l}.k", (kv, d)
        yield f"{l}.v", (kv, d)
        yield f"{l}.o", (d, d)
        yield f"{l}.g2", (d,)
        yield f"{l}.gate", (F, d)
        yield f"{l}.up", (F, d)
        yield f"{l}.down", (d, F)
    yield "g", (d,)


def _weights(s, seed):
    """The flat FP32 buffer on the GPU: BF16-representable N(0, 0.02), gains 1."""
    n = sum(math.prod(shape) for _, shape in _tensors(s))
    g = torch.Generator(device="cuda").manual_seed(seed * 1000003 + 17)
    w = (torch.randn(n, generator=g, device="cuda") * 0.02).to(torch.bfloat16).float()
    off = 0
    for _, shape in _tensors(s):
        if len(shape) == 1:
            w[off:off + shape[0]] = 1.0
        off += math.prod(shape)
    return w


def _stream(rng, n, V):
    """n token ids: Zipf(1.1) draws and recurring phrases, through a permutation."""
    p = np.arange(1, V + 1, dtype=np.float64) ** -1.1
    c = np.cumsum(p)
    c /= c[-1]
    perm = rng.permutation(V).astype(np.int32)
    iid = perm[np.minimum(np.searchsorted(c, rng.random(n + 600)), V - 1)]
    phrases = [iid[n + 8 * j: n + 8 * j + int(k)] for j, k in enumerate(rng.integers(2, 9, 64))]
    out, at, have = [], 0, 0
    picks, single = rng.integers(0, 64, n + 1), rng.integers(1, 6, n + 1)
    for j in range(n + 1):
        if have >= n:
            break
        out += [phrases[min(int(picks[j]), int(picks[-1 - j]))], iid[at:at + single[j]]]
        at += int(single[j])
        have += len(out[-1]) + len(out[-2])
    return np.ascontiguousarray(np.concatenate(out)[:n], dtype=np.int32)


def _streams(c, seed):
    """The case's streams: log-uniform lengths that belong to the case, tokens from the seed."""
    rng = np.random.default_rng([c["n"], c["lo"], c["hi"]])
    lens = np.exp(rng.uniform(math.log(c["lo"]), math.log(c["hi"] + 1), c["n"])).astype(np.int64)
    lens = np.clip(lens, c["lo"], c["hi"])
    lens[rng.integers(0, c["n"])] = c["hi"]
    rng = np.random.default_rng([seed, 91])
    return [_stream(rng, int(k), SHAPES[c["shape"]].vocab) for k in lens]


def _step_tokens(c, seed):
    rng = np.random.default_rng([seed, 92])
    return np.stack([_stream(rng, c["steps"], SHAPES[c["shape"]].vocab) for _ in range(c["n"])])


def _context(c, seed, rows=0, max_streams=None):
    s = SHAPES[c["shape"]]
    cfg = nc24.make_config(s, fmt=c["fmt"], path=c["path"], max_streams=max_streams or c["n"], prefill_rows=rows,
                           rule=c.get("rule", "paper"), skip=c.get("skip", False), coder=c.get("coder", "arith"))
    return nc24.Context(cfg, _weights(s, seed).cpu().numpy())


def _gemm_inputs(c, seed):
    g = torch.Generator(device="cuda").manual_seed(seed * 7919 + 3)
    W = torch.randn(c["M"], c["K"], generator=g, device="cuda") * 0.02
    X = torch.randn(c["N"], c["K"], generator=g, device="cuda")
    if not c["fp8"]:
        return W.to(torch.bfloat16), X.to(torch.bfloat16), None, None
    ws, xs = W.abs().amax(1) / 448, X.abs().amax(1) / 448
    return (W / ws[:, None]).to(torch.float8_e4m3fn), (X / xs[:, None]).to(torch.float8_e4m3fn), ws, xs


def _nll_inputs(c, seed):
    """Logits, a head some way into a stream, an N-gram's sparse-plus-flat
    distribution, mixer weights; a third of the rows in warm-up."""
    n, V = c["n"], c["V"]
    g = torch.Generator(device="cuda").manual_seed(seed * 104729 + 5)
    z = torch.randn(n, V, generator=g, device="cuda")
    b = torch.randn(n, V, generator=g, device="cuda") * 0.01
    png = torch.full((n, V), 1.0, device="cuda")
    hot = torch.randint(0, V, (n, 40), generator=g, device="cuda")
    png.scatter_(1, hot, 0.02 * V)
    png /= png.sum(1, keepdim=True)
    theta = torch.log(torch.rand(n, 2, generator=g, device="cuda") * 0.8 + 0.1)
    target = torch.where(torch.rand(n, generator=g, device="cuda") < 0.5, hot[:, 0],
                         torch.randint(0, V, (n,), generator=g, device="cuda")).to(torch.int32)
    warm = (torch.rand(n, generator=g, device="cuda") < 0.33).to(torch.int32)
    return z, b, png, theta, target, warm


def _probs(c, seed):
    g = torch.Generator(device="cuda").manual_seed(seed * 15485863 + 7)
    return torch.softmax(torch.randn(c["n"], c["V"], generator=g, device="cuda") * 2.0, dim=1)


def prepare(case, seed):
    c = dict(case)
    k = c["kind"]
    if k == "gemm":
        W, X, ws, xs = _gemm_inputs(c, seed)
        bn = next((b for b in (32, 64, 128) if c["N"] <= b), 128)
        return dict(c, W=W, X=X, ws=ws, xs=xs, bn=bn, Y=torch.empty(c["N"], c["M"], device="cuda"))
    if k == "cdf":
        return dict(c, p=_probs(c, seed), cdf=torch.empty(c["n"], c["V"] + 1, dtype=torch.int32, device="cuda"))
    if k == "mixnll":
        z, b, png, theta, target, warm = _nll_inputs(c, seed)
        return dict(c, z=z, b=b.requires_grad_(), png=png, theta=theta.requires_grad_(), target=target, warm=warm)
    V = SHAPES[c["shape"]].vocab
    if k == "step":
        new = lambda w, dt: torch.zeros(c["steps"], c["n"], w, dtype=dt, device="cuda")     # noqa: E731
        return dict(c, ctx=_context(c, seed), ids=np.arange(c["n"], dtype=np.int32),
                    tok=np.ascontiguousarray(_step_tokens(c, seed).T),
                    z=new(V, torch.float32), pt=new(V, torch.float32), png=new(V, torch.float32),
                    p=new(V, torch.float32), cdf=new(V + 1, torch.int32))
    streams = _streams(c, seed)
    if k == "decode":
        ctx = _context(c, seed, rows=1024)
        return dict(c, ctx=ctx, data=ctx.encode(streams))
    ctx = _context(c, seed, rows=c["rows"])
    if k == "encode":
        lines = (np.random.default_rng([seed, 93]).random(V) < 0.05).astype(np.uint8)
        # a buffer of fixed size for the container: at most 26 bits a token and 40 bytes a stream
        room = 64 + c["n"] * 40 + sum(t.size for t in streams) * 26 // 8
        return dict(c, ctx=ctx, streams=streams, lines=lines, out=np.zeros(room, dtype=np.uint8))
    lens = np.array([t.size for t in streams], dtype=np.int64)
    new = lambda: torch.zeros(c["n"], V, device="cuda")                                     # noqa: E731
    return dict(c, ctx=ctx, tok=torch.from_numpy(np.concatenate(streams)).cuda(),
                offs=np.concatenate([[0], np.cumsum(lens)[:-1]]).astype(np.int64), lens=lens,
                iv=torch.zeros(c["n"], int(lens.max()), 2, dtype=torch.int32, device="cuda"),
                z=new(), pt=new(), png=new(), p=new())


def _ok(status, what):
    if status:
        raise nc24.NcError(status, what)


def run(st):
    k = st["kind"]
    if k == "gemm":
        _ok(nc24.nc_gemm_tc(st["W"], st["X"], st["Y"], bn=st["bn"], w_scale=st["ws"], x_scale=st["xs"],
                            fp8=st["fp8"]), "nc_gemm_tc")
        return st["Y"]
    if k == "cdf":
        _ok(nc24.nc_probs_to_cdf(st["p"], st["cdf"]), "nc_probs_to_cdf")
        return st["cdf"]
    if k == "mixnll":
        b, theta = st["b"], st["theta"]
        b.grad = theta.grad = None
        loss = mixed_nll(b, theta, st["z"], st["png"], st["target"], st["warm"], st["tau"])
        loss.sum().backward()
        return dict(loss=loss.detach(), db=b.grad, dtheta=theta.grad)
    ctx = st["ctx"]
    if k == "step":
        ids, tok = st["ids"], st["tok"]
        for i in ids:
            ctx.stream_open(int(i), st["steps"])
        for t in range(st["steps"]):
            ctx.step_probe(ids, z=st["z"][t], p_tilde=st["pt"][t], p_ng=st["png"][t], p=st["p"][t],
                           cdf_out=st["cdf"][t])
            ctx.update_bias(ids, tok[t])
        state = [ctx.stream_state(int(i)) for i in ids]
        for i in ids:
            ctx.stream_close(int(i))
        return dict(z=st["z"], p_tilde=st["pt"], p_ng=st["png"], p=st["p"], cdf=st["cdf"],
                    bias=np.stack([s[0] for s in state]), theta=np.stack([s[1] for s in state]))
    if k == "decode":
        out = ctx.decode(st["data"])
        return dict(tokens=np.concatenate(out), lens=np.array([o.size for o in out]))
    if k == "encode":
        data = (ctx.encode_file(st["streams"][0], st["lines"], st["n"]) if st["file"] else ctx.encode(st["streams"]))
        st["out"][:] = 0
        st["out"][:len(data)] = np.frombuffer(data, dtype=np.uint8)
        return dict(container=st["out"], nbytes=len(data))
    ctx.encode_probe(st["tok"], st["offs"], st["lens"], st["iv"], st["iv"].shape[1], st["at"], z=st["z"],
                     p_tilde=st["pt"], p_ng=st["png"], p=st["p"])
    return dict(intervals=st["iv"], z=st["z"], p_tilde=st["pt"], p_ng=st["png"], p=st["p"])


# --------------------------------------------------------------------- work

def _model_work(s, fmt, tokens, ctx_sum, forwards):
    """Bytes (the weights once per dependent forward: they exceed the L2) and
    flops of the model over `tokens` tokens with `ctx_sum` window entries."""
    d, F, kv = s.d_model, s.d_ffn, s.n_kv_heads * D_HEAD
    par = s.vocab * d + s.n_layers * (2 * d * d + 2 * kv * d + 3 * F * d)
    esz = {"fp32": 4, "bf16": 2, "fp8": 1}[fmt]
    kvb = 2 * kv * s.n_layers * (4 if fmt == "fp32" else 2)
    return forwards * par * esz + tokens * kvb, 2.0 * par * tokens + 4.0 * d * s.n_layers * ctx_sum


def _window(s, n):
    """Window entries over a stream's n positions (slides included)."""
    a = np.arange(n, dtype=np.int64)
    start = np.where(a < s.ctx_len, 0, ((a - s.ctx_len) // s.slide + 1) * s.slide)
    return float((a - start + 1).sum())


def work(case):
    c, k = case, case["kind"]
    if k == "gemm":
        e = 1 if c["fp8"] else 2
        return dict(bytes=e * c["K"] * (c["M"] + c["N"]) + 4 * c["M"] * c["N"], flops=2 * c["M"] * c["N"] * c["K"])
    if k == "cdf":
        return dict(bytes=c["n"] * (8 * c["V"] + 4), flops=2 * c["n"] * c["V"])
    if k == "mixnll":         # z, b, the targets' probabilities; db written; two passes' exponentials
        return dict(bytes=c["n"] * (12 * c["V"] + 40), flops=12 * c["n"] * c["V"])
    s = SHAPES[c["shape"]]
    if k == "step":
        by, fl = _model_work(s, c["fmt"], c["n"] * c["steps"], c["n"] * _window(s, c["steps"]), c["steps"])
        return dict(bytes=by + c["n"] * c["steps"] * 20 * s.vocab + 4 * c["n"] * s.vocab, flops=fl)
    lens = [c["hi"]] + [int((c["hi"] - c["lo"]) / max(math.log(c["hi"] / c["lo"]), 1e-9)) or c["lo"]
                        if c["hi"] > c["lo"] else c["hi"]] * (c["n"] - 1)
    if c.get("file"):
        lens = [c["hi"] // c["n"]] * c["n"]
    tok = sum(lens)
    by, fl = _model_work(s, c["fmt"], tok, sum(_window(s, n) for n in lens), c["hi"] if k == "decode" else 1)
    return dict(bytes=by + tok * 12 + (c["n"] * s.vocab * 16 if k == "probe" else 0), flops=fl)


# -------------------------------------------------------------------- exact

def _stored(w, fmt):
    """FP64 values of a matrix as its storage format holds them (the weights
    are BF16 values already; E4M3 with one scale per output row)."""
    if fmt != "fp8":
        return w.double()
    sc = w.abs().amax(1, keepdim=True) / 448
    sc = torch.where(sc > 0, sc, torch.ones_like(sc))
    return (w / sc).to(torch.float8_e4m3fn).double() * sc.double()


def _logits(c, seed, toks):
    """FP64 logits [n, T, V] of n streams of T inputs (no window slide: T <= L)."""
    s = SHAPES[c["shape"]]
    flat, W, off = _weights(s, seed), {}, 0
    for name, shape in _tensors(s):
        m = math.prod(shape)
        t = flat[off:off + m].view(shape)
        W[name] = t.double() if len(shape) == 1 else _stored(t, c["fmt"])
        off += m
    n, T = toks.shape
    hq, hk = s.n_heads, s.n_kv_heads
    j = torch.arange(32, dtype=torch.float64, device="cuda")
    ang = torch.arange(T, dtype=torch.float64, device="cuda")[:, None] * s.rope_theta ** (-2.0 * j / D_HEAD)
    co, si = ang.cos()[:, None], ang.sin()[:, None]

    def norm(x, g):
        return x / torch.sqrt((x * x).mean(-1, keepdim=True) + s.rms_eps) * g

    def rot(x):
        a, b = x[..., :32], x[..., 32:]
        return torch.cat([a * co - b * si, b * co + a * si], -1)

    mask = torch.full((T, T), -math.inf, dtype=torch.float64, device="cuda").triu(1)
    x = W["embed"][torch.from_numpy(toks.astype(np.int64)).cuda()]
    for l in range(s.n_layers):
        a = norm(x, W[f"{l}.g1"])
        q = rot((a @ W[f"{l}.q"].T).view(n, T, hq, D_HEAD))
        k = rot((a @ W[f"{l}.k"].T).view(n, T, hk, D_HEAD)).repeat_interleave(hq // hk, 2)
        v = (a @ W[f"{l}.v"].T).view(n, T, hk, D_HEAD).repeat_interleave(hq // hk, 2)
        w = torch.softmax(torch.einsum("nihd,njhd->nhij", q, k) / 8.0 + mask, -1)
        x = x + torch.einsum("nhij,njhd->nihd", w, v).reshape(n, T, -1) @ W[f"{l}.o"].T
        f = norm(x, W[f"{l}.g2"])
        x = x + (torch.nn.functional.silu(f @ W[f"{l}.gate"].T) * (f @ W[f"{l}.up"].T)) @ W[f"{l}.down"].T
    return norm(x, W["g"]) @ W["embed"].T


class _NGram:
    """Orders 1..3 over exact contexts, 64 continuations each, Laplace unigram."""

    def __init__(self, V):
        self.V, self.N, self.uni, self.tab, self.hist = V, 0, np.zeros(V), {}, ()

    def predict(self):
        P = (self.uni + 1.0) / (self.N + self.V)
        for k in range(1, ORDER + 1):
            e = self.tab.get(self.hist[-k:]) if len(self.hist) >= k else None
            if e:
                n = sum(c for _, c in e)
                P *= 1.0 - n / (n + 5.0)
                for t, cnt in e:
                    P[t] += cnt / (n + 5.0)
        return P

    def update(self, t):
        for k in range(1, min(ORDER, len(self.hist)) + 1):
            e = self.tab.setdefault(self.hist[-k:], [])
            hit = next((x for x in e if x[0] == t), None)
            if hit:
                hit[1] += 1
            elif len(e) < 64:
                e.append([t, 1])
            else:
                e[min(range(64), key=lambda i: (e[i][1], i))] = [t, 1]
        self.uni[t] += 1
        self.N += 1
        self.hist = (self.hist + (t,))[-ORDER:]


def _replay(z, toks, want):
    """The distributions at the positions in `want` (each [n, V] FP64) and the
    final head and mixer state, from logits z [n, T, V] and the coded tokens."""
    n, T, V = z.shape
    ng = [_NGram(V) for _ in range(n)]
    b = torch.zeros(n, V, dtype=torch.float64, device="cuda")
    th = torch.log(torch.tensor([[W_LLM, 1 - W_LLM]], dtype=torch.float64, device="cuda")).repeat(n, 1)
    rows, out = torch.arange(n, device="cuda"), []
    for t in range(T):
        pt = torch.softmax(z[:, t] + b, -1)
        tt = torch.from_numpy(toks[:, t].astype(np.int64)).cuda()
        warm = t < WARMUP
        png = None
        if t in want or not warm:
            png = torch.from_numpy(np.stack([g.predict() for g in ng])).cuda()
        w = torch.softmax(th, -1)
        if t in want:
            out.append((z[:, t], pt, png, pt if warm else w[:, :1] * pt + w[:, 1:] * png))
        if not warm:
            th = torch.log_softmax(th + ETA * torch.log(torch.stack([pt[rows, tt], png[rows, tt]], 1)), -1)
        b = b - ALPHA * pt
        b[rows, tt] += ALPHA
        for r in range(n):
            ng[r].update(int(toks[r, t]))
    return out, b, th


def exact(case, seed):
    c, k = case, case["kind"]
    if k == "gemm":
        W, X, ws, xs = _gemm_inputs(c, seed)
        Y = X.double() @ W.double().T
        return Y * ws.double() * xs.double()[:, None] if c["fp8"] else Y
    if k == "mixnll":
        z, b, png, theta, target, warm = _nll_inputs(c, seed)
        b, theta = b.double().requires_grad_(), theta.double().requires_grad_()
        t = target.long()[:, None]
        pt = torch.softmax(z.double() / c["tau"] + b, -1).gather(1, t)[:, 0]
        w = torch.softmax(theta, -1)
        mix = w[:, 0] * pt + w[:, 1] * png.double().gather(1, t)[:, 0]
        loss = -torch.log(torch.where(warm.bool(), pt, mix))
        loss.sum().backward()
        return dict(loss=loss.detach(), db=b.grad, dtheta=theta.grad)
    if k == "step":
        toks = _step_tokens(c, seed)
        fed = np.concatenate([np.zeros((c["n"], 1), np.int32), toks[:, :-1]], 1)
        out, b, th = _replay(_logits(c, seed, fed), toks, range(c["steps"]))
        z, pt, png, p = (torch.stack([o[i] for o in out]) for i in range(4))
        return dict(z=z, p_tilde=pt, p_ng=png, p=p, cdf=None, bias=b, theta=th)
    if k == "probe":
        streams, at = _streams(c, seed), c["at"]
        long = [j for j, t in enumerate(streams) if t.size > at]
        if len(long) * at > 40000:
            return None
        toks = np.stack([streams[j][:at + 1] for j in long])
        fed = np.concatenate([np.zeros((len(long), 1), np.int32), toks[:, :-1]], 1)
        res = [[torch.zeros(c["n"], SHAPES[c["shape"]].vocab, dtype=torch.float64, device="cuda")] for _ in range(4)]
        for a in range(0, len(long), 32):
            got = _replay(_logits(c, seed, fed[a:a + 32]), toks[a:a + 32], (at,))[0][0]
            for i in range(4):
                res[i][0][long[a:a + 32]] = got[i]
        return dict(intervals=None, z=res[0][0], p_tilde=res[1][0], p_ng=res[2][0], p=res[3][0])
    return None
