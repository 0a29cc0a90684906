"""Routes of the per-token step that round trips do not tell apart.

* The model forward of nc_step_probe is replayed from a graph kept per cluster
  size of the attention (chosen by the longest stream of the batch).  Short and
  long streams stepped alone and together, in every order of the sizes and on
  a stream that cannot be captured, give the logits that a per-token encode of
  another context gives, bit for bit.
* The decoder's symbol search: targets on both edges of a symbol's interval,
  around the first maximum (whose count takes the residual) and at the ends,
  as one-token rANS streams whose state is the target, against the CDF.
* A status raised in one row among many reaches the host and is cleared.
"""
import ctypes as C
import struct

import numpy as np
import pytest

import synthetic as S

pytestmark = pytest.mark.gpu

SHAPE = S.ModelShape(n_layers=1, d_model=128, n_heads=2, n_kv_heads=1, d_ffn=128, vocab=499, ctx_len=2048, slide=512)
LENS = (20, 300, 600, 1100)                          # windows of 1, 2, 4 and 8 CTAs' chunks
CHECK = (0, 1, 19, 255, 256, 257, 299, 511, 512, 513, 599, 1023, 1024, 1025, 1099)


@pytest.mark.parametrize("fmt,path,stream", [("bf16", "tc", None), ("bf16", "gemv", None), ("fp32", "gemv", None),
                                             ("bf16", "tc", 1)], ids=["tc", "gemv", "fp32", "legacy_stream"])
def test_kept_step_graphs(fmt, path, stream):
    import torch
    from paper_2602_19626_gb300 import nc24 as nc
    w, V = S.flat_weights(SHAPE, 4), SHAPE.vocab
    toks = [S.token_stream(11, j, n, V) for j, n in enumerate(LENS)]
    conf = dict(fmt=fmt, path=path, warmup=7, max_streams=4)
    want = {}
    ref = nc.Context(nc.make_config(SHAPE, **conf), w)
    flat, lens = torch.from_numpy(np.concatenate(toks)).cuda(), np.array(LENS)
    offs = np.concatenate([[0], np.cumsum(LENS)[:-1]])
    iv = torch.zeros(4, max(LENS), 2, dtype=torch.int32, device="cuda")
    for k in CHECK:
        z = torch.zeros(4, V, device="cuda")
        ref.encode_probe(flat, offs, lens, iv, max(LENS), k, z=z)
        want[k] = z.cpu().numpy()
    ref.close()

    ctx = nc.Context(nc.make_config(SHAPE, stream=stream, **conf), w)   # 1: cudaStreamLegacy, not capturable
    live = list(range(4))
    for j in live:
        ctx.stream_open(j, LENS[j])
    z = torch.zeros(4, V, device="cuda")

    def step(ids, k):
        ctx.step_probe(ids, z=z)
        if k in want:
            got = z.cpu().numpy()
            for i, j in enumerate(ids):
                assert np.array_equal(got[i], want[k][j]), (k, j, ids)
        ctx.update_bias(ids, [toks[j][k] for j in ids])

    for k in range(max(LENS)):
        live = [j for j in range(4) if k < LENS[j]]
        if k % 3 == 0:
            step(live, k)                            # the longest stream's class
        else:
            for j in live if k % 3 == 1 else live[::-1]:
                step([j], k)                         # each stream's own
    for j in range(4):
        ctx.stream_close(j)
    ctx.stream_open(9, LENS[3])                      # a slot and a class used before
    toks.append(toks[3])
    for k in range(3):
        ctx.step_probe([9], z=z)
        if k in want:
            assert np.array_equal(z.cpu().numpy()[0], want[k][3])
        ctx.update_bias([9], [toks[3][k]])
    ctx.close()


@pytest.mark.parametrize("V,n", [(499, 1), (499, 40), (16384, 1), (16384, 40), (16390, 40)])
def test_decoder_search_on_interval_edges(V, n):
    from paper_2602_19626_gb300 import nc24 as nc
    shape = S.ModelShape(n_layers=1, d_model=64, n_heads=1, n_kv_heads=1, d_ffn=64, vocab=V, ctx_len=128, slide=32)
    w = S.flat_weights(shape, 6) * np.float32(12)    # a peaked distribution
    ctx = nc.Context(nc.make_config(shape, fmt="bf16", path="tc", coder="rans", max_streams=n), w)
    ctx.stream_open(0, 1)
    cdf = ctx.step_cdf([0])[0].astype(np.int64)
    ctx.stream_close(0)
    head = ctx.encode([np.zeros(1, np.int32)])[:10]
    top = int(np.argmax(np.diff(cdf)))
    near = [s for s in (0, 1, top - 1, top, top + 1, V // 3, V - 2, V - 1) if 0 <= s < V]
    targets = sorted({int(t) for s in near for t in (cdf[s], cdf[s + 1] - 1)})
    if n > 1:
        targets += [int(t) for t in np.random.default_rng(V).integers(0, 1 << 24, n - len(targets))]
    for t0 in range(0, len(targets), n):
        part = targets[t0:t0 + n]
        blob = (head[:7] + struct.pack("<H", len(part)) + head[9:] + struct.pack("<III", 1, 64, 8) * len(part) +
                b"".join(struct.pack("<Q", (1 << 31) + t) for t in part))
        buf = np.frombuffer(blob, np.uint8).copy()
        out = [np.full(1, -1, np.int32) for _ in part]
        ptrs = (C.c_void_p * len(part))(*[o.ctypes.data for o in out])
        lens = np.zeros(len(part), np.int64)
        # the streams do not end in rANS's initial state: reported after the tokens
        assert nc.lib.nc_decode(ctx.h, buf.ctypes.data, buf.size, ptrs, lens.ctypes.data) == nc.NC_ECORRUPT
        got = np.array([o[0] for o in out])
        assert np.array_equal(got, np.searchsorted(cdf, part, side="right") - 1)
    ctx.close()


def test_one_raised_status_among_many_rows():
    import torch
    from paper_2602_19626_gb300 import nc24 as nc
    shape = S.ModelShape(n_layers=1, d_model=64, n_heads=1, n_kv_heads=1, d_ffn=64, vocab=99, ctx_len=32, slide=8)
    n = 1100                                         # more rows than the gathering block has threads
    ctx = nc.Context(nc.make_config(shape, fmt="bf16", path="tc", max_streams=n), S.flat_weights(shape, 1))
    iv = torch.zeros(n, 2, 2, dtype=torch.int32, device="cuda")
    offs, lens = np.arange(n) * 2, np.full(n, 2)
    for bad in (0, 33, 1023, 1024, 1099):
        toks = torch.ones(2 * n, dtype=torch.int32, device="cuda")
        toks[2 * bad + 1] = 99
        with pytest.raises(nc.NcError) as e:
            ctx.encode_intervals(toks, offs, lens, iv, 2)
        assert e.value.status == nc.NC_EINVAL, bad
        ctx.encode_intervals(torch.ones_like(toks), offs, lens, iv, 2)
    ctx.close()
