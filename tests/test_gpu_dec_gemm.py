"""Projections of a decode step: the few-row kernels (up to 64 rows) give the
logits of the general tensor-core GEMM bit for bit.

A context of 65 streams takes the general kernels, smaller ones the few-row
variants (1 row per warp, 32- and 64-row tiles).  Both accumulate the same
products in the same order, so the bound is equality.  The shapes have K
blocks with a zero-filled tail (FFN 688) and the widths of the full model."""
import numpy as np
import pytest

import synthetic as S

pytestmark = pytest.mark.gpu

NARROW = S.ModelShape(n_layers=2, d_model=256, n_heads=4, n_kv_heads=2, d_ffn=688, vocab=999, ctx_len=128, slide=32)
WIDE = S.ModelShape(n_layers=2, d_model=576, n_heads=9, n_kv_heads=3, d_ffn=1536, vocab=999, ctx_len=128, slide=32)


def logits(nc, shape, w, fmt, max_streams, n, steps=3):
    import torch
    ctx = nc.Context(nc.make_config(shape, fmt=fmt, path="tc", warmup=2, max_streams=max_streams), w)
    ids = np.arange(n)
    toks = np.stack([S.token_stream(5, j, steps, shape.vocab) for j in range(n)])
    for j in ids:
        ctx.stream_open(int(j), steps)
    out = []
    for k in range(steps):
        z = torch.zeros(n, shape.vocab, device="cuda")
        ctx.step_probe(ids, z=z)
        ctx.update_bias(ids, toks[:, k])
        out.append(z.cpu().numpy())
    ctx.close()
    return out


@pytest.mark.parametrize("fmt", ["bf16", "fp8"])
@pytest.mark.parametrize("shape", [NARROW, WIDE], ids=["narrow", "wide"])
def test_few_row_projections_equal_general(fmt, shape):
    from paper_2602_19626_gb300 import nc24 as nc
    w = S.flat_weights(shape, 3)
    ref = logits(nc, shape, w, fmt, 65, 64)
    for n in (1, 8, 9, 32, 33, 64):
        got = logits(nc, shape, w, fmt, n, n)
        for k in range(len(ref)):
            assert np.array_equal(got[k], ref[k][:n]), (n, k)
