"""Decode attention over a BF16 cache: the cluster of a row's chunks has 1, 2,
4 or 8 CTAs by the longest stream of the launch, and every size gives the bits
of the prefill attention (equality: same products, sums and merge order).

Lengths sit at the edges of a chunk (256 positions) and of each cluster size;
the last crosses a window slide.  Two ragged streams share each launch."""
import numpy as np
import pytest

import synthetic as S

pytestmark = pytest.mark.gpu

SHAPE = S.ModelShape(n_layers=1, d_model=128, n_heads=2, n_kv_heads=1, d_ffn=128, vocab=499, ctx_len=2048, slide=512)
WIDE_GROUP = S.ModelShape(n_layers=1, d_model=256, n_heads=4, n_kv_heads=1, d_ffn=64, vocab=499, ctx_len=512, slide=128)


@pytest.mark.parametrize("path", ["gemv", "tc"])
@pytest.mark.parametrize("shape,lens", [(SHAPE, (256, 3)), (SHAPE, (257, 64)), (SHAPE, (513, 255)),
                                        (SHAPE, (1025, 1024)), (SHAPE, (2100, 700)), (WIDE_GROUP, (700, 130))])
def test_decode_attention_equals_prefill(shape, lens, path):
    import torch
    from paper_2602_19626_gb300 import nc24 as nc
    w = S.flat_weights(shape, 2)
    toks = [S.token_stream(9, j, n, shape.vocab) for j, n in enumerate(lens)]
    flat = torch.from_numpy(np.concatenate(toks)).cuda()
    offs = np.concatenate([[0], np.cumsum(lens)[:-1]])
    out = []
    for rows in (0, 256):
        ctx = nc.Context(nc.make_config(shape, fmt="bf16", path=path, warmup=9, max_streams=2, prefill_rows=rows), w)
        iv = torch.zeros(2, max(lens), 2, dtype=torch.int32, device="cuda")
        ctx.encode_intervals(flat, offs, np.array(lens), iv, max(lens))
        out.append(iv.cpu().numpy())
        ctx.close()
    assert np.array_equal(out[0], out[1])
