"""The status words that nc_probs_to_cdf and nc_gemm_tc lease: 256 per device,
a call that finds none allocates its own.

* A stream that is being captured is refused, the capture goes on and no word
  is lost: with allocation made to fail, later calls still find one.
* 300 calls at once (each waiting behind a sleep on its stream, with the
  legacy stream asleep for longer, so that nothing ordered there has run
  yet): every call reports its own rows, also those that allocated.
"""
import threading

import pytest

import synthetic as S

pytestmark = pytest.mark.gpu

TINY = S.ModelShape(n_layers=1, d_model=64, n_heads=1, n_kv_heads=1, d_ffn=64, vocab=499, ctx_len=128, slide=32)


def _rows(V, bad):
    import torch
    p = torch.full((1, V), 1.0 / V, device="cuda")
    if bad:
        p[0, V // 2] = float("nan")
    return p, torch.empty(1, V + 1, dtype=torch.int32, device="cuda")


def test_captured_stream_is_refused_and_no_word_is_lost(gpu_lib, monkeypatch):
    import torch
    nc = gpu_lib
    p, cdf = _rows(1000, False)
    W = torch.randn(64, 64, device="cuda").bfloat16()
    Y = torch.empty(64, 64, device="cuda")
    assert nc.nc_probs_to_cdf(p, cdf, 24, 1) == nc.NC_OK and nc.nc_gemm_tc(W, W, Y) == nc.NC_OK
    x = torch.zeros(4, device="cuda")
    g, s = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        g.capture_begin(capture_error_mode="thread_local")
        x += 1
        got = {nc.nc_probs_to_cdf(p, cdf, 24, 1) for _ in range(300)} | {nc.nc_gemm_tc(W, W, Y) for _ in range(300)}
        x += 1
        g.capture_end()
    assert got == {nc.NC_ECUDA}
    g.replay()
    torch.cuda.synchronize()
    assert x.tolist() == [2.0] * 4
    cfg, w = nc.make_config(TINY, fmt="bf16"), S.flat_weights(TINY, 0)
    monkeypatch.setenv("NC24_FAIL_ALLOC_AFTER", "0")
    with pytest.raises(nc.NcError) as e:
        nc.Context(cfg, w)
    assert e.value.status == nc.NC_ENOMEM
    try:
        assert nc.nc_probs_to_cdf(p, cdf, 24, 1) == nc.NC_OK and nc.nc_gemm_tc(W, W, Y) == nc.NC_OK
    finally:
        monkeypatch.delenv("NC24_FAIL_ALLOC_AFTER")
        nc.Context(cfg, w).close()                   # allocations succeed again


def test_more_calls_at_once_than_words(gpu_lib):
    import torch
    nc = gpu_lib
    n, V = 300, 1000
    streams = [torch.cuda.Stream() for _ in range(32)]
    args = [_rows(V, bad=i % 3 == 0) for i in range(n)]
    nc.nc_probs_to_cdf(*args[1], 24, 1)
    for turn in range(2):
        got, gate = [None] * n, threading.Barrier(n)
        torch.cuda.synchronize()
        for s in streams:
            with torch.cuda.stream(s):
                torch.cuda._sleep(2_000_000_000)     # about a second
        torch.cuda._sleep(3_000_000_000)             # on the legacy stream

        def call(i):
            gate.wait()
            got[i] = nc.nc_probs_to_cdf(*args[i], 24, 1, stream=streams[i % 32])

        threads = [threading.Thread(target=call, args=(i,)) for i in range(n)]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        assert got == [nc.NC_ENUMERIC if i % 3 == 0 else nc.NC_OK for i in range(n)], turn
