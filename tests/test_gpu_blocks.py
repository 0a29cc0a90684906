"""Building blocks at the edges of their kernels' pieces: the quantiser against
the oracle (exact) and the mixed NLL against float64.

Quantiser: vocabularies around the 128-symbol pieces of a warp and the 4,096
symbols of a cluster's piece; five rows start at every offset of a 16-byte
vector.  Mixed NLL: lengths around the 4-value loads, row counts on both sides
of the block-size rule.  Its bounds: a term's exponential and the sums carry
at most about 2^-23 each and sums of up to 2^16 terms over 2^5 partial sums
grow with the tree, so 1e-5 relative leaves a factor of ten."""
import numpy as np
import pytest

from oracle import cdf as Q

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("V", [2, 127, 128, 129, 4095, 4096, 4099, 8193, 16385, 32768, 32770, 49151, 65535])
def test_quantiser_pieces(V):
    import torch
    from paper_2602_19626_gb300 import nc24 as nc
    rng = np.random.default_rng(V)
    P = rng.dirichlet(np.full(V, 0.3), size=5).astype(np.float32)
    P[1] = 0.0
    P[1, V - 1] = 1.0
    P[2] = np.float32(1.0) / np.float32(V)
    cdf = torch.full((5, V + 1), -1, dtype=torch.int32, device="cuda")
    assert nc.nc_probs_to_cdf(torch.from_numpy(P).cuda(), cdf, 24, 1) == nc.NC_OK
    got = cdf.cpu().numpy().astype(np.uint32)
    for i in range(5):
        assert np.array_equal(got[i], Q.probs_to_cdf(P[i], 1 << 24, 1)), i


def test_quantiser_reports_one_bad_row_and_recovers():
    import torch
    from paper_2602_19626_gb300 import nc24 as nc
    V = 5000
    p = torch.full((9, V), 1.0 / V, device="cuda")
    cdf = torch.empty(9, V + 1, dtype=torch.int32, device="cuda")
    for bad in (float("nan"), float("inf"), -0.5, 2.0):
        q = p.clone()
        q[7, V - 1] = bad
        assert nc.nc_probs_to_cdf(q, cdf, 24, 1) == nc.NC_ENUMERIC
        assert nc.nc_probs_to_cdf(p, cdf, 24, 1) == nc.NC_OK


@pytest.mark.parametrize("n", [1, 152, 153])
@pytest.mark.parametrize("V", [2, 3, 1003, 4096, 49153])
def test_mixed_nll_lengths(n, V):
    import torch
    from paper_2602_19626_gb300.autograd import mixed_nll
    g = torch.Generator(device="cuda").manual_seed(n * 100003 + V)
    z = torch.randn(n, V, generator=g, device="cuda") * 3
    z[:, V // 2] = -float("inf")                     # a masked symbol
    b = (torch.randn(n, V, generator=g, device="cuda") * 0.1).requires_grad_()
    png = torch.softmax(torch.randn(n, V, generator=g, device="cuda"), 1)
    th = torch.randn(n, 2, generator=g, device="cuda").requires_grad_()
    t = torch.randint(0, V, (n,), generator=g, device="cuda")
    t[t == V // 2] = 0
    warm = (torch.rand(n, generator=g, device="cuda") < 0.5).to(torch.int32)
    loss = mixed_nll(b, th, z, png, t.to(torch.int32), warm, 0.8)
    loss.sum().backward()
    b2, th2 = b.detach().double().requires_grad_(), th.detach().double().requires_grad_()
    pt = torch.softmax(z.double() / 0.8 + b2, 1).gather(1, t[:, None])[:, 0]
    w = torch.softmax(th2, 1)
    want = -torch.log(torch.where(warm.bool(), pt, w[:, 0] * pt + w[:, 1] * png.double().gather(1, t[:, None])[:, 0]))
    want.sum().backward()
    for a, c in ((loss.detach(), want.detach()), (b.grad, b2.grad), (th.grad, th2.grad)):
        assert torch.isfinite(a).all()
        assert float((a.double() - c).norm() / c.norm().clamp_min(1e-30)) < 1e-5


def test_mixed_nll_non_finite_rows():
    import torch
    from paper_2602_19626_gb300.autograd import mixed_nll
    V = 1000
    z = torch.zeros(4, V, device="cuda")
    z[0, 3] = float("nan")
    z[1] = -float("inf")
    z[2, 5] = float("inf")
    arg = dict(b=torch.zeros(4, V, device="cuda"), theta=torch.zeros(4, 2, device="cuda"), z=z,
               p_ng=torch.full((4, V), 1.0 / V, device="cuda"), target=torch.zeros(4, dtype=torch.int32, device="cuda"),
               warm=torch.ones(4, dtype=torch.int32, device="cuda"))
    loss = mixed_nll(**arg)
    assert torch.isnan(loss[:3]).all() and torch.isfinite(loss[3])


@pytest.mark.parametrize("fp8,K", [(False, 192), (False, 200), (True, 208)])
def test_gemm_two_ctas_per_sm_equals_one(fp8, K):
    """From two tiles per SM on, nc_gemm_tc runs two CTAs per SM (bn up to
    128); bn 256 and few rows take one.  Every output accumulates its K blocks
    in one order, so the results are equal, ragged edges included."""
    import torch
    from paper_2602_19626_gb300 import nc24 as nc
    M, N = 1303, 3601                                # 11 x 29 tiles at bn 128
    g = torch.Generator(device="cuda").manual_seed(K)
    W = torch.randn(M, K, generator=g, device="cuda")
    X = torch.randn(N, K, generator=g, device="cuda")
    sc = dict(w_scale=None, x_scale=None)
    if fp8:
        sc = dict(w_scale=W.abs().amax(1) / 448, x_scale=X.abs().amax(1) / 448)
        W, X = (W / sc["w_scale"][:, None]).to(torch.float8_e4m3fn), (X / sc["x_scale"][:, None]).to(torch.float8_e4m3fn)
    else:
        W, X = W.to(torch.bfloat16), X.to(torch.bfloat16)
    ref = torch.empty(N, M, device="cuda")
    assert nc.nc_gemm_tc(W, X, ref, bn=256, fp8=fp8, **sc) == nc.NC_OK
    for bn in (32, 64, 128):
        Y = torch.full((N, M), float("nan"), device="cuda")
        assert nc.nc_gemm_tc(W, X, Y, bn=bn, fp8=fp8, **sc) == nc.NC_OK
        assert torch.equal(Y, ref), bn
    few = torch.empty(65, M, device="cuda")
    if fp8:
        sc["x_scale"] = sc["x_scale"][:65].contiguous()
    assert nc.nc_gemm_tc(W, X[:65].contiguous(), few, bn=128, fp8=fp8, **sc) == nc.NC_OK
    assert torch.equal(few, ref[:65])
