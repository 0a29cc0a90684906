"""A row of the mixed NLL has the same bits alone, in any batch and at any
alignment: the sums run in one order.  Rows of V not a multiple of four start
at every offset of a 16-byte vector, and the tensors may start at any float.

The float64 bound of the sum: 512 partial sums of up to 2^7 terms each, by
increasing symbol, then 9 additions: under 2^7 + 9 roundings of 2^-24 for the
sum, one of 2^-23 in each exponential, 2^-23 for the logarithm and the score's
own rounding (2^-24 of |s| <= 16): 2e-5 absolute on the loss leaves a factor of two."""
import pytest

pytestmark = pytest.mark.gpu


def _run(nc, z, b, png, th, t, w, g, tau):
    import torch
    n, V = z.shape
    loss = torch.empty(n, device="cuda")
    db, dth = torch.empty(n, V, device="cuda"), torch.empty(n, 2, device="cuda")
    assert nc.nc_mix_nll_fwd(z, b, png, th, t, w, tau, loss) == nc.NC_OK
    assert nc.nc_mix_nll_bwd(z, b, png, th, t, w, g, tau, db, dth) == nc.NC_OK
    torch.cuda.synchronize()
    return loss, db, dth


@pytest.mark.parametrize("V", [2, 511, 513, 4096, 4099, 50001])
def test_row_alone_equals_row_in_batch(gpu_lib, V):
    import torch
    nc = gpu_lib
    gen = torch.Generator(device="cuda").manual_seed(V)
    row = [torch.randn(1, V, generator=gen, device="cuda") * 3, torch.randn(1, V, generator=gen, device="cuda") * 0.1,
           torch.softmax(torch.randn(1, V, generator=gen, device="cuda"), 1),
           torch.randn(1, 2, generator=gen, device="cuda"), torch.tensor([V // 2], dtype=torch.int32, device="cuda"),
           torch.zeros(1, dtype=torch.int32, device="cuda"), torch.full((1,), 0.7, device="cuda")]
    want = _run(nc, *row, 0.8)
    s = row[0].double() / 0.8 + row[1].double()
    p = torch.softmax(s, 1)[0, V // 2]
    w = torch.softmax(row[3].double(), 1)[0]
    exact = -torch.log(w[0] * p + w[1] * row[2].double()[0, V // 2])
    assert abs(float(want[0][0]) - float(exact)) < 2e-5
    for n in (152, 153):
        got = _run(nc, *(x.repeat(n, *[1] * (x.dim() - 1)) for x in row), 0.8)
        for a, c in zip(got, want):
            assert torch.equal(a, c.expand_as(a)), n
    for off in (1, 2, 3):                            # the same row starting off a 16-byte vector
        moved = list(row)
        for i in (0, 1):
            flat = torch.empty(V + off, device="cuda")
            flat[off:] = row[i][0]
            moved[i] = flat[off:].view(1, V)
        for a, c in zip(_run(nc, *moved, 0.8), want):
            assert torch.equal(a, c), off
