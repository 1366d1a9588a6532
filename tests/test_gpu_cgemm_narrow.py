"""Complex64 products of at most four columns, 64 to 255 rows and a sum of at
most eight (64 x 4 tiles, two a block), at their edges, against the plain
definition; operands and result on and off 16 bytes."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("off", [0, 1])
@pytest.mark.parametrize("batch,m,n,k", [(1, 64, 1, 1), (3, 65, 2, 3), (7, 127, 3, 4), (5, 128, 4, 5), (301, 255, 4, 8),
                                         (33, 64, 3, 7), (2, 255, 1, 8)])
def test_narrow(batch, m, n, k, off):
    import torch
    import paper_1907_11217_gb300 as tz
    g = torch.Generator(device="cuda").manual_seed(m + 3 * n + 5 * k)
    A, B = (torch.randn(2 * (batch * r * k + off), device="cuda", generator=g)[2 * off:] for r in (m, n))
    gap = 3  # elements between the products of a batch
    sc = m * n + gap
    buf = torch.full((2 * (batch * sc + off),), float("nan"), device="cuda")
    tz.tz_op_cgemm("c64", batch, m, n, k, A, m * k, B, n * k, buf[2 * off:], sc)
    out = torch.view_as_complex(buf[2 * off:].view(batch, sc, 2).double())
    assert bool(torch.isnan(out[:, m * n:].real).all()) and bool(torch.isnan(buf[: 2 * off]).all())
    a, b = (torch.view_as_complex(x.reshape(batch, r, k, 2).double()) for x, r in ((A, m), (B, n)))
    err = (out[:, : m * n].reshape(batch, m, n) - torch.matmul(a, b.transpose(1, 2))).abs()
    bound = torch.matmul(a.abs(), b.abs().transpose(1, 2))
    assert bool((err <= 4 * (k + 2) * 2.0 ** -24 * bound).all())
