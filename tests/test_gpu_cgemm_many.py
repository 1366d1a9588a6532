"""A batch of more tiles than one grid has blocks (2^31 - 1): one operand and
one result for all (strides of zero), through the complex64 tiles."""
import pytest

pytestmark = pytest.mark.gpu


def test_more_tiles_than_blocks_of_a_grid():
    import torch
    import paper_1907_11217_gb300 as tz
    m, n, k = 1, 17, 1  # 32 x 32 tiles, one a block
    batch = 2 ** 31 + 5
    A, B, C = (torch.randn(s, 2, device="cuda") for s in (m * k, n * k, m * n))
    C.fill_(float("nan"))
    tz.tz_op_cgemm("c64", batch, m, n, k, A, 0, B, 0, C, 0)
    torch.cuda.synchronize()
    want = torch.view_as_complex(A)[:, None] * torch.view_as_complex(B)[None, :]
    torch.testing.assert_close(torch.view_as_complex(C), want.reshape(-1))
