"""Wide tensor-core product, row-major C written by bulk stores: a warp's 64
columns hold an odd number of 8-column chunks, so that its last store of a tile
and its first of the next use the same staging buffer. Several tiles a CTA,
short K (the stores of one tile run into the next), every batch compared."""
import pytest

pytestmark = pytest.mark.gpu

TOL = {"tf32x3": 2.0 ** -18, "bf16x3": 2.0 ** -14, "fp16x3": 2.0 ** -18}


# live columns of the two halves of the last column tile: 64 + 2, 64 + 8, 8,
# 18 (chunks 1), 64 + 24 (3), 40 (5), 64 + 50 (7)
@pytest.mark.parametrize("pairs", [0, 1], ids=["single", "pairs"])
@pytest.mark.parametrize("prec", sorted(TOL))
@pytest.mark.parametrize("batch,m,n,k", [(800, 128, 66, 4), (800, 128, 72, 32), (600, 256, 136, 16),
                                         (400, 256, 146, 32), (800, 256, 88, 8), (300, 512, 168, 36),
                                         (400, 512, 114, 64)])
def test_odd_chunks(pairs, prec, batch, m, n, k):
    import torch
    import paper_1907_11217_gb300 as tz
    if pairs and m % 256:
        pytest.skip("pairs take whole 256-row tiles")
    g = torch.Generator(device="cuda").manual_seed(m + 3 * n + 7 * k)
    A, B = (torch.randn(batch, r, k, 2, device="cuda", generator=g) for r in (m, n))
    C = torch.full((batch, m, n, 2), float("nan"), device="cuda")
    scratch = torch.empty(tz.tz_op_cgemm_scratch_bytes(prec, batch, m, n, k), dtype=torch.uint8, device="cuda")
    tz.tz_tune_tc_pairs(pairs)
    try:
        for _ in range(3):
            tz.tz_op_cgemm(prec, batch, m, n, k, A, m * k, B, n * k, C, m * n, scratch=scratch)
    finally:
        tz.tz_tune_tc_pairs(-1)
    tz.tz_op_cgemm_status(prec, scratch)
    a, b = (torch.view_as_complex(x.double()) for x in (A, B))
    ref = torch.matmul(a, b.transpose(1, 2))
    bound = torch.matmul(a.abs(), b.abs().transpose(1, 2))
    err = (torch.view_as_complex(C.double()) - ref).abs()
    assert bool((err <= (TOL[prec] + 4 * (k + 2) * 2.0 ** -24) * bound).all()), float((err / bound).max())
