"""Products of a known form (wide or narrow tiles; asserted) against the plain
definition, every batch compared: plain, bulk and scattered stores, split K."""
import json

import pytest

pytestmark = pytest.mark.gpu

TOL = {"tf32x3": 2.0 ** -18, "bf16x3": 2.0 ** -14, "fp16x3": 2.0 ** -18}


# wide in every precision: odd N (plain stores; 97 and 193 columns leave one of a
# tile's halves nearly empty), an odd number of 8-column chunks (bulk stores),
# split K with and without 8-column partials, more tiles than CTAs
WIDE = [(300, 256, 255, 40), (600, 128, 97, 40), (200, 256, 193, 40), (10, 2432, 257, 132), (800, 128, 72, 64),
        (400, 256, 136, 64), (300, 256, 200, 200), (1, 2432, 256, 8192), (1, 4864, 127, 8192)]
# narrow in BF16 and TF32: the last column tile nearly empty, rows of C off 32 bytes
NARROW = [(24, 2048, 130, 32), (16, 1024, 490, 16), (40, 1024, 161, 20)]


@pytest.mark.parametrize("pair", [0, 1], ids=["single", "pairs"])
@pytest.mark.parametrize("prec", sorted(TOL))
@pytest.mark.parametrize("shape", WIDE + NARROW)
def test_product(prec, shape, pair):
    import torch
    import paper_1907_11217_gb300 as tz
    batch, m, n, k = shape
    form = tz.tz_debug_tc_form(prec, batch, m, n, k, pair=pair)
    assert form["wide"] == (shape in WIDE or prec == "fp16x3")
    if pair and form["ctas"] == 1:
        pytest.skip("no pairs for this shape")
    g = torch.Generator(device="cuda").manual_seed(m + 3 * n + 7 * k)
    A, B = (torch.randn(batch, r, k, 2, device="cuda", generator=g) for r in (m, n))
    C = torch.full((batch, m, n, 2), float("nan"), device="cuda")
    scratch = torch.empty(tz.tz_op_cgemm_scratch_bytes(prec, batch, m, n, k), dtype=torch.uint8, device="cuda")
    tz.tz_tune_tc_pairs(pair)
    try:
        tz.tz_op_cgemm(prec, batch, m, n, k, A, m * k, B, n * k, C, m * n, scratch=scratch)
    finally:
        tz.tz_tune_tc_pairs(-1)
    tz.tz_op_cgemm_status(prec, scratch)
    a, b = (torch.view_as_complex(x.double()) for x in (A, B))
    bound = torch.matmul(a.abs(), b.abs().transpose(1, 2))
    err = (torch.view_as_complex(C.double()) - torch.matmul(a, b.transpose(1, 2))).abs()
    assert bool((err <= (TOL[prec] + 4 * (k + 2) * 2.0 ** -24) * bound).all()), float((err / bound).max())


@pytest.mark.parametrize("prec", ["tf32x3", "fp16x3"])
def test_scattered_wide_product(prec):
    """5x6 depth 1+24+1, 256 bitstrings a group: a wide product (batch 8, 4096 x
    128 x 32) that writes through its scatter map."""
    import paper_1907_11217_gb300 as tz
    import tz_inputs as ti
    from tests import gpu_util as gu
    spec = gu.grid_spec(5, 6, 24, 4)
    bits = ti.random_bitstrings(30, 256, 9)
    amps = {}
    for p in ("c128", prec):
        plan, *_ = gu.make_plan(tz, spec, batch_log2=8, log2_max=26, precision=p, restarts=16, max_bitstrings=256,
                                small_log2=8)
        amps[p] = tz.tz_contract_amplitudes(plan, bits)
    steps = json.loads(plan.describe())["steps"]
    assert any(s["tc"] and not s["row_major"] and
               tz.tz_debug_tc_form(prec, s["batch"], s["M"], s["N"], s["K"], scatter=True)["wide"] for s in steps)
    assert gu.rel_err(amps[prec], amps["c128"], 30) <= 1e-5
