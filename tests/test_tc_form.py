"""Which form a tensor-core product takes (host only): wide tiles or narrow."""
import pytest

import paper_1907_11217_gb300 as tz


# (batch, m, n, k), and whether BF16 / TF32 take wide tiles: a last column tile
# that is mostly empty, rows of C off 32 bytes with a short sum, a last wave that
# narrow tiles fill better; then whole tiles, long sums, large B, split K
@pytest.mark.parametrize("prec", ["tf32x3", "bf16x3"])
@pytest.mark.parametrize("shape,wide", [
    ((16, 4096, 130, 32), False), ((16, 4096, 160, 32), False), ((16, 4096, 426, 32), False),
    ((16, 4096, 490, 32), False), ((16, 4096, 1022, 16), False), ((3, 2048, 512, 64), False),
    ((2, 2048, 128, 1024), False), ((1, 8192, 64, 2048), False),
    ((16, 4096, 512, 32), True), ((16, 4096, 1000, 16), True), ((16, 4096, 130, 1024), True),
    ((8, 32768, 256, 512), True), ((1, 16384, 1024, 2048), True), ((300, 256, 129, 200), True),
    ((800, 128, 72, 64), True), ((1, 2432, 256, 8192), True)])
def test_wide_or_narrow(prec, shape, wide):
    assert tz.tz_debug_tc_form(prec, *shape)["wide"] == wide


def test_fp16_takes_wide_tiles_beyond_64_columns():
    for n in (65, 72, 128, 130, 426, 490):
        for batch, m, k in ((1, 128, 64), (16, 4096, 32), (2, 2048, 1024)):
            f = tz.tz_debug_tc_form("fp16x3", batch, m, n, k)
            assert f["wide"] and f["ctas"] == 1 and f["launches"] == 1 + 1 + (f["ksplit"] > 1)
    assert tz.tz_debug_tc_form("fp16x3", 16, 4096, 64, 32) == {"wide": False, "ctas": 1, "ksplit": 1, "launches": 3}


def test_pairs_and_split():
    form = tz.tz_debug_tc_form
    assert form("bf16x3", 16, 4096, 512, 32)["ctas"] == 2
    assert form("bf16x3", 16, 4096, 512, 32, pair=0)["ctas"] == 1
    assert form("fp16x3", 16, 4096, 512, 32, pair=1)["ctas"] == 2
    assert form("tf32x3", 129, 384, 512, 32, pair=1)["ctas"] == 1  # no whole 256-row tiles
    assert form("bf16x3", 1, 2432, 256, 8192)["ksplit"] > 1
    assert form("bf16x3", 1, 2432, 256, 8192, ksplit=1)["ksplit"] == 1
    assert form("bf16x3", 1, 2432, 256, 8192, scatter=True)["ksplit"] == 1
    with pytest.raises(tz.TzError):
        form("bf16x3", 1, 100, 128, 64)
    with pytest.raises(tz.TzError):
        form("c64", 1, 128, 128, 64)
