"""The launch settings of the tensor-core products (L2 prefetch distance of A,
L2 priorities) on wide tiles: they change no result, whatever their value
(distances beyond a tile's k-blocks and beyond the product's last tile, split
K, pairs, bulk, plain and scattered stores)."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SHAPES = [(200, 256, 136, 36), (3, 256, 127, 260), (1, 512, 128, 8192)]


def results():
    """One product per precision, shape and form, as bytes."""
    import torch
    import paper_1907_11217_gb300 as tz
    out = []
    for batch, m, n, k in SHAPES:
        g = torch.Generator(device="cuda").manual_seed(k)
        A, B = (torch.randn(batch, r, k, 2, device="cuda", generator=g) for r in (m, n))
        for prec in ("tf32x3", "bf16x3", "fp16x3"):
            for pairs in (0, 1):
                C = torch.full((batch, m, n, 2), float("nan"), device="cuda")
                nb = tz.tz_op_cgemm_scratch_bytes(prec, batch, m, n, k)
                scratch = torch.empty(nb, dtype=torch.uint8, device="cuda")
                tz.tz_tune_tc_pairs(pairs)
                tz.tz_op_cgemm(prec, batch, m, n, k, A, m * k, B, n * k, C, m * n, scratch=scratch)
                tz.tz_tune_tc_pairs(-1)
                tz.tz_op_cgemm_status(prec, scratch)
                assert bool(torch.isfinite(C).all())
                out.append(C.cpu().numpy().tobytes())
    return out


def test_prefetch_distance():
    import paper_1907_11217_gb300 as tz
    try:
        tz.tz_tune_tc_prefetch(0)
        want = results()
        for d in (1, 7, 64):
            tz.tz_tune_tc_prefetch(d)
            assert results() == want, d
    finally:
        tz.tz_tune_tc_prefetch(-1)


def test_l2_priorities():
    """TZ_TC_L2 is read once per process: 0 (A evict first, C normal) against
    this process's setting."""
    import hashlib
    code = ("import hashlib, tests.test_gpu_tc_wide_settings as t\n"
            "print(hashlib.sha256(b''.join(t.results())).hexdigest())")
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, env=dict(os.environ, TZ_TC_L2="0"),
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    assert r.stdout.split()[-1] == hashlib.sha256(b"".join(results())).hexdigest()
