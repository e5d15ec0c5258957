"""Packed H·v on vectors that start on an odd element (views into a flat buffer): the kernel that moves rows in pairs of
elements is left for the one that moves single elements; searched, from the table, and with the autotuner's choices."""
from __future__ import annotations

import pytest

from gpu_common import torch_cuda
from test_gpu_packed import _setup

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tune", [False, True])
@pytest.mark.parametrize("name,two_s,two_M", [("icosahedron", 1, 2), ("cuboctahedron", 2, 10), ("tetrahedron", 5, 2)])
def test_shifted_vectors_match_aligned(name, two_s, two_M, tune):
    """Each result is within 3e-6 of the largest output of the exact one (FP32); FP16 adds one rounding of each."""
    torch = torch_cuda()
    F, og, sec, mb = _setup(name, two_s, two_M)
    rows = F.ftlm_multiblock_packed_rows(mb)
    gen = torch.Generator("cuda").manual_seed(3)
    F.ftlm_set_autotune(1 if tune else 0)
    try:
        for table in (False, True):
            if table:
                F.ftlm_sector_build_entries(sec)
            for B in (6, 8, 16, 24, 32):
                for dt, code, tol in ((torch.float32, F.F32, 6e-6), (torch.float16, F.F16, 6e-6 + 2.0 ** -10)):
                    x = torch.randn(rows, B, device="cuda", generator=gen).to(dt)
                    ref = torch.empty_like(x)
                    F.ftlm_hv_packed(mb, code, B, x, ref)
                    bound = tol * float(ref.abs().max())
                    for sx, sy in ((1, 0), (0, 1), (1, 1), (2, 3)):
                        xb = torch.empty(rows * B + 4, dtype=dt, device="cuda")
                        yb = torch.full((rows * B + 4,), 7.0, dtype=dt, device="cuda")
                        xs, ys = xb[sx:sx + rows * B].view(rows, B), yb[sy:sy + rows * B].view(rows, B)
                        xs.copy_(x)
                        F.ftlm_hv_packed(mb, code, B, xs, ys)
                        assert float((ys.double() - ref.double()).abs().max()) <= bound, (table, B, dt, sx, sy)
                        assert bool((yb[:sy] == 7).all()) and bool((yb[sy + rows * B:] == 7).all())
    finally:
        F.ftlm_set_autotune(-1)
