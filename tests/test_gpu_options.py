"""Geometry options and the autotuner of the packed H·v."""
from __future__ import annotations

import pytest

from gpu_common import ftlm, product_group, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("warps", ["2", "4", "6"])
def test_single_blocks_run_at_any_warp_count(warps, monkeypatch):
    """FTLM_HV_WARPS sets the warp kernels' CTAs; the one-thread kernel has one size and keeps it."""
    torch = torch_cuda()
    F = ftlm()
    sec = F.ftlm_build_sector(product_group("icosahedron"), 3, 14)
    mb = F.ftlm_build_multiblock(sec, [8])
    rows = F.ftlm_multiblock_packed_rows(mb)
    for table in (False, True):
        if table:
            F.ftlm_sector_build_entries(sec)
        for code, dt in ((F.F64, torch.float64), (F.F32, torch.float32), (F.F16, torch.float16)):
            for B in (1, 4):
                x = torch.randn(rows, B, device="cuda", generator=torch.Generator("cuda").manual_seed(B)).to(dt)
                ref, y = torch.empty_like(x), torch.empty_like(x)
                F.ftlm_hv_packed(mb, code, B, x, ref)
                with monkeypatch.context() as m:
                    m.setenv("FTLM_HV_WARPS", warps)
                    F.ftlm_hv_packed(mb, code, B, x, y)
                assert torch.equal(y, ref)


def test_autotuner_times_each_candidate_once():
    """The two-columns-per-lane kernel has no choice of rho tables or own-row prefetch: warps (8, 4), buffers (1 to 4) and
    tiles (three) are its candidates, and the default."""
    torch = torch_cuda()
    F = ftlm()
    sec = F.ftlm_build_sector(product_group("icosahedron"), 3, 14)
    F.ftlm_sector_build_entries(sec)
    mb = F.ftlm_build_multiblock(sec, list(range(10)))
    x = torch.randn(F.ftlm_multiblock_packed_rows(mb), 8, device="cuda")
    ref, y = torch.empty_like(x), torch.empty_like(x)
    F.ftlm_hv_packed(mb, F.F32, 8, x, ref)
    F.ftlm_set_autotune(1)
    try:
        F.ftlm_hv_packed(mb, F.F32, 8, x, y)
        report = F.ftlm_autotune_report().strip()
    finally:
        F.ftlm_set_autotune(-1)
    assert torch.equal(y, ref)
    assert len(report.splitlines()) == 1 and int(report.split("tried=")[1]) <= 25
