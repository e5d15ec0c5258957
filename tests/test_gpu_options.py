"""Geometry options of the packed H·v on single blocks."""
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
