"""Rounding of the one-thread-per-representative kernel (FP32 vectors) against that of a warp per representative, which a
call inside a stream capture runs: sums of four flips instead of one chain over all of them."""
from __future__ import annotations

import pytest

from gpu_common import ftlm, product_group, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,two_s,two_M,irrep", [("icosahedron", 3, 0, 8), ("icosahedron", 3, 0, 2),
                                                    ("complete:11", 3, 1, 6), ("square:4x6", 1, 0, 0)])
@pytest.mark.parametrize("B", [1, 2, 4, 8, 12, 32])
def test_no_chain_over_all_flips(name, two_s, two_M, irrep, B):
    """F flips in a chain of sums of four round like (4 + F / 4) / 2 additions, in a warp of Q groups like
    F / 2Q + log2 Q; with the roundings both share the ratio of the errors stays below 1.25 (one chain over all
    flips: 1.4 to 1.6 at B = 4 and 8)."""
    torch = torch_cuda()
    F = ftlm()
    mb = F.ftlm_build_multiblock(F.ftlm_build_sector(product_group(name), two_s, two_M), [irrep])
    rows, d = F.ftlm_multiblock_packed_rows(mb), F.ftlm_multiblock_info(mb)["dims"][0]
    gen = torch.Generator("cuda").manual_seed(B)
    x = torch.empty(rows, B, device="cuda", dtype=torch.float64)
    F.ftlm_multiblock_pack(mb, F.F64, B, [torch.randn(d, B, device="cuda", generator=gen).double()], x)
    x = x.float()  # in the range of the projectors, up to rounding
    ref, y, yw = torch.empty(rows, B, device="cuda", dtype=torch.float64), torch.empty_like(x), torch.empty_like(x)
    F.ftlm_hv_packed(mb, F.F64, B, x.double(), ref)
    F.ftlm_hv_packed(mb, F.F32, B, x, y)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        F.ftlm_hv_packed(mb, F.F32, B, x, yw, stream=torch.cuda.current_stream())
    yw.fill_(float("nan"))
    graph.replay()
    torch.cuda.synchronize()
    assert float((y.double() - ref).norm()) <= 1.25 * float((yw.double() - ref).norm())
