"""Rounding of the two-columns-per-lane kernel against that of the kernel with one column per lane, which x and y off a
pair of elements take: a flip's products are summed before they meet the accumulators in both."""
from __future__ import annotations

import pytest

from gpu_common import torch_cuda
from test_gpu_packed import _setup

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,two_s,two_M", [("icosahedron", 3, 0), ("icosahedron", 1, 0), ("cuboctahedron", 2, 0)])
@pytest.mark.parametrize("B", [8, 16, 24, 32])
def test_no_further_from_fp64_than_the_warp_kernel(name, two_s, two_M, B):
    """Norm-wise errors over a whole sector; the sums of a flip's groups meet in another order, worth a few percent."""
    torch = torch_cuda()
    F, og, sec, mb = _setup(name, two_s, two_M)
    F.ftlm_sector_build_entries(sec)
    rows = F.ftlm_multiblock_packed_rows(mb)
    dims = F.ftlm_multiblock_info(mb)["dims"]
    gen = torch.Generator("cuda").manual_seed(B)
    xs = [torch.randn(d, B, device="cuda", generator=gen).double() for d in dims]
    x = torch.empty(rows, B, device="cuda", dtype=torch.float64)
    F.ftlm_multiblock_pack(mb, F.F64, B, xs, x)  # in the range of the projectors
    x = x.float()
    ref = torch.empty(rows, B, device="cuda", dtype=torch.float64)
    F.ftlm_hv_packed(mb, F.F64, B, x.double(), ref)
    y = torch.empty_like(x)
    F.ftlm_hv_packed(mb, F.F32, B, x, y)
    flat = torch.empty(2 * rows * B + 2, device="cuda")
    x1, y1 = flat[1:1 + rows * B].view(rows, B), flat[1 + rows * B:1 + 2 * rows * B].view(rows, B)
    x1.copy_(x)
    F.ftlm_hv_packed(mb, F.F32, B, x1, y1)
    assert float((y.double() - ref).norm()) <= 1.06 * float((y1.double() - ref).norm())
