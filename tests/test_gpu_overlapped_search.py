"""Search path in FP32 arithmetic: the table kernel is launched while the build of its entries still runs.

Calls in a row without a synchronisation in between (the next build overwrites the workspace that the last
table kernel reads), on sectors from a few representatives to several runs of the workspace, on the default and on
another stream: every output must equal the table path's element by element (both sum in the same order).
"""
import pytest

from gpu_common import ftlm, product_group, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,two_s,two_M,irreps,B", [("icosahedron", 1, 0, None, 8), ("icosahedron", 3, 4, None, 6),
                                                       ("icosahedron", 3, 2, [9], 5), ("cuboctahedron", 2, 0, None, 24),
                                                       ("icosidodecahedron", 1, 0, None, 8)])
@pytest.mark.parametrize("side_stream", [False, True])
def test_back_to_back_searches_match_the_table(name, two_s, two_M, irreps, B, side_stream):
    torch = torch_cuda()
    F = ftlm()
    g = product_group(name)
    sec = F.ftlm_build_sector(g, two_s, two_M)
    mb = F.ftlm_build_multiblock(sec, irreps or list(range(len(F.ftlm_group_info(g)["dims"]))))
    rows = F.ftlm_multiblock_packed_rows(mb)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(5)
    for dt, tdt in ((F.F32, torch.float32), (F.F16, torch.float16)):
        xs = [torch.randn((rows, B), device="cuda", generator=gen).to(tdt) for _ in range(3)]
        ys = [torch.full_like(xs[0], float("nan")) for _ in range(6)]
        torch.cuda.synchronize()
        st = torch.cuda.Stream() if side_stream else torch.cuda.current_stream()
        with torch.cuda.stream(st):
            for i, y in enumerate(ys):
                F.ftlm_hv_packed(mb, dt, B, xs[i % 3], y, stream=st.cuda_stream)
        torch.cuda.synchronize()
        F.ftlm_sector_build_entries(sec)
        for i, y in enumerate(ys):
            want = torch.full_like(y, float("nan"))
            F.ftlm_hv_packed(mb, dt, B, xs[i % 3], want)
            torch.cuda.synchronize()
            assert torch.equal(y, want), (dt, i)
        F.ftlm_basis_check(F.ftlm_multiblock_block(mb, 0))
        F.ftlm_sector_free_entries(sec)
