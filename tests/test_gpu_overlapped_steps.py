"""Lanczos step loop: launches that overlap the end of the one before give the coefficients of launches kept apart.

While profiling is on, events stand between the kernels of a step and the loop is a CUDA graph of separate launches; the
arithmetic is the same, so the coefficients are equal bit by bit.
"""
import numpy as np
import pytest

from gpu_common import ftlm, product_group, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,two_s,two_M,irreps,R", [("icosahedron", 3, 2, None, 8), ("icosahedron", 3, 2, [8], 1),
                                                       ("icosahedron", 3, 2, [3], 4), ("cuboctahedron", 2, 0, None, 24)])
@pytest.mark.parametrize("table", [False, True])
def test_overlapped_steps_match_separate_ones(name, two_s, two_M, irreps, R, table):
    torch_cuda()
    F = ftlm()
    g = product_group(name)
    sec = F.ftlm_build_sector(g, two_s, two_M)
    ids = irreps or list(range(len(F.ftlm_group_info(g)["dims"])))
    mb = F.ftlm_build_multiblock(sec, ids)
    if table:
        F.ftlm_sector_build_entries(sec)
    for dt in (F.F32, F.F16, F.F64):
        a0, b0, s0 = F.ftlm_lanczos_multi(mb, dt, R, 10, 3, ids, F.GAUSS)
        F.ftlm_profile_enable(True)
        try:
            a1, b1, s1 = F.ftlm_lanczos_multi(mb, dt, R, 10, 3, ids, F.GAUSS)
        finally:
            F.ftlm_profile_enable(False)
        assert np.array_equal(s0, s1) and np.array_equal(a0, a1) and np.array_equal(b0, b1), dt
