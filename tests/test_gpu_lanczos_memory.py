"""A Lanczos call that has room for its vectors and its sums runs, whether or not its flip tables and padded rows fit as well."""
from __future__ import annotations

import numpy as np
import pytest

from gpu_common import ftlm, product_group, torch_cuda

pytestmark = pytest.mark.gpu


def test_runs_without_room_for_the_flip_tables():
    """24 parts of ten blocks at 32 chains: vectors of 4.3 GB, flip tables of 168 MB, partial sums of the start vectors of
    75 MB.  With less than the sums left beside the tables the call does without tables: another kernel, so the
    coefficients agree to the rounding of FP32 (1e-5 of the largest after two steps)."""
    torch = torch_cuda()
    F = ftlm()
    sec = F.ftlm_build_sector(product_group("icosahedron"), 3, 0)
    n = F.ftlm_sector_info(sec)["n_reps"]
    P, R = 24, 32
    mb = F.ftlm_build_multiblock(sec, list(range(10)))
    ids = np.arange(10 * P).reshape(P, 10)
    run = lambda: F.ftlm_lanczos_sets([mb] * P, F.F32, R, 2, 5, ids)
    ref = run()
    vectors, tables = 3 * P * n * 32 * R * 4, P * n * 481
    for extra in (16, 32, 48, 64, 160):  # MB beside vectors and tables; then beside the vectors alone
        torch.cuda.empty_cache()
        left = vectors + (extra << 20) + (tables if extra < 100 else 0)
        fill = torch.empty(torch.cuda.mem_get_info()[0] - left, dtype=torch.uint8, device="cuda")
        try:
            got = run()
        finally:
            del fill
            torch.cuda.empty_cache()
        for u, v in zip(ref, got):
            assert np.abs(u - v).max() <= 1e-5 * np.abs(u).max(), extra
