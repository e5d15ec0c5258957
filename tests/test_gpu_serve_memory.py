"""Serving under a cap that holds a job's tables and vectors: memory that a job can do without never keeps it out."""
from __future__ import annotations

import numpy as np
import pytest

from gpu_common import ftlm, product_group, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cap_mb", [40, 400])
def test_job_runs_with_and_without_room_for_its_flip_table(cap_mb):
    """1.2e5 representatives at four chains of dimension 3: tables 7 MB, vectors 17 MB, flip table 57 MB."""
    torch_cuda()
    F = ftlm()
    g = product_group("icosidodecahedron")
    sec = F.ftlm_build_sector(g, 1, 12)
    table = F.ftlm_sector_info(sec)["n_reps"] * 481
    srv = F.Server(cap_bytes=cap_mb << 20, n_workers=1, max_parts=4)
    try:
        ids = [srv.submit(g, 1, 12, 2, 4, 8, 3, i, F.RADEMACHER, F.F32) for i in range(2)]
        res = [srv.wait(i, 120.0) for i in ids]
        peak = srv.stats()["peak_charged"]
    finally:
        srv.close()
    assert peak <= cap_mb << 20
    assert (peak > table) == (cap_mb == 400)
    blk = F.ftlm_build_block(sec, 2)
    for i, (info, a, b, st) in enumerate(res):
        a1, b1, s1 = F.ftlm_lanczos(blk, F.F32, 4, 8, 3, i, F.RADEMACHER)
        assert np.array_equal(st, s1)  # FP32 rounding in another order of sums, grown over eight steps
        assert np.abs(a - a1).max() <= 1e-4 * np.abs(a1).max() and np.abs(b - b1).max() <= 1e-4 * np.abs(b1).max()


def test_padded_rows_of_one_chain_are_charged():
    """Dimension 5 at one chain, FP32: 32 bytes a representative for the padded copy, beside 60 for the vectors."""
    torch_cuda()
    F = ftlm()
    g = product_group("icosidodecahedron")
    n = F.ftlm_sector_info(F.ftlm_build_sector(g, 1, 12))["n_reps"]
    srv = F.Server(cap_bytes=1 << 30)
    try:
        srv.wait(srv.submit(g, 1, 12, 8, 1, 4, 3, 0, F.RADEMACHER, F.F32), 120.0)
        stats = srv.stats()
    finally:
        srv.close()
    assert stats["peak_charged"] - stats["resident_table_bytes"] >= (60 + 481 + 32) * n
