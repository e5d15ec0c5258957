"""Lanczos recurrence kernels at the edges of their thread layout: chain counts that make the CTA's rows x chains 1,
not a power of two, the full 1024 threads or more than one batch, and sets whose parts share or straddle CTAs."""
from __future__ import annotations

import numpy as np
import pytest

from gpu_common import ftlm, product_group
from helpers import oracle_group
from oracle.basis import BlockBasis, SectorBasis
from oracle.lanczos import lanczos, start_vectors
from workloads import cluster

pytestmark = pytest.mark.gpu
N_STEPS = 8


def _oracle(osec, ir, R, seed, bid, rows):
    ob = BlockBasis(osec, ir).with_hamiltonian(cluster("cuboctahedron").bonds)
    V0 = start_vectors(ob.dim, R, seed, bid)
    return [lanczos(ob.hv, V0[:, r], N_STEPS) for r in rows]


@pytest.mark.parametrize("R", [1, 3, 24, 31, 32, 33])
def test_lanczos_sets_match_oracle(R):
    """Three sectors in one launch; the first and last chain of a block of every dimension (FP64, 1e-10 as the
    parity bar of the coefficients)."""
    F = ftlm()
    g, og = product_group("cuboctahedron"), oracle_group("cuboctahedron")
    sectors = [0, 2, 12]  # 12: one digit sum short of the top, a few representatives
    secs = [F.ftlm_build_sector(g, 2, m) for m in sectors]
    irreps = list(range(len(og.irreps)))
    sets = [F.ftlm_build_multiblock(s, irreps) for s in secs]
    ids = np.arange(len(sets) * len(irreps)).reshape(len(sets), -1) + 5
    a, b, st = F.ftlm_lanczos_sets(sets, F.F64, R, N_STEPS, 9, ids)
    for p, m in enumerate(sectors[:2]):
        osec = SectorBasis(og, 2, m)
        for ir in (0, 4, 9):
            rows = sorted({0, R - 1})
            for r, (al, be) in zip(rows, _oracle(osec, ir, R, 9, int(ids[p, ir]), rows)):
                assert st[p, ir, r] == N_STEPS
                assert np.allclose(a[p, ir, r], al, rtol=1e-10, atol=1e-10)
                assert np.allclose(b[p, ir, r], be, rtol=1e-10, atol=1e-10)
    dims = F.ftlm_multiblock_info(sets[2])["dims"]
    assert all(st[2, k].max(initial=0) <= min(N_STEPS, dims[k]) for k in range(len(dims)))


@pytest.mark.parametrize("R", [1, 2, 7, 32])
def test_single_blocks_match_oracle(R):
    """Blocks of dimension 1 and 3 (rows x chains from 1 to 96), FP64 and FP32 vectors."""
    F = ftlm()
    g, og = product_group("cuboctahedron"), oracle_group("cuboctahedron")
    sec, osec = F.ftlm_build_sector(g, 2, 0), SectorBasis(og, 2, 0)
    for ir in (1, 8):
        blk = F.ftlm_build_block(sec, ir)
        rows = sorted({0, R - 1})
        ref = _oracle(osec, ir, R, 3, 17, rows)
        # FP32 vectors: 6e-8 rounding of every stored entry, eight steps, coefficients of order |H| = 24
        for dt, tol in ((F.F64, 1e-10), (F.F32, 5e-5)):
            a, b, _ = F.ftlm_lanczos(blk, dt, R, N_STEPS, 3, 17)
            for r, (al, be) in zip(rows, ref):
                assert np.allclose(a[r], al, rtol=tol, atol=tol)
                assert np.allclose(b[r], be, rtol=tol, atol=tol)
