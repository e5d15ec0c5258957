"""One-thread-per-representative kernel: every column split (B = 1, odd, 2 mod 4, 4 mod 4) and row size, padded rows
(dimension 3 and 5 in FP32 and FP16 above 2^18 representatives), several parts with padded rows, searched and from
the table."""
from __future__ import annotations

import numpy as np
import pytest

from gpu_common import ftlm, product_group, torch_cuda
from helpers import oracle_group
from oracle.basis import BlockBasis, SectorBasis
from workloads import cluster, rand_block_vectors

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,two_s,two_M,irreps", [("icosahedron", 3, 14, (1, 3, 7, 9)), ("petersen", 2, 2, (0, 6)),
                                                     ("complete:7", 1, 1, (0, 6)), ("icosahedron", 1, 0, (2, 8))])
def test_column_splits_match_oracle(name, two_s, two_M, irreps):
    torch = torch_cuda()
    F = ftlm()
    g, og, bonds = product_group(name), oracle_group(name), cluster(name).bonds
    sec, osec = F.ftlm_build_sector(g, two_s, two_M), SectorBasis(og, two_s, two_M)
    for ir in irreps:
        if ir >= len(og.irreps):
            continue
        ob = BlockBasis(osec, ir).with_hamiltonian(bonds)
        if ob.dim == 0:
            continue
        mb = F.ftlm_build_multiblock(sec, [ir])
        rows = F.ftlm_multiblock_packed_rows(mb)
        for B in (1, 2, 3, 4, 6, 7, 8, 12, 31, 32):
            X = rand_block_vectors(ob.dim, B, seed=ir + B)
            ref = ob.hv(X)
            x = torch.from_numpy(X).float().cuda()
            xp = torch.empty((rows, B), dtype=torch.float32, device="cuda")
            F.ftlm_multiblock_pack(mb, F.F32, B, [x], xp)
            out = []
            for table in (False, True):
                if table:
                    F.ftlm_sector_build_entries(sec)
                yp, y = torch.full_like(xp, float("nan")), torch.empty_like(x)
                F.ftlm_hv_packed(mb, F.F32, B, xp, yp)
                F.ftlm_basis_check(F.ftlm_multiblock_block(mb, 0))
                F.ftlm_multiblock_unpack(mb, F.F32, B, yp, [y])
                assert np.abs(y.cpu().numpy() - ref).max() <= 3e-6 * (np.abs(ref).max() + 1e-300), (ir, B, table)
                out.append(yp)
            F.ftlm_sector_free_entries(sec)
            assert torch.equal(out[0], out[1])
            # FP16 storage: FP32 arithmetic on the stored values, one rounding of each output
            xh = xp.half()
            yh, yf = torch.empty_like(xh), torch.empty_like(xp)
            F.ftlm_hv_packed(mb, F.F16, B, xh, yh)
            F.ftlm_hv_packed(mb, F.F32, B, xh.float(), yf)
            assert float((yh.double() - yf.double()).abs().max()) <= 2.0 ** -11 * float(yf.abs().max()) + 6e-8


@pytest.mark.parametrize("irrep", [2, 8])  # dimensions 3 and 5
def test_padded_rows(irrep):
    """4.6e5 representatives at B = 1: the padded copy is used; against FP64 (3e-6), FP16 against FP32 (one rounding)."""
    torch = torch_cuda()
    F = ftlm()
    sec = F.ftlm_build_sector(product_group("icosidodecahedron"), 1, 8)
    assert F.ftlm_sector_info(sec)["n_reps"] >= 1 << 18
    F.ftlm_sector_build_entries(sec)
    mb = F.ftlm_build_multiblock(sec, [irrep])
    rows = F.ftlm_multiblock_packed_rows(mb)
    x = torch.randn((rows, 1), device="cuda", generator=torch.Generator("cuda").manual_seed(2)).half()
    y64 = torch.empty((rows, 1), dtype=torch.float64, device="cuda")
    y32, y16 = torch.empty((rows, 1), device="cuda"), torch.empty_like(x)
    F.ftlm_hv_packed(mb, F.F64, 1, x.double(), y64)
    F.ftlm_hv_packed(mb, F.F32, 1, x.float(), y32)
    F.ftlm_hv_packed(mb, F.F16, 1, x, y16)
    scale = float(y64.abs().max())
    assert float((y32.double() - y64).abs().max()) <= 3e-6 * scale
    assert float((y16.double() - y32.double()).abs().max()) <= 2.0 ** -11 * scale


def test_padded_rows_in_parts():
    """Two sectors in one Lanczos launch at R = 1, each above 2^17 rows (together above the padded copy's bound)."""
    F = ftlm()
    g = product_group("icosidodecahedron")
    sets = []
    for m in (8, 10):
        sec = F.ftlm_build_sector(g, 1, m)
        F.ftlm_sector_build_entries(sec)
        sets.append(F.ftlm_build_multiblock(sec, [8]))
    ids = np.array([[3], [4]])
    a, b, st = F.ftlm_lanczos_sets(sets, F.F32, 1, 5, 7, ids)
    for i, mb in enumerate(sets):
        a1, b1, s1 = F.ftlm_lanczos_multi(mb, F.F32, 1, 5, 7, ids[i])
        assert np.array_equal(st[i], s1)
        assert np.allclose(a[i], a1, rtol=1e-12) and np.allclose(b[i], b1, rtol=1e-12)
