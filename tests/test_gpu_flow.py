"""Two-right-hand-sides-per-lane table kernel and the search path that feeds it: every lane split (B = 6..32, even),
sets of I_h, O_h and T_d, spin-flip blocks with both signs, more flips per representative than the two prefetched
rounds, lane-copied gathers, FP16 storage, and Lanczos sets with and without the flips searched once."""
from __future__ import annotations

import os

import numpy as np
import pytest

from gpu_common import ftlm, product_group, torch_cuda
from oracle.basis import BlockBasis, SectorBasis
from oracle.group import Group
from test_gpu_packed import _packed_hv, _setup
from workloads import cluster, clusters, rand_block_vectors

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,two_s,two_M", [("icosahedron", 1, 2), ("icosahedron", 3, 20), ("cuboctahedron", 2, 10),
                                              ("tetrahedron", 5, 2), ("tetrahedron", 1, 0)])
def test_every_lane_split_matches_oracle(name, two_s, two_M):
    """FP32 bar of the packed H·v (3e-6 of the largest output), searched and from the table, bitwise alike."""
    torch = torch_cuda()
    F, og, sec, mb = _setup(name, two_s, two_M)
    bonds = cluster(name).bonds
    dims = F.ftlm_multiblock_info(mb)["dims"]
    osec = SectorBasis(og, two_s, two_M)
    blocks = [BlockBasis(osec, k).with_hamiltonian(bonds) if d else None for k, d in enumerate(dims)]
    widths = (6, 8, 10, 14, 16, 18, 24, 26, 30, 32)
    found = {}
    for table in (False, True):
        if table:
            F.ftlm_sector_build_entries(sec)
        for B in widths:
            xs = [rand_block_vectors(d, B, seed=7 * k + B) for k, d in enumerate(dims)]
            ys, xp, yp = _packed_hv(F, torch, mb, dims, xs, B, F.F32)
            if table:
                assert torch.equal(found[B], yp)
                os.environ["FTLM_HV_GATHER"] = "direct"
                try:
                    y2 = torch.full_like(yp, float("nan"))
                    F.ftlm_hv_packed(mb, F.F32, B, xp, y2)
                finally:
                    del os.environ["FTLM_HV_GATHER"]
                assert torch.equal(yp, y2)
                # FP16 storage of the same vectors: FP32 arithmetic, one rounding of each output
                xh = xp.half()
                yh, yf = torch.empty_like(xh), torch.empty_like(xp)
                F.ftlm_hv_packed(mb, F.F16, B, xh, yh)
                F.ftlm_hv_packed(mb, F.F32, B, xh.float(), yf)
                assert float((yh.double() - yf.double()).abs().max()) <= 2.0 ** -11 * float(yf.abs().max())
                continue
            found[B] = yp.clone()
            for k, d in enumerate(dims):
                if d:
                    ref = blocks[k].hv(xs[k])
                    assert np.abs(ys[k] - ref).max() <= 3e-6 * (np.abs(ref).max() + 1e-300), (B, k)


def test_spin_flip_sets():
    """G x Z_2 at M = 0: the ten Gamma- blocks in one set against each block alone (the single-block kernels)."""
    torch = torch_cuda()
    F = ftlm()
    g = product_group("icosahedron")
    sec = F.ftlm_build_sector_flip(g, 3)
    for z in (0, 1):
        mb = F.ftlm_build_multiblock(sec, list(range(z, 20, 2)))
        dims = F.ftlm_multiblock_info(mb)["dims"]
        xs = [rand_block_vectors(d, 8, seed=k) for k, d in enumerate(dims)]
        ys, _, _ = _packed_hv(F, torch, mb, dims, xs, 8, F.F32)
        for k, d in enumerate(dims):
            one = F.ftlm_build_block(sec, 2 * k + z)
            x = torch.from_numpy(xs[k]).cuda()
            y = torch.empty_like(x)
            F.ftlm_hv(one, F.F64, 8, x, y)
            ref = y.cpu().numpy()
            assert np.abs(ys[k] - ref).max() <= 3e-6 * (np.abs(ref).max() + 1e-300)


def test_many_flips_per_representative():
    """More than 64 flips of a representative (the rounds beyond the two prefetched ones): the cuboctahedron's sites
    under its rotations (irreps 1, 1, 2, 3, 3) at s = 1 with bonds to the three nearest shells (60 bonds)."""
    torch = torch_cuda()
    F = ftlm()
    V = clusters._cuboctahedron_vertices()
    gens = np.stack([clusters._perm_from_matrix(clusters._rot(ax, an), V)
                     for ax, an in (((0, 0, 1), np.pi / 2), ((1, 1, 1), 2 * np.pi / 3))])
    d2 = np.rint(((V[:, None] - V[None]) ** 2).sum(2)).astype(int)
    bonds = np.array([(i, j) for i in range(12) for j in range(i + 1, 12) if d2[i, j] in (2, 4, 6)], dtype=np.int32)
    og = Group(gens, bonds)
    g = F.ftlm_group_init(gens, bonds)
    F.ftlm_group_set_irreps(g, [ir.rho for ir in og.irreps])
    sec = F.ftlm_build_sector(g, 2, 0)
    labels, _ = F.ftlm_sector_export(sec)
    dig = (labels[:, None] >> (2 * np.arange(12, dtype=np.uint64))) & np.uint64(3)
    n = sum(((dig[:, i] < 2) & (dig[:, j] > 0)).astype(int) + ((dig[:, i] > 0) & (dig[:, j] < 2)) for i, j in bonds)
    assert len(bonds) == 60 and n.max() > 64
    mb = F.ftlm_build_multiblock(sec, list(range(5)))
    dims = F.ftlm_multiblock_info(mb)["dims"]
    xs = [rand_block_vectors(d, 8, seed=k) for k, d in enumerate(dims)]
    ys, _, _ = _packed_hv(F, torch, mb, dims, xs, 8, F.F32)
    osec = SectorBasis(og, 2, 0)
    for k in range(5):
        ref = BlockBasis(osec, k).with_hamiltonian(bonds).hv(xs[k])
        assert np.abs(ys[k] - ref).max() <= 3e-6 * np.abs(ref).max()


@pytest.mark.parametrize("R", [6, 24])
def test_lanczos_sets_fp32_on_searched_flips(R):
    """FP32 chains on two sectors: with the sectors' entry tables and with the call's own flips the table kernel
    does the same work, so the coefficients are equal; one sector with a table and one without mixes both."""
    F = ftlm()
    g = product_group("icosahedron")
    secs = [F.ftlm_build_sector(g, 3, m) for m in (8, 10)]
    sets = [F.ftlm_build_multiblock(s, list(range(10))) for s in secs]
    ids = np.arange(20).reshape(2, 10)
    ref = F.ftlm_lanczos_sets(sets, F.F32, R, 6, 4, ids)
    for k in range(2):
        F.ftlm_sector_build_entries(secs[k])
        got = F.ftlm_lanczos_sets(sets, F.F32, R, 6, 4, ids)
        for u, v in zip(ref, got):
            assert np.array_equal(u, v)
