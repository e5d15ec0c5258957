"""A set's Lanczos coefficients do not depend on the sets it runs with: partial sums are added in the order of the set's
own tiles, so a mix gives the bits of each set alone."""
from __future__ import annotations

import numpy as np
import pytest

from gpu_common import ftlm, product_group

pytestmark = pytest.mark.gpu


def _mix_equals_alone(F, sets, dtype, R, n_steps):
    K = len(F.ftlm_multiblock_info(sets[0])["dims"])
    ids = np.arange(len(sets) * K).reshape(len(sets), K)
    mix = F.ftlm_lanczos_sets(sets, dtype, R, n_steps, 7, ids)
    for i, mb in enumerate(sets):
        alone = F.ftlm_lanczos_sets([mb], dtype, R, n_steps, 7, ids[i:i + 1])
        for u, v in zip(mix, alone):
            assert np.array_equal(u[i], v[0]), i


@pytest.mark.parametrize("name,two_s,Ms,irreps,R", [("icosidodecahedron", 1, (10, 8), (8,), 1),
                                                    ("icosidodecahedron", 1, (12, 8, 10), (2,), 4),
                                                    ("icosahedron", 3, (6, 2, 0), tuple(range(10)), 8),
                                                    ("icosahedron", 3, (2, 0), tuple(range(10)), 3)])
@pytest.mark.parametrize("dtype", ["F64", "F32", "F16"])
def test_more_tiles_than_ctas(name, two_s, Ms, irreps, R, dtype):
    F = ftlm()
    g = product_group(name)
    secs = [F.ftlm_build_sector(g, two_s, m) for m in Ms]
    for sec in secs:
        F.ftlm_sector_build_entries(sec)
    sets = [F.ftlm_build_multiblock(sec, list(irreps)) for sec in secs]
    _mix_equals_alone(F, sets, getattr(F, dtype), R, 4)


@pytest.mark.parametrize("entries", [None, 1])
@pytest.mark.parametrize("dtype", ["F64", "F32", "F16"])
def test_a_large_part_leaves_the_others_their_tables(dtype, entries):
    """At four chains of dimension 3 the sector of 1.2e5 representatives has its flips searched once a call, those of
    2.5e5 and 4.6e5 (64 MB and twice the vectors are less than their tables) search in every step; with an entry
    table on one of them, too."""
    F = ftlm()
    g = product_group("icosidodecahedron")
    secs = [F.ftlm_build_sector(g, 1, m) for m in (8, 12, 10)]
    if entries is not None:
        F.ftlm_sector_build_entries(secs[entries])
    _mix_equals_alone(F, [F.ftlm_build_multiblock(sec, [2]) for sec in secs], getattr(F, dtype), 4, 4)
