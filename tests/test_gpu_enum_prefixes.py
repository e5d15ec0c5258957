"""Enumeration under live prefixes (sectors above 2^17 labels): bit-exact tables for digit bases that are no power of
two, small groups (few dead prefixes), sums near the ends of the range, and the spin flip's signed elements."""
from __future__ import annotations

import numpy as np
import pytest

from gpu_common import ftlm, product_group
from helpers import masks_from_words, oracle_group, pack_labels
from oracle.basis import SectorBasis
from oracle.group import SpinFlipExtended

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,two_s,two_M", [("ring:9", 4, 0), ("ring:9", 4, 6), ("cuboctahedron", 2, -2),
                                              ("square:4x6", 1, 8), ("tetrahedron", 5, 0),
                                              ("cuboctahedron", 4, 22), ("icosahedron", 3, -10), ("ring:20", 1, 0)])
def test_sector_bit_exact(name, two_s, two_M):
    F = ftlm()
    og = oracle_group(name)
    sec = F.ftlm_build_sector(product_group(name), two_s, two_M)
    osec = SectorBasis(og, two_s, two_M)
    labels, masks = F.ftlm_sector_export(sec)
    assert np.array_equal(labels, pack_labels(osec.reps, og.n_sites, two_s))
    assert np.array_equal(masks, masks_from_words(osec.stab, og.order))


@pytest.mark.parametrize("name,two_s", [("square:4x6", 1), ("icosahedron", 3), ("cuboctahedron", 4)])
def test_flip_sector_bit_exact(name, two_s):
    F = ftlm()
    ext = SpinFlipExtended(oracle_group(name))
    sec = F.ftlm_build_sector_flip(product_group(name), two_s)
    osec = SectorBasis(ext, two_s, 0)
    labels, masks = F.ftlm_sector_export(sec)
    assert np.array_equal(labels, pack_labels(osec.reps, osec.n_sites, two_s))
    words = np.zeros_like(masks)
    words[:, :osec.stab.shape[1]] = osec.stab
    assert np.array_equal(masks, words)
