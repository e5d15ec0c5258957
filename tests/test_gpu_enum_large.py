"""Enumeration of sectors with more live labels than fit 256 MB of findings: the 36-site ring at M = 0 under D_36 (9.1e9
labels), in its own order (7.8e8 live ones: findings kept) and with its sites renamed so that fewer prefixes die (1.0e9:
the write pass tests again over longer chunks)."""
from __future__ import annotations

import math

import numpy as np
import pytest

from gpu_common import ftlm, torch_cuda
from oracle.group import Group
from workloads import cluster

pytestmark = pytest.mark.gpu
RENAMED = [23, 5, 17, 1, 13, 3, 26, 35, 21, 20, 30, 31, 16, 7, 34, 29, 33, 10, 32, 0, 11, 27, 8, 12, 9, 15, 28, 22, 19, 24,
           6, 14, 18, 2, 4, 25]


@pytest.mark.parametrize("renamed", [False, True])
def test_ring36_orbits_cover_the_sector(renamed):
    F = ftlm()
    c = cluster("ring:36")
    q = np.array(RENAMED if renamed else range(36))
    qi = np.argsort(q)
    gens = np.stack([q[g[qi]] for g in c.gens]).astype(np.int32)
    bonds = q[np.asarray(c.bonds)].astype(np.int32)
    g = F.ftlm_group_init(gens, bonds)
    sec = F.ftlm_build_sector(g, 1, 0)
    if renamed:  # scratch of the build: 64 MB for the prefixes, 63 MB for counts and offsets (0.5 GB with findings)
        torch = torch_cuda()
        own = F.ftlm_sector_info(sec)["device_bytes"]
        del sec
        torch.cuda.empty_cache()
        fill = torch.empty(torch.cuda.mem_get_info()[0] - own - (256 << 20), dtype=torch.uint8, device="cuda")
        sec = F.ftlm_build_sector(g, 1, 0)
        del fill
        torch.cuda.empty_cache()
    labels, masks = F.ftlm_sector_export(sec)
    assert np.all(labels[1:] > labels[:-1])
    total = 0
    for i in range(0, len(labels), 1 << 24):  # orbit sizes add up to the sector: no label missing, none twice
        part = slice(i, i + (1 << 24))
        assert np.all(np.bitwise_count(labels[part]) == 18)
        total += int((72 // np.bitwise_count(masks[part]).astype(np.int64).sum(axis=1)).sum())
    assert total == math.comb(36, 18)
    rng = np.random.default_rng(1)
    pick = np.unique(np.concatenate([rng.integers(0, len(labels), 20000), np.arange(2000),
                                     np.nonzero(masks[:, 0] != 1)[0][:2000]]))
    lab, m = labels[pick], masks[pick]
    perms = Group(gens, bonds).perms
    assert len(perms) == 72
    for g, perm in enumerate(perms):
        img = np.zeros_like(lab)
        for k in range(36):
            img |= ((lab >> np.uint64(k)) & np.uint64(1)) << np.uint64(perm[k])
        assert np.all(img >= lab)
        assert np.array_equal(img == lab, ((m[:, g // 64] >> np.uint64(g % 64)) & np.uint64(1)).astype(bool))
