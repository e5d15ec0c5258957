"""Ritz pairs and thermal sums at the edges of their kernels: chain counts around one and several per CTA, step
counts up to 512 (the shared-memory limit of a CTA's chains), scales near the ends of the FP64 range, decoupled
matrices, and distributions so narrow that the centred second moment needs its own pass."""
from __future__ import annotations

import numpy as np
import pytest

from gpu_common import ftlm

pytestmark = pytest.mark.gpu
EPS = np.finfo(np.float64).eps


def _tri(a, b, m):
    return np.diag(a[:m]) + np.diag(b[:m - 1], 1) + np.diag(b[:m - 1], -1)


@pytest.mark.parametrize("n_chains,ld,scale", [(1, 1, 1.0), (3, 33, 1e200), (152, 60, 1.0), (153, 60, 1e-200),
                                               (700, 128, 1.0), (4900, 24, 30.0), (20, 512, 1.0)])
def test_ritz_edges(n_chains, ld, scale):
    F = ftlm()
    rng = np.random.default_rng(11)
    a = rng.normal(size=(n_chains, ld))
    b = 3.0 + rng.random((n_chains, ld))
    m = rng.integers(0, ld + 1, n_chains).astype(np.int32)
    m[0] = ld
    if n_chains > 2:
        b[1, ::3] = 0.0   # decoupled blocks
        a[2] = 1.0        # equal diagonal
    th, w = F.ftlm_ritz(a * scale, b * scale, m)
    for c in range(0, n_chains, max(1, n_chains // 40)):
        n = int(m[c])
        assert np.all(th[c, n:] == 0) and np.all(w[c, n:] == 0)
        if n == 0:
            continue
        T = _tri(a[c], b[c], n)
        x = th[c, :n] / scale
        tol = 16 * n * EPS * np.linalg.norm(T, 2)  # backward error of QL: a small multiple of n eps |T|
        assert np.all(np.diff(x) >= 0)
        assert np.abs(x - np.linalg.eigvalsh(T)).max() <= tol
        mom = np.eye(n)[0]
        for k in range(4):  # first-component moments (T^k)_00; each rotation perturbs them by a few eps
            ref = mom[0]
            assert abs(np.sum(w[c, :n] * x ** k) - ref) <= (k + 1) * 16 * n * EPS * np.linalg.norm(T, 2) ** k
            mom = T @ mom


@pytest.mark.parametrize("n_blocks,R,ld,shift", [(1, 1, 1, 0.0), (5, 3, 7, 0.0), (40, 24, 60, 0.0), (3, 2, 12, 1e7)])
def test_thermo_edges(n_blocks, R, ld, shift):
    """shift: every chain but one sits that far above the ground state, with almost all of the weight."""
    F = ftlm()
    rng = np.random.default_rng(5)
    blocks, th, W, msq = [], [], [], []
    for i in range(n_blocks):
        m = ld if i else max(1, ld // 2)
        a, b = rng.normal(size=(R, ld)), 1.0 + rng.random((R, ld))
        dim = 10 + i
        if i:
            a, dim = a + shift, dim * (10 ** 9 if shift else 1)
        blocks.append(dict(two_M=i % 3, d_gamma=1 + i % 5, dim=dim, alpha=a, beta=b, steps=np.full(R, m, dtype=np.int32)))
        for r in range(R):
            ev, U = np.linalg.eigh(_tri(a[r], b[r], m))
            th.append(ev)
            W.append((2.0 if i % 3 else 1.0) * (1 + i % 5) * dim / R * U[0] ** 2)
            msq.append(np.full(m, 0.25 * (i % 3) ** 2))
    th, W, msq = np.concatenate(th), np.concatenate(W), np.concatenate(msq)
    T = np.array([1.0, 10.0]) if not shift else np.array([1e7, 1e9])
    lnZ, E, C, chi, E0 = F.ftlm_thermo(blocks, T, 2.0)
    e0 = th.min()
    z = W * np.exp(-(th - e0) / T[:, None])
    Z = z.sum(1)
    x = (z * (th - e0)).sum(1) / Z
    c = (z * (th - e0 - x[:, None]) ** 2).sum(1) / Z / T ** 2
    # Ritz values carry n eps |T|: relative to T in the exponent, absolute in E; C is a ratio of such sums
    d = 64 * ld * EPS * max(1.0, np.abs(th).max())
    assert abs(E0 - e0) <= d
    assert np.all(np.abs(lnZ - (np.log(Z) - e0 / T)) <= 4 * d / T + 1e-13)
    assert np.all(np.abs(E - (e0 + x)) <= 4 * d * (1 + np.abs(th).max() / T))
    spread = np.sqrt((z * (th - e0 - x[:, None]) ** 2).sum(1) / Z)
    assert np.all(np.abs(C - c) <= 1e-12 * c + 16 * d * (spread + d) / T ** 2 * (1 + spread / T))
    assert np.all(np.abs(chi - 4.0 * (z * msq).sum(1) / Z / T) <= 1e-12 + 4 * d / T ** 2)
