"""Accuracy of the thermal pipeline against quadruple precision: the exponential over its range, the moments about the mean,
and the rotation of the eigensolve."""
from __future__ import annotations

import numpy as np
import pytest

from gpu_common import ftlm, torch_cuda

pytestmark = pytest.mark.gpu
U = 2.0 ** -53
LD = np.longdouble
needs_quad = pytest.mark.skipif(np.finfo(LD).nmant < 63, reason="no extended precision on this host")


@needs_quad
@pytest.mark.parametrize("x", [1.0, 0.7310585786300049, 3.0e-7, 123456.789])
def test_boltzmann_factor(x):
    """Two chains of one step: energy 0 with weight 1 and M^2 = 0, energy x with weight 2^-60 and M^2 = 1.  Z rounds to
    1, so chi = beta 2^-60 e^{-beta x} with one rounding beside the exponential's: 2 ulp of the table's exp2, half
    an ulp of the last addition and the polynomial's remainder, at most 8 units of 2^-53 in all."""
    torch = torch_cuda()
    F = ftlm()
    bx = np.concatenate([np.geomspace(1e-12, 1e-2, 200), np.linspace(0.01, 600.0, 20000)])
    T = x / bx
    beta = 1.0 / T
    d = lambda a, t=torch.float64: torch.tensor(a, dtype=t, device="cuda")
    out, E0 = torch.zeros(4 * len(T), dtype=torch.float64, device="cuda"), torch.zeros(1, dtype=torch.float64, device="cuda")
    F.ftlm_thermo_noalloc(2, 1, d([1, 1], torch.int32), d([0.0, x]), d([0.0, 0.0]), d([1.0, 2.0 ** -60]), d([0.0, 1.0]),
                          len(T), d(T), 1.0, out, E0)
    chi = out.cpu().numpy()[3 * len(T):]
    ref = LD(2.0) ** -60 * beta.astype(LD) * np.exp(-beta.astype(LD) * LD(x))
    assert float(np.abs(chi.astype(LD) / ref - 1).max()) <= 8 * U


@needs_quad
@pytest.mark.parametrize("n,low,scale,shift", [(10000, -4.5, 1.0, 0.0), (10000, -7.5, 1.0, 0.0), (10000, -7.5, 3e3, -2e4),
                                               (2500, -30.0, 1.0, 0.0), (40000, -3.0, 1e-3, 5.0)])
def test_moments(n, low, scale, shift):
    """Chains of one step, so energies and weights are the inputs: a normal distribution with one value far below it.
    Sums over 1e4 values in a tree carry a few units of 2^-53 (rms under 2), the Boltzmann factors' own errors
    average out and their common part cancels; 16 units for z, E's distance to the mean of the levels, C and chi.
    C is as good as if it were centred: the distance of the lowest level does not enter."""
    torch = torch_cuda()
    F = ftlm()
    rng = np.random.default_rng(n)
    th = rng.normal(size=n) * scale
    th[n // 3] = low * scale
    th += shift
    W, msq = rng.random(n) + 0.1, rng.random(n)
    T = scale * np.array([0.4, 0.7, 1.0, 2.0, 5.0, 20.0, 300.0])
    d = lambda a, t=torch.float64: torch.tensor(a, dtype=t, device="cuda")
    out, E0 = torch.zeros(4 * len(T), dtype=torch.float64, device="cuda"), torch.zeros(1, dtype=torch.float64, device="cuda")
    F.ftlm_thermo_noalloc(n, 1, d(np.ones(n), torch.int32), d(th), d(np.zeros(n)), d(W), d(msq), len(T), d(T), 1.0, out, E0)
    lnZ, E, C, chi = out.cpu().numpy().reshape(4, len(T))
    assert float(E0) == th.min()
    beta = (1.0 / T).astype(LD)[:, None]
    x = th.astype(LD) - LD(th.min())
    z = W.astype(LD) * np.exp(-beta * x)
    Z = z.sum(1)
    m = (z * x).sum(1) / Z
    var = (z * (x - m[:, None]) ** 2).sum(1) / Z
    b = beta[:, 0]
    assert np.all(np.abs(lnZ - (np.log(Z) - b * LD(th.min()))) <= 16 * U * (1 + np.abs(np.log(Z)) + np.abs(b * th.min())))
    assert np.all(np.abs(E - (LD(th.min()) + m)) <= 16 * U * (np.abs(th.min() + m) + np.sqrt(var)))
    assert np.all(np.abs(C / (b * b * var) - 1) <= 16 * U), (np.abs(C / (b * b * var) - 1) / U).astype(float)
    assert np.all(np.abs(chi / (b * (z * msq).sum(1) / Z) - 1) <= 16 * U)


@needs_quad
@pytest.mark.parametrize("scale", [1.0, 1e-140, 3e140])
def test_rotation_of_two_steps(scale):
    """Chains of two steps take one rotation (a second sweep only to find the off-diagonal negligible): its 1 / sqrt
    comes from the hardware's approximation and one step of a third-order iteration.  Shift, rotation and squares
    add up to at most 32 units of 2^-53 in the weights where the levels are no closer than a tenth of the matrix."""
    F = ftlm()
    rng = np.random.default_rng(2)
    n = 20000
    a = rng.normal(size=(n, 2))
    b = np.stack([10.0 ** rng.uniform(-6, 2, n) * rng.choice([-1.0, 1.0], n), np.zeros(n)], 1)
    half = (a[:, 1] - a[:, 0]) / 2
    keep = np.hypot(half, b[:, 0]) >= 0.05 * np.maximum(np.abs(a).max(1), np.abs(b[:, 0]))
    a, b = a[keep] * scale, b[keep] * scale
    th, w = F.ftlm_ritz(a, b, np.full(len(a), 2, dtype=np.int32))
    al, bl = a.astype(LD), b.astype(LD)[:, 0]
    h, mid = (al[:, 1] - al[:, 0]) / 2, (al[:, 1] + al[:, 0]) / 2
    r = np.sqrt((h / scale) ** 2 + (bl / scale) ** 2) * LD(scale)
    norm = np.abs(mid) + r
    assert np.all(np.abs(th[:, 0] - (mid - r)) <= 16 * U * norm) and np.all(np.abs(th[:, 1] - (mid + r)) <= 16 * U * norm)
    w0 = (1 + h / r) / 2  # weight of the lower level: cos^2, from the side that does not cancel
    w0 = np.where(h >= 0, w0, (bl / r) ** 2 / (2 * (1 - h / r)))
    w1 = np.where(h >= 0, (bl / r) ** 2 / (2 * (1 + h / r)), (1 - h / r) / 2)
    assert np.all(np.abs(w[:, 0] - w0) <= 32 * U) and np.all(np.abs(w[:, 1] - w1) <= 32 * U)
