"""The exponential of the thermal sums against quadruple precision over its whole range."""
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
