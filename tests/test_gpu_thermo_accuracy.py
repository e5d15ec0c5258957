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
