"""dK/dnu near nu = 0, where it is a sum of t (1 - e^{-2 nu t}): its relative
error must not be that of 1 - e^{-2 nu t} taken from a rounded exponential."""
import numpy as np
import pytest

import paper_2502_00356_gb300 as bk

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nu", [1e-10, 1e-8, 1e-7, 1e-6, 1e-4, 1e-3, 0.02])
def test_relative_error_of_dk_dnu(nu):
    """Against the trapezoid rule with expm1 in FP64.  A node's t (1 - w) is held to
    2^-56 and 1 - w to a few 2^-63; for x <= 0.05 the nodes that matter have t > 1, so
    that 2 nu t^2 > 2 nu: 2^-56 / (2 nu) < 1e-17 / nu, twice over, besides the form's
    1e-12.  (The rounding of e^{-2 nu h} alone is up to 2^-54 / (2 nu h), 1e-16 / nu.)"""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    bk.build()
    x = torch.as_tensor(np.exp(np.linspace(np.log(1e-3), np.log(0.05), 4000)), device="cuda")
    v = torch.full_like(x, nu)
    got = bk.bk_eval_grad(x, v)
    t = torch.arange(0, 20 * 20, dtype=torch.float64, device="cuda") / 20
    f = torch.exp(-x[:, None] * torch.cosh(t) + nu * t) / 40.0
    want = (f * t * -torch.expm1(-2 * nu * t)).sum(1)  # (the integrand vanishes at t = 0)
    k = (f * (1 + torch.exp(-2 * nu * t))).sum(1) - f[:, 0]
    torch.cuda.synchronize()
    assert float((got[0] / k - 1).abs().max()) <= 1e-11
    assert float((got[2] / want - 1).abs().max()) <= 1e-11 + 2e-17 / nu
