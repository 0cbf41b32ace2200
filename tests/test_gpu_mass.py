"""The FP64 forms keep the mass of a closed planar lattice to rounding noise over long runs."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1310_1871_gb300 import amlbm  # noqa: E402


@pytest.mark.parametrize("kw", [dict(), dict(tile=(16, 8), schedule="split"), dict(tile=(32, 8), schedule="split"),
                                dict(tile=(32, 8), schedule="fused"), dict(tile=(32, 8), schedule="pair")])
@pytest.mark.parametrize("tau,G,opts", [(1.0, -5.0, {}), (0.65, -5.0, {}), (1.2, -4.8, dict(wall="noslip"))])
def test_mass_of_a_drop_is_kept(tau, G, opts, kw):
    """A site's step changes its mass by the rounding of one sum, at most about 2^-53 of it.
    Were every one of 20,000 steps to repeat the same roundings at each of the 2048 sites,
    signs at random, the total would move by 20,000 2^-53 / sqrt(2048) = 5e-14: held to 1e-13.
    (Factors 1 - 1/tau and 1/(9 tau) that do not sum to one move it by 1e-12.)"""
    Nz, Nr, steps = 64, 32, 20000
    z, r = np.arange(Nz)[None, :] - Nz / 2, np.arange(Nr)[:, None] + 0.5
    rho = 0.16 + 0.5 * (1.93 - 0.16) * (1.0 - np.tanh((np.hypot(z, r) - 12.0) / 2.0))
    b = amlbm.Batch([amlbm.InstanceSpec(Nz, Nr, tau, G, axisym=False, **opts)], storage="f64", **kw)
    b.init_fields(0, rho)
    m0 = math.fsum(b.read_f(0).ravel())
    b.step(steps)
    m = math.fsum(b.read_f(0).ravel())
    b.close()
    assert abs(m - m0) <= 1e-13 * m0
