"""FP64 gradients against the same derivative in 80-bit arithmetic (the scheme of the CPU
oracle with long double in place of double, complex step; its values stand below rounded to
53 bits, since long double is not the same on every host)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1310_1871_gb300 import amlbm  # noqa: E402

AMPS = np.array([0.03, -0.02, 0.01, 0.015])
# Nz, Nr, T, tau, G, dJ/dG, dJ/dtau, dJ/da of the drop of radius 0.375 min(Nz / 2, Nr)
CASES = [
    (48, 24, 1, 0.9, -5.0, 7.287207838782537e-06, -7.463296027760339e-07,
     [0.1035144285134533, -0.00032542782415046243, 0.00398843343896098, -0.0009285226645135022]),
    (64, 32, 20, 0.8, -5.0, 0.00020061806756918086, 5.844321082722014e-05,
     [0.07882807821077015, -0.00041837249676060354, 0.003689868410222586, -0.0006081409604969421]),
    (48, 24, 40, 0.8, -5.1, 0.0018731157307112275, -3.956296109633351e-05,
     [0.04158843138396565, -0.0007068624085226245, 0.0026302165490535976, 3.950036347830678e-05]),
    (64, 24, 19, 0.9, -5.0, 0.0003586371607451852, 0.00023472106113556784,
     [0.08939125999771502, -0.0005801472283623699, 0.005145674312084932, -0.0005606626025458342]),
    (48, 36, 19, 0.9, -5.0, 0.00034556178777366974, 0.00021820643715379456,
     [0.08926866724914768, -0.0005781318760574343, 0.005123273432437946, -0.0005601053776730808]),
]


@pytest.mark.parametrize("Nz,Nr,T,tau,G,dG,dtau,da", CASES)
def test_gradients_to_twelve_digits(Nz, Nr, T, tau, G, dG, dtau, da):
    """The rounding of a population is 1e-16 of it and enters dJ/da, dJ/dG with a factor of some
    tens; dJ/dtau is a sum over sites and steps that leaves down to a hundredth of its terms.
    So 1e-13 and 1e-12.  (From sums over mu instead of its differences dJ/dtau is off by 5e-12
    to 1.4e-11 here.)"""
    lat = amlbm.Lattice(Nz, Nr, tau=tau, G=G, storage="f64")
    _, g, t, a = lat.adjoint(T, AMPS, Nz / 2, 0.375 * min(Nz / 2, Nr))
    lat.close()
    assert abs(t - dtau) <= 1e-12 * abs(dtau)
    assert abs(g - dG) <= 1e-13 * abs(dG)
    assert np.abs(a - da).max() <= 1e-13 * np.abs(da).max()
