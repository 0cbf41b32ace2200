"""amlbm_batch_diagnostics_all gives each instance what amlbm_batch_diagnostics gives it,
whatever the size of the batch (which decides how many sites a thread adds)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1310_1871_gb300 import amlbm  # noqa: E402


@pytest.mark.parametrize("storage", ["f32", "f64"])
@pytest.mark.parametrize("n", [10, 11, 21, 22])  # of 30,402 sites each: around 311,296 and 622,592 in all
def test_all_equals_single(storage, n):
    shapes = [(160, 190), (97, 61), (262, 90)] + [(162, 186)] * (n - 2)
    b = amlbm.Batch([amlbm.InstanceSpec(z, r, 1.0, -5.0) for z, r in shapes], storage=storage)
    rng = np.random.default_rng(n)
    for k, (z, r) in enumerate(shapes):
        u = 0.01 * rng.standard_normal((2, r, z))
        b.init_fields(k, 0.2 + 1.7 * rng.random((r, z)), u[0], u[1])
    par = [dict(zc=z / 2, R=0.4 * r, rho_l=1.9, rho_v=0.2) for z, r in shapes]
    every = b.diagnostics_all(par)
    for k, q in enumerate(par):
        assert b.diagnostics(k, **q) == every[k]
    b.close()
