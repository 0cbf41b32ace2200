"""The FP64 form's two-kernel step (amlbm_step_split64.cu), the library's own choice for
FP64, against the fused schedule: the same operations on the same values, so the
states must be bit-identical for every kind of lattice it takes (odd and ragged
sizes, walls, inlet and outlet rows, both forcings, both source discretisations) and
on every tile it chooses (8 x 4 and 16 x 8 with several threads per site, 32 x 8 and
32 x 16 with one), and so must rho and u of the read-back."""
import numpy as np
import pytest

from paper_1310_1871_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1310_1871_gb300 import amlbm  # noqa: E402

CASES = [dict(), dict(wall="noslip", gz=1e-4, forcing="guo"), dict(src="link"), dict(axisym=False, wall="noslip"),
         dict(z_bc="noslip", r_lo="inlet", r_off=9.0, wall="outlet", rho_out=0.97, G=-3.0),
         dict(z_bc="noslip", wall="noslip", src="link"), dict(r_lo="inlet", r_off=3.0, wall="noslip", G=-3.0)]


@pytest.mark.parametrize("case", CASES)
@pytest.mark.parametrize("Nz,Nr,tile", [(5, 6, (8, 4)), (33, 21, (8, 4)), (197, 97, (16, 8)), (255, 131, (32, 8)),
                                        (1026, 470, (32, 16))])
def test_split64_equals_fused_bitwise(Nz, Nr, tile, case):
    kw = dict(case)
    G = kw.pop("G", -4.9)
    spec = amlbm.InstanceSpec(Nz, Nr, 0.9, G, **kw)
    fl = I.noisy(Nz, Nr, seed=Nz, base=0.9, amp=0.02)
    out = []
    for args in (dict(tile=(32, 8), schedule="fused"), dict()):
        b = amlbm.Batch([spec], storage="f64", **args)
        if kw.get("r_lo") == "inlet":
            b.set_inlet(0, 1e-3 * np.sin(np.arange(Nz)), 2e-3 + 1e-3 * np.cos(np.arange(Nz)))
        b.init_fields(0, *fl)
        b.step(8)
        out.append([*b.read(0), b.read_f(0)])
        if not args:
            assert (b.schedule, b.tile) == ("split", tile)
        b.close()
    assert np.isfinite(out[0][3]).all()
    for x, y in zip(*out):
        assert np.array_equal(x, y), np.abs(x - y).max()
