"""The row kernel (amlbm_step_row.cu, the library's choice for small lattices of the
FP32-arithmetic forms) against the persistent fused kernel, bit for bit: lattices smaller
than a tile, of one tile, just larger and of many ragged ones, at the lowest, a middle and
the tallest tile, for every kind of boundary, forcing, source and shift; the read-back
against the pair schedule's; and the rule that chooses it."""
import numpy as np
import pytest

from paper_1310_1871_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1310_1871_gb300 import amlbm  # noqa: E402

KINDS = [dict(), dict(wall="noslip", gz=1e-4, forcing="guo"), dict(src="link"), dict(axisym=False, src="link"),
         dict(z_bc="noslip", r_lo="inlet", r_off=9.0, wall="outlet", rho_out=0.97, G=-3.0),
         dict(z_bc="noslip", wall="noslip", src="link"), dict(r_lo="inlet", r_off=3.0, wall="noslip", G=-3.0)]
FORMS = [("f32", {}), ("f32", dict(shift="equilibrium")), ("f16", {}), ("f16", dict(rounding="stochastic")),
         ("bf16", {}), ("bf16", dict(shift="equilibrium"))]


def run(spec, storage, steps=9, **how):
    b = amlbm.Batch([spec], storage=storage, **how)
    if spec.r_lo == "inlet":
        b.set_inlet(0, 1e-3 * np.sin(np.arange(spec.Nz)), 2e-3 + 1e-3 * np.cos(np.arange(spec.Nz)))
    b.init_fields(0, *I.noisy(spec.Nz, spec.Nr, seed=spec.Nz, base=0.9, amp=0.02))
    b.step(steps)
    out, kind = [b.read_f(0), *b.read(0)], (b.schedule, b.tile)
    b.close()
    return out, kind


def same(ref, got):
    assert np.isfinite(ref[0]).all()
    for a, b in zip(ref, got):
        assert np.array_equal(a, b), np.abs(a - b).max()


@pytest.mark.parametrize("storage,form", FORMS)
@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("Nz,Nr", [(4, 6), (5, 7), (26, 10), (27, 11), (53, 8), (131, 61)])
def test_rows_equal_fused_bitwise(Nz, Nr, kind, storage, form):
    kw = dict(kind, **form)
    spec = amlbm.InstanceSpec(Nz, Nr, 0.9, kw.pop("G", -4.9), **kw)
    ref, _ = run(spec, storage, tile=(32, 8), schedule="fused")
    for H in (4, 7, 10):
        same(ref, run(spec, storage, tile=(26, H), schedule="fused")[0])


@pytest.mark.parametrize("Nz,Nr", [(1, 4), (2, 5), (3, 30)])
def test_narrow_periodic_lattices(Nz, Nr):
    spec = amlbm.InstanceSpec(Nz, Nr, 0.9, -4.9)
    same(run(spec, "f32", tile=(32, 8), schedule="fused")[0], run(spec, "f32")[0])


def test_choice_in_16_bits_with_the_equilibrium_shift():
    for Nz, Nr, tile in ((768, 256, (64, 24)), (512, 160, (48, 2)), (700, 700, (48, 10))):
        spec = amlbm.InstanceSpec(Nz, Nr, 0.9, -4.9, shift="equilibrium")
        got, kind = run(spec, "f16", 4)
        assert kind == ("pair", tile)
        same(run(spec, "f16", 4, tile=(32, 8), schedule="fused")[0], got)


@pytest.mark.parametrize("Nz,Nr,kw,tile", [
    (64, 32, {}, ("fused", (26, 4))), (256, 128, {}, ("fused", (26, 9))), (520, 150, {}, ("fused", (26, 10))),
    (520, 152, {}, ("pair", None)), (780, 200, dict(src="link"), ("fused", (26, 10))),
    (780, 204, dict(src="link"), ("fused", (26, 16)))])
def test_choice_and_read_back(Nz, Nr, kw, tile):
    """The rule at its edges, and that the state and its read-back do not depend on it."""
    spec = amlbm.InstanceSpec(Nz, Nr, 0.9, -4.9, **kw)
    got, kind = run(spec, "f32")
    assert kind[0] == tile[0] and (tile[1] is None or kind[1] == tile[1]), kind
    other = dict(tile=(32, 8), schedule="fused") if kw else dict(tile=(64, 24), schedule="pair")
    same(run(spec, "f32", **other)[0], got)
