"""The strip kernel of the pair schedule (amlbm_step_strip.cu, the library's choice for the
FP32-arithmetic forms) against the fused schedule, bit for bit: lattices that are one
strip wrapping around the period (up to 64 columns), that are just wider, that end in a
ragged strip, strips shorter and taller than the lattice, both walls and forcings, and
lattices with different options in one batch; and the packed arithmetic it stands on,
against the scalar operations."""
import os
import subprocess

import numpy as np
import pytest

from paper_1310_1871_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1310_1871_gb300 import amlbm, build  # noqa: E402

FORMS = [("f32", dict()), ("f32", dict(wall="noslip", gz=1e-4, forcing="guo")), ("f32", dict(shift="equilibrium")),
         ("f16", dict()), ("f16", dict(shift="equilibrium")), ("bf16", dict()), ("bf16", dict(shift="equilibrium")),
         ("f16", dict(rounding="stochastic", axisym=False))]


def run(specs, storage, steps, **how):
    b = amlbm.Batch(specs, storage=storage, **how)
    for k, s in enumerate(specs):
        b.init_fields(k, *I.noisy(s.Nz, s.Nr, seed=k + s.Nz, base=0.9, amp=0.02))
    b.step(steps)
    out = [x for k in range(len(specs)) for x in (b.read_f(k), *b.read(k))]
    kind = (b.schedule, b.tile)
    b.close()
    return out, kind


@pytest.mark.parametrize("storage,kw", FORMS)
@pytest.mark.parametrize("Nz,Nr", [(2, 4), (6, 5), (62, 9), (64, 33), (66, 12), (96, 4), (98, 61), (190, 130)])
def test_strips_equal_fused_bitwise(Nz, Nr, storage, kw):
    spec = [amlbm.InstanceSpec(Nz, Nr, 0.9, -4.9, **kw)]
    ref, _ = run(spec, storage, 20, tile=(32, 8), schedule="fused")
    for rows in (2, 6, 18, 66):
        got, kind = run(spec, storage, 20, tile=(48, rows), schedule="pair")
        for a, b in zip(ref, got):
            assert np.array_equal(a, b), (kind, np.abs(a - b).max())


@pytest.mark.parametrize("kw", [dict(), dict(wall="noslip", gz=1e-4, forcing="guo"), dict(shift="equilibrium"),
                                dict(axisym=False)])
@pytest.mark.parametrize("Nz,Nr", [(1, 8), (3, 5), (47, 9), (49, 4), (63, 33), (65, 20), (97, 61), (255, 65)])
def test_odd_widths_equal_fused_bitwise(Nz, Nr, kw):
    """FP32 lattices of odd width, alone and beside even ones (among them one that is a
    single strip): the library's own choice for batches of some size (the last lattice); a
    requested pair schedule refuses them."""
    odd, large = amlbm.InstanceSpec(Nz, Nr, 0.9, -4.9, **kw), amlbm.InstanceSpec(512, 160, 0.9, -4.9, **kw)
    for specs in ([odd, large], [amlbm.InstanceSpec(64, 12, 0.9, -4.9), odd, amlbm.InstanceSpec(150, 31, 1.0, -5.0), large]):
        ref, _ = run(specs, "f32", 20, tile=(32, 8), schedule="fused")
        got, kind = run(specs, "f32", 20)
        assert kind[0] == "pair" and kind[1][0] == 48
        for a, b in zip(ref, got):
            assert np.array_equal(a, b), (kind, np.abs(a - b).max())
    with pytest.raises(amlbm.AmlbmError):
        amlbm.Batch([odd], storage="f32", tile=(48, 6), schedule="pair")


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
def test_strips_of_mixed_lattices_equal_fused_bitwise(storage):
    """Different sizes, walls, forcings and shifts in one batch (the kernel that branches on
    the options), and a uniform batch large enough for several rounds of strips."""
    mixed = [amlbm.InstanceSpec(40, 20, 0.9, -5.0), amlbm.InstanceSpec(130, 33, 1.0, -4.8, wall="noslip"),
             amlbm.InstanceSpec(66, 47, 0.8, -5.0, forcing="guo"), amlbm.InstanceSpec(64, 9, 1.1, -4.9, axisym=False),
             amlbm.InstanceSpec(100, 50, 0.9, -5.0, shift="equilibrium"), amlbm.InstanceSpec(512, 160, 0.9, -5.0)]
    many = [amlbm.InstanceSpec(2 * (30 + 7 * k % 90), 20 + 11 * k % 101, 0.9, -4.9) for k in range(120)]
    for specs in (mixed, many):
        ref, _ = run(specs, storage, 10, tile=(26, 16), schedule="fused")
        got, kind = run(specs, storage, 10)
        assert kind[0] == "pair" and kind[1][0] == 48
        for a, b in zip(ref, got):
            assert np.array_equal(a, b), kind


def test_strip_heights():
    """Every height the library may choose is accepted, others are refused."""
    spec = [amlbm.InstanceSpec(64, 32, 0.9, -5.0)]
    for rows in (2, 6, 18, 22, 254, 1022):
        amlbm.Batch(spec, storage="f32", tile=(48, rows), schedule="pair").close()
    for rows in (1, 4, 24, 1026):
        with pytest.raises(amlbm.AmlbmError) as e:
            amlbm.Batch(spec, storage="f32", tile=(48, rows), schedule="pair")
        assert e.value.code == amlbm.EINVAL


def test_packed_arithmetic_rounds_as_scalar(tmp_path):
    exe = str(tmp_path / "packed_check")
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "packed_check.cu")
    subprocess.run([build._nvcc(), *build.ARCH, "-O3", "-std=c++17", "-fmad=false", "-I", build.INCLUDE, "-I",
                    build.CSRC, src, "-o", exe], check=True, capture_output=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout + r.stderr
