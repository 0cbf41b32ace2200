"""The adjoint's transposed stencils at the boundaries and at the edges of its tiles: the
gradient against the FP64 oracle's complex step on lattices whose sizes leave ragged
tiles in both directions, that are narrower than a stencil, with a free-slip and a
no-slip outer wall and in the planar model; and the amplitudes' map for low and high
Legendre degrees and counts on both sides of its kernels' sizes."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1310_1871_gb300 import amlbm  # noqa: E402


def check(Nz, Nr, T, ckpt, amps, l0=2, wall="freeslip", axisym=True):
    lat = amlbm.Lattice(Nz, Nr, tau=0.9, G=-5.0, storage="f64", wall=wall, axisym=axisym)
    R = 0.3 * min(Nz, 2 * Nr)
    J, dG, dtau, dA = lat.adjoint(T, amps, Nz / 2, R, l0=l0, ckpt_every=ckpt)
    lat.close()
    o = O.Oracle(Nz, Nr, tau=0.9, G=-5.0, axisym=int(axisym),
                 wall=O.WALL_NOSLIP if wall == "noslip" else O.WALL_FREESLIP)
    J_ref, g_ref = o.grad(T, Nz / 2, R, 2.0, 1.93, 0.16, np.asarray(amps, float), l0=l0)
    g = np.concatenate([[dG, dtau], dA])
    assert abs(J - J_ref) <= 1e-9 * abs(J_ref)
    # the complex step is exact to rounding; per component against the largest
    assert np.abs(g - g_ref).max() <= 1e-8 * np.abs(g_ref).max(), (g, g_ref)


@pytest.mark.parametrize("wall,axisym", [("freeslip", True), ("noslip", True), ("freeslip", False)])
@pytest.mark.parametrize("Nz,Nr", [(3, 6), (31, 9), (33, 4), (34, 13), (70, 21), (200, 50)])
def test_gradient_on_ragged_lattices(Nz, Nr, wall, axisym):
    check(Nz, Nr, 7, 3, [0.04, -0.02], wall=wall, axisym=axisym)


@pytest.mark.parametrize("n,l0", [(0, 2), (1, 0), (4, 2), (5, 1), (16, 2), (17, 3), (32, 2), (2, 70)])
def test_gradient_of_many_amplitudes(n, l0):
    amps = 0.01 * np.cos(np.arange(n) + 1.0)
    check(48, 24, 4, 2, amps, l0=l0)
