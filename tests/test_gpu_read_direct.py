"""Reads of FP64 fields on both sides of the size from which they are copied straight into the
caller's arrays (10,240 sites), into pageable and page-locked arrays."""
import ctypes
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1310_1871_gb300 import amlbm  # noqa: E402


def batch(Nz, Nr):
    b = amlbm.Batch([amlbm.InstanceSpec(Nz, Nr, 0.9, 0.0, axisym=False)], storage="f64")
    rng = np.random.default_rng(Nz)
    b.init_fields(0, 1.0 + 0.1 * rng.random((Nr, Nz)), 0.01 * rng.random((Nr, Nz)), 0.01 * rng.random((Nr, Nz)))
    return b


def read(b, arrays):
    p = [None if a is None else a.ctypes.data_as(ctypes.POINTER(ctypes.c_double)) for a in arrays]
    assert b.lib.amlbm_batch_read(b.h, 0, *p, None) == 0


@pytest.mark.parametrize("Nz,Nr", [(128, 80), (129, 80), (300, 200)])
@pytest.mark.parametrize("locked", [False, True])
def test_fields(Nz, Nr, locked):
    b = batch(Nz, Nr)
    f = b.read_f(0)
    make = lambda: (torch.full((Nr, Nz), -1.0, dtype=torch.float64).pin_memory() if locked else
                    torch.full((Nr, Nz), -1.0, dtype=torch.float64)).numpy()
    rho, uz, ur = make(), make(), make()
    read(b, (rho, uz, ur))
    eps = 9 * 2.0 ** -52  # nine populations of at most 1, added in either order
    assert np.abs(f.sum(0) - rho).max() <= eps
    assert np.abs(rho * uz - (f[1] - f[3] + f[5] - f[6] - f[7] + f[8])).max() <= eps
    for q, whole in enumerate((rho, uz, ur)):
        one = [None, None, None]
        one[q] = make()
        read(b, one)
        assert np.array_equal(one[q], whole)
    b.close()


def test_large_read_takes_no_longer_than_copies():
    """Three fields of 2 M sites: at most four times the time of three plain copies of that
    size (the read-back kernel before them takes about as long; in pieces of 2^20 bytes it is 14)."""
    Nz, Nr = 2048, 1024
    b = batch(Nz, Nr)
    host = [torch.empty(Nr, Nz, dtype=torch.float64) for _ in range(3)]
    dev = torch.zeros(Nr, Nz, dtype=torch.float64, device="cuda")

    def best(call):
        t = []
        for _ in range(12):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            call()
            t.append(time.perf_counter() - t0)
        return min(t)

    plain = best(lambda: [h.copy_(dev) for h in host])
    fields = best(lambda: read(b, [h.numpy() for h in host]))
    b.close()
    assert fields <= 4.0 * plain
