"""The page-locked blocks behind the diagnostics, the read-back and the whole-batch
initialisation: fields larger than a block and missing fields, more batches and threads at
once than blocks are kept, and a call that fails, against the device's own arrays."""
import ctypes
import threading

import numpy as np
import pytest

from paper_1310_1871_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1310_1871_gb300 import amlbm  # noqa: E402


@pytest.mark.parametrize("storage", ["f64", "f32"])
@pytest.mark.parametrize("Nz,Nr", [(5, 4), (208, 210), (420, 331)])
def test_read_is_the_state(Nz, Nr, storage):
    """rho and j of the populations themselves, on both sides of one block (2^20 bytes)."""
    b = amlbm.Batch([amlbm.InstanceSpec(Nz, Nr, 0.9, 0.0, axisym=False)], storage=storage)
    b.init_fields(0, *I.noisy(Nz, Nr, seed=Nz, base=0.9, amp=0.02))
    f = b.read_f(0)
    rho, uz, ur = b.read(0)
    cz = np.array([0, 1, 0, -1, 0, 1, -1, -1, 1.0])[:, None, None]
    tol = 1e-14 if storage == "f64" else 1e-6  # nine terms of at most 1, rounded to 53 or 24 bits
    assert np.abs(f.sum(0) - rho).max() < 9 * tol
    assert np.abs((cz * f).sum(0) / rho - uz).max() < 9 * tol
    one = np.empty_like(ur)
    p = lambda a: a.ctypes.data_as(ctypes.POINTER(ctypes.c_double))
    assert b.lib.amlbm_batch_read(b.h, 0, None, None, p(one), None) == 0
    assert np.array_equal(one, ur)
    b.close()


def test_threads_and_failed_calls():
    """Twelve threads, each with its own stream and lattices of its own values."""
    errors = []

    def work(i):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                specs = [amlbm.InstanceSpec(40 + i, 20, 1.0, 0.0, axisym=False)] * 2
                b = amlbm.Batch(specs, storage="f32", stream=torch.cuda.current_stream())
                for turn in range(20):
                    v = 0.5 + 0.01 * i + 0.001 * turn
                    n = b.sites
                    b.init_all(np.full(n, v, np.float32))
                    with pytest.raises(amlbm.AmlbmError):
                        b.init_all(np.full(n, -1.0, np.float32))
                    b.step(2)
                    d = b.diagnostics_all(as_array=True)
                    want = v * specs[0].Nz * 20
                    assert abs(d[1, 0] - want) < 1e-5 * want and abs(b.diagnostics(0)["mass2d"] - want) < 1e-5 * want
                    assert np.abs(b.read(1)[0] - v).max() < 1e-6
                b.close()
        except BaseException as e:  # noqa: BLE001
            errors.append(e)

    t = [threading.Thread(target=work, args=(i,)) for i in range(12)]
    [x.start() for x in t]
    [x.join() for x in t]
    assert not errors, errors[0]
