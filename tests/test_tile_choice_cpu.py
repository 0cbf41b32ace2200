"""A schedule requested without a tile gets one of its own (no GPU: the tile is chosen and
checked before the workspace, which is too small here)."""
import ctypes

import pytest

from paper_1310_1871_gb300 import amlbm


def create(shapes, storage, schedule, tile=(0, 0), **kw):
    lib = amlbm.load()
    inst = amlbm.instances_c([amlbm.InstanceSpec(z, r, 1.0, -5.0, **kw) for z, r in shapes], storage)
    tune, h = amlbm.Tune(*tile, 0, amlbm.SCHEDULE[schedule]), ctypes.c_void_p()
    # an aligned device address that is never dereferenced, with too few bytes
    return lib.amlbm_batch_create(len(shapes), inst, ctypes.byref(tune), None, ctypes.c_void_p(1 << 20), 16,
                                  ctypes.byref(h))


BATCHES = [[(64, 32)], [(2, 4)], [(26, 10)] * 200, [(3648, 17)], [(512, 160)], [(1024, 512)],
           [(4 * k, 2 * k) for k in range(10, 61)]]


@pytest.mark.parametrize("storage", ["f64", "f32", "f16", "bf16"])
@pytest.mark.parametrize("schedule", ["fused", "split", "pair"])
@pytest.mark.parametrize("q", range(len(BATCHES)))
def test_schedule_without_a_tile(q, schedule, storage):
    assert create(BATCHES[q], storage, schedule) == amlbm.ENOMEM


@pytest.mark.parametrize("storage,kw", [("f64", {}), ("f32", {}), ("f16", dict(shift="equilibrium"))])
def test_what_a_schedule_cannot_take_is_still_refused(storage, kw):
    for schedule, extra in (("pair", dict(src="link")), ("split", dict(forcing="guo"))):
        for shapes in ([(64, 32)], [(1024, 512)]):
            assert create(shapes, storage, schedule, **extra, **kw) == amlbm.EINVAL
    assert create([(63, 32)], storage, "pair", **kw) == amlbm.EINVAL
    assert create([(64, 32)], storage, "fused", (128, 8), **kw) == amlbm.EINVAL


def test_own_choice_can_be_requested():
    """The FP64 kernels on a bounded lattice, strips on an odd width: refused as a request
    unless they are what the library takes by itself."""
    discs = dict(z_bc="noslip", r_lo="inlet", r_off=9.0, wall="outlet")
    for kw in (discs, dict(forcing="guo")):
        assert create([(32, 111)], "f64", "split", (8, 4), **kw) == amlbm.ENOMEM
        assert create([(32, 111)], "f64", "split", (16, 8), **kw) == amlbm.EINVAL
        assert create([(32, 111)], "f64", "split", **kw) == amlbm.EINVAL
        assert create([(32, 111)], "f32", "split", (32, 8), **kw) == amlbm.EINVAL
    own = [create([(1025, 512)], "f32", "pair", (48, h)) == amlbm.ENOMEM for h in range(2, 130, 4)]
    assert sum(own) == 1
    assert all(create([(1025, 512)], "f16", "pair", (48, h)) == amlbm.EINVAL for h in range(2, 130, 4))
