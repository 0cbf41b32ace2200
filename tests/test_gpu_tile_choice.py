"""The tile the library takes for a requested schedule computes the same state."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1310_1871_gb300 import amlbm  # noqa: E402


@pytest.mark.parametrize("storage", ["f64", "f32", "bf16"])
@pytest.mark.parametrize("shapes", [[(2, 4)], [(64, 32)], [(26, 10)] * 20, [(1024, 260), (30, 9)]])
def test_schedule_without_a_tile_equals_fused(shapes, storage):
    def run(**kw):
        b = amlbm.Batch([amlbm.InstanceSpec(z, r, 0.9, -4.9) for z, r in shapes], storage=storage, **kw)
        rng = np.random.default_rng(5)
        for k, (z, r) in enumerate(shapes):
            b.init_fields(k, 1.0 + 0.1 * rng.random((r, z)))
        b.step(6)
        out = [b.read_f(k) for k in range(len(shapes))]
        kind = b.schedule
        b.close()
        return out, kind

    ref, _ = run(tile=(32, 8), schedule="fused")
    for schedule in ("fused", "split", "pair"):
        got, kind = run(schedule=schedule)
        assert kind == schedule
        for a, c in zip(ref, got):
            assert np.array_equal(a, c), schedule


DISCS = dict(z_bc="noslip", r_lo="inlet", r_off=9.0, wall="outlet")


@pytest.mark.parametrize("shapes,storage,kw", [([(32, 111)], "f64", DISCS), ([(192, 120)], "f64", dict(forcing="guo")),
                                               ([(401, 300), (96, 48)], "f32", {}),
                                               ([(32, 111)], "f32", DISCS), ([(700, 400)], "f32", {})])
def test_own_choice_is_a_candidate_and_can_be_requested(shapes, storage, kw):
    """The autotuner times what the library takes without a request, and the schedule and
    tile a batch reports make the same batch again."""
    specs = [amlbm.InstanceSpec(z, r, 1.0, 0.0 if "z_bc" in kw else -5.0, **kw) for z, r in shapes]

    def run(**opt):
        b = amlbm.Batch(specs, storage=storage, **opt)
        for k, (z, r) in enumerate(shapes):
            b.init_fields(k, 1.0 + 0.01 * np.random.default_rng(k).random((r, z)))
        b.step(5)
        out = [b.read_f(k) for k in range(len(shapes))]
        kind = (b.schedule, b.tile)
        b.close()
        return out, kind

    ref, own = run()
    got, kind = run(schedule=own[0], tile=own[1])
    assert kind == own and all(np.array_equal(a, c) for a, c in zip(ref, got))
    _, _, cands = amlbm.autotune_raw(specs, storage, steps=5)
    assert [(c["schedule"], tuple(c["tile"])) for c in cands].count(own) == 1
