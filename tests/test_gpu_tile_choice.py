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
