"""Captured chunks of the step replay the direct launches bit for bit on every kernel that the
library chooses by itself: rows, strips, the two FP64 kernels and the persistent grid."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1310_1871_gb300 import amlbm  # noqa: E402


@pytest.mark.parametrize("shapes,storage,kw,kind", [
    ([(64, 32)], "f64", {}, ("split", (8, 4))), ([(197, 97)], "f64", dict(forcing="guo"), ("split", (16, 8))),
    ([(256, 128)], "f64", {}, ("split", (32, 8))), ([(200, 100)], "f32", {}, ("fused", None)),
    ([(512, 200), (64, 40)], "f32", {}, ("pair", None)), ([(513, 200), (64, 40)], "f32", {}, ("pair", None)),
    ([(512, 200)], "bf16", {}, ("pair", None)), ([(768, 256)], "f16", dict(shift="equilibrium"), ("pair", (64, 24))),
    ([(700, 300)], "f32", dict(src="link"), ("fused", (26, 16)))])
def test_chunks_equal_direct_launches(shapes, storage, kw, kind):
    stream = torch.cuda.Stream()
    out = []
    for chunk in (0, 4):
        with torch.cuda.stream(stream):
            b = amlbm.Batch([amlbm.InstanceSpec(z, r, 0.9, -4.9, **kw) for z, r in shapes], storage=storage,
                            graph_chunk=chunk, stream=stream)
            assert b.schedule == kind[0] and (kind[1] is None or b.tile == kind[1])
            for k, (z, r) in enumerate(shapes):
                b.init_fields(k, 1.0 + 0.1 * np.random.default_rng(k).random((r, z)))
            b.step(11)  # two chunks and three single steps: the next chunks start from the other parity
            b.step(9)
            d = b.diagnostics_all(as_array=True)
            out.append([b.read_f(k) for k in range(len(shapes))] + [d])
            b.close()
    for a, c in zip(*out):
        assert np.array_equal(a, c)
