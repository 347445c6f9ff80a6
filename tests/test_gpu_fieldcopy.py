"""Device-side copies of a field into and out of the padded layout (rows shorter than a warp, at and
just past one and four 32-element segments), in every storage type: values are exact in FP32 and
FP64 and rounded once to FP16 times the scale in FP16 storage."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2206_00638_gb300 import sbpsat as sb  # noqa: E402


@pytest.mark.parametrize("precision", [sb.FP32, sb.FP64, sb.FP32_FP16STORE])
@pytest.mark.parametrize("n", [(4, 4, 4), (30, 9, 8), (31, 8, 11), (126, 5, 9), (127, 12, 8), (200, 8, 8)])
def test_device_copies_match_host_values(n, precision):
    sim = sb.Sim(n, (1e-3,) * 3, (sb.PEC,) * 6, precision=precision, field_scale=(2.0, 0.5))
    rng = np.random.default_rng(7)
    for c in range(6):
        a = rng.uniform(-1.0, 1.0, size=sim.shape(c)).astype(sim.dtype)
        want = a
        if precision == sb.FP32_FP16STORE:
            scale = np.float32(2.0 if c < 3 else 0.5)
            want = (a * (np.float32(1) / scale)).astype(np.float16).astype(np.float32) * scale
        sim.set_field(c, torch.from_numpy(a).cuda())
        out = torch.full(sim.shape(c), 9.0, dtype=torch.from_numpy(a).dtype, device="cuda")
        sim.field(c, out=out)
        assert np.array_equal(out.cpu().numpy(), want)
        assert np.array_equal(sim.field(c), want)          # the host copy
        sim.set_field(c, a)                                # and the host path in
        sim.field(c, out=out)
        assert np.array_equal(out.cpu().numpy(), want)
    sim.close()
