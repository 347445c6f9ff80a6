"""In-place half-steps on both sides of the sizes where vector width and z-chunk change (0.2 M nodes:
2 -> 4 planes; 2.5 M: vectors of 2 -> 4 in FP32; 64 M: 4 -> 16 planes), with and without mu_r."""
import numpy as np
import pytest

from paper_2206_00638_gb300 import workloads as wl
from tests import parity

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2206_00638_gb300 import sbpsat  # noqa: E402

P, M, A = wl.PEC, wl.PMC, wl.ABSORBING
FACES = (P, M, A, P, M, A)


@pytest.mark.parametrize("mu", [None, (1.0, 3.0)])
@pytest.mark.parametrize("n", [(57, 55, 57), (56, 57, 58), (133, 135, 134), (135, 134, 136)])
def test_sizes_of_the_rules_against_oracle(n, mu):
    w = wl.random_box(n, h=(1e-3, 1.1e-3, 0.9e-3), faces=FACES, seed=12, mu_range=mu)
    sims = parity.gpu_run(w, 6, sbpsat.FP32)
    blocks = parity.oracle_run(w, 6, sims[0].dt)
    assert max(parity.compare(sims, blocks)[0]) < 1e-5
    assert parity.probe_error(sims, blocks) < 1e-5
    sims[0].close()


@pytest.mark.parametrize("precision", [sbpsat.FP32, sbpsat.FP32_FP16STORE])
def test_chunks_of_sixteen_planes(precision, monkeypatch):
    """65.4 M nodes in place, with 32- and 64-bit indices, and in one pass (FP16 storage on request)."""
    n = (403, 401, 399)
    gen = torch.Generator(device="cuda").manual_seed(2)
    eps = np.random.default_rng(2).uniform(1, 4, (n[2], n[1], n[0])).astype(np.float32)
    start = [(torch.rand(wl.field_shape(n, c), generator=gen, device="cuda") - 0.5) / (1 if c < 3 else 377)
             for c in range(6)]
    out = []
    for path, fused in (("inplace", False), ("inplace64", False), ("onepass", True)):
        monkeypatch.setenv("SBP_STEP_PATH", path)
        monkeypatch.delenv("SBP_NO_FUSED", raising=False)
        if not fused:
            monkeypatch.setenv("SBP_NO_FUSED", "1")
        s = sbpsat.Sim(n, (1e-3,) * 3, FACES, eps_r=eps, precision=precision)
        for c in range(6):
            s.set_field(c, start[c])
        s.step(2)
        assert ("fused_interior" in s.step_timed(1)) == fused
        out.append([s.field(c, out=torch.empty_like(start[c])) for c in range(6)])
        torch.cuda.synchronize()
        s.close()
    for a, b, c in zip(*out):
        assert torch.equal(a, b) and torch.equal(a, c)
