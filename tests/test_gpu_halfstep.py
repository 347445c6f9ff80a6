"""In-place half-steps: sizes at the edges of the box, its vectors and the rules that choose vector
width and z-chunk, every face type, with and without mu_r, against the oracle (tolerances of the
parity tests: FP32 1e-5, FP64 1e-11), and bit for bit against the one-pass path where both run."""
import numpy as np
import pytest

from paper_2206_00638_gb300 import workloads as wl
from tests import parity

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2206_00638_gb300 import sbpsat  # noqa: E402

P, M, A = sbpsat.PEC, sbpsat.PMC, sbpsat.ABSORBING
TOL = {sbpsat.FP32: 1e-5, sbpsat.FP64: 1e-11}
# the smallest grids, boxes of 0, 1 and a few vectors, 200 k nodes (vectors of 2 or 4 begin), 4 M (4 planes -> 8)
SIZES = [(4, 4, 4), (5, 7, 6), (8, 4, 9), (9, 8, 7), (11, 13, 10), (34, 7, 8), (66, 57, 53), (73, 50, 59)]


@pytest.mark.parametrize("precision", [sbpsat.FP32, sbpsat.FP64])
@pytest.mark.parametrize("mu", [None, (1.0, 3.0)])
@pytest.mark.parametrize("n", SIZES)
def test_against_oracle(n, mu, precision):
    for faces in ((P, M, A, P, M, A), (A, A, P, A, A, M)):
        w = wl.random_box(n, h=(1e-3, 1.1e-3, 0.9e-3), faces=faces, seed=11, mu_range=mu)
        sims = parity.gpu_run(w, 12, precision)
        blocks = parity.oracle_run(w, 12, sims[0].dt)
        assert max(parity.compare(sims, blocks)[0]) < TOL[precision]
        assert parity.probe_error(sims, blocks) < TOL[precision]
        sims[0].close()


@pytest.mark.parametrize("precision", [sbpsat.FP32, sbpsat.FP32_FP16STORE])
@pytest.mark.parametrize("n", [(8, 8, 8), (13, 9, 21), (67, 40, 33), (72, 61, 50), (130, 66, 131), (260, 131, 127)])
def test_bitwise_equal_to_one_pass(n, precision, monkeypatch):
    w = wl.random_box(n, faces=(A, M, P, A, P, M), seed=5)
    out = []
    for path in ("onepass", "inplace", "inplace64"):
        monkeypatch.setenv("SBP_STEP_PATH", path)
        s = parity.gpu_run(w, 9, precision)[0]
        out.append([s.field(c) for c in range(6)] + [s.probes()])
        s.close()
    for a, b, c in zip(*out):
        assert np.array_equal(a, b) and np.array_equal(a, c)


@pytest.mark.parametrize("axis", [0, 1, 2])
def test_joined_blocks_bitwise_on_both_paths(axis, monkeypatch):
    w = wl.coupled_boxes((26, 33, 21), (26, 33, 21), axis, seed=3)
    out = []
    for path in ("onepass", "inplace"):
        monkeypatch.setenv("SBP_STEP_PATH", path)
        sims = parity.gpu_run(w, 7, sbpsat.FP32)
        out.append([s.field(c) for s in sims for c in range(6)])
        for s in sims:
            s.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)


def test_steps_replay_from_a_captured_graph():
    """Half-steps launched with a programmatic dependency can be captured: replays step on."""
    stream = torch.cuda.Stream()
    w = wl.random_box((40, 31, 28), seed=9, sources=False, nprobes=0)
    with torch.cuda.stream(stream):
        a = sbpsat.from_workload(w, stream=stream)[0]
        b = sbpsat.from_workload(w, stream=stream)[0]
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=stream):
            a.step(3)
        g.replay()
        g.replay()
        b.step(6)
        for c in range(6):
            assert np.array_equal(a.field(c), b.field(c))
