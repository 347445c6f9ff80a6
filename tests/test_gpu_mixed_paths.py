"""Blocks joined across the two step paths: one that steps in one pass with one that steps in place
(a large and a small block of one group), bit for bit against both in place, run and captured."""
import numpy as np
import pytest

from paper_2206_00638_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2206_00638_gb300 import sbpsat  # noqa: E402

P, M, A = wl.PEC, wl.PMC, wl.ABSORBING


def _group(w, paths, monkeypatch, precision=sbpsat.FP32):
    sims = []
    for b, path in zip(w.blocks, paths):
        monkeypatch.setenv("SBP_STEP_PATH", path)
        sims += sbpsat.from_workload(wl.Workload("one", [b], [], w.cfl, w.steps), precision=precision)
        sims[-1].reserve_probes(64)
    for a, fa, b, fb in w.links:
        sims[a].connect(fa, sims[b], fb)
    return sims


def _state(sims):
    out = [s.field(c) for s in sims for c in range(6)] + [s.probes() for s in sims]
    for s in sims:
        s.close()
    return out


def _same(a, b):
    return all(np.array_equal(x, y) for x, y in zip(a, b))


@pytest.mark.parametrize("precision", [sbpsat.FP32, sbpsat.FP32_FP16STORE])
@pytest.mark.parametrize("axis", [0, 1, 2])
def test_joined_blocks_on_different_paths(axis, precision, monkeypatch):
    w = wl.coupled_boxes((26, 33, 21), (26, 33, 21), axis, facesA=(A, P, M, A, P, M), facesB=(P, A, A, M, M, P), seed=3)
    out = []
    for paths in (("inplace", "inplace"), ("onepass", "inplace"), ("inplace", "onepass")):
        sims = _group(w, paths, monkeypatch, precision)
        sbpsat.step_group(sims, 9)
        out.append(_state(sims))
    assert _same(out[0], out[1]) and _same(out[0], out[2])


def test_complex_pair_on_different_paths(monkeypatch):
    w = [wl.random_box((20, 17, 23), seed=q, sources=False, nprobes=0) for q in (5, 6)]
    out = []
    for paths in (("inplace", "inplace"), ("onepass", "inplace")):
        sims = []
        for v, path in zip(w, paths):
            monkeypatch.setenv("SBP_STEP_PATH", path)
            sims += sbpsat.from_workload(v)
        for axis in range(3):
            sbpsat.connect_phase(sims[0], sims[1], axis, 0.4 + axis)
        sbpsat.step_group(sims, 8)
        out.append([s.field(c) for s in sims for c in range(6)])
    assert _same(*out)


@pytest.mark.parametrize("paths", [("inplace", "inplace"), ("onepass", "inplace"), ("inplace", "onepass")])
def test_captured_group(paths, monkeypatch):
    """A group's steps captured on a stream that has joined another: field copies, events and half-steps
    that start early keep their order in the graph."""
    w = wl.coupled_boxes((26, 33, 21), (26, 33, 21), 2, seed=4)
    stream, other = torch.cuda.Stream(), torch.cuda.Stream()
    with torch.cuda.stream(stream):
        sims = _group(w, paths, monkeypatch)
        ref = _group(w, ("inplace", "inplace"), monkeypatch)
        new = torch.rand(sims[0].shape(0), device="cuda")
        src = torch.zeros_like(new)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=stream):
            fork = torch.cuda.Event()
            fork.record(stream)
            other.wait_event(fork)
            with torch.cuda.stream(other):
                src.copy_(new)
                join = torch.cuda.Event()
                join.record(other)
            stream.wait_event(join)
            sbpsat.step_group(sims, 2)
            sims[0].set_field(0, src)
            sbpsat.step_group(sims, 4)
        for s in sims + ref:
            assert s.step_index == (6 if s in sims else 0)
        g.replay()
        sbpsat.step_group(ref, 2)
        ref[0].set_field(0, new)
        sbpsat.step_group(ref, 4)
        torch.cuda.synchronize()
        assert _same(_state(sims), _state(ref))
