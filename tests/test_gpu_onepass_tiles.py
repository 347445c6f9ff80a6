"""Every tile of the one-pass step against the in-place half-steps, bit for bit.  Small grids step in
place unless SBP_STEP_PATH asks for one pass, so each test asks for it and checks which kernels ran."""
import threading

import numpy as np
import pytest

from paper_2206_00638_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2206_00638_gb300 import sbpsat  # noqa: E402

P, M, A = wl.PEC, wl.PMC, wl.ABSORBING
STEPS = 30


def _sim(w, path, monkeypatch, precision=sbpsat.FP32, **env):
    monkeypatch.setenv("SBP_STEP_PATH", path)
    for k, v in env.items():
        monkeypatch.setenv(k, str(v))
    s = sbpsat.from_workload(w, precision=precision)[0]
    for k in env:
        monkeypatch.delenv(k)
    s.reserve_probes(w.steps)
    return s


def _state(s, path):
    """Fields and probes after a last step whose kernels show the path."""
    assert ("fused_interior" in s.step_timed(1)) == (path == "onepass")
    return [s.field(c) for c in range(6)] + [s.probes()]


def _same(a, b):
    return all(np.array_equal(x, y) for x, y in zip(a, b))


@pytest.mark.parametrize("precision", [sbpsat.FP32, sbpsat.FP32_FP16STORE])
@pytest.mark.parametrize("width, rows", [(64, 8), (64, 16), (128, 8), (128, 12)])
@pytest.mark.parametrize("n", [(70, 43, 37), (140, 30, 21), (300, 26, 13), (33, 20, 17), (8, 9, 10)])
def test_tile_equals_in_place(n, width, rows, precision, monkeypatch):
    w = wl.random_box(n, faces=(A, P, M, A, P, M), seed=23, steps=STEPS)
    out = []
    for path in ("onepass", "inplace"):
        s = _sim(w, path, monkeypatch, precision, SBP_FUSED_WIDTH=width, SBP_FUSED_ROWS=rows, SBP_FUSED_KCHUNK=9)
        assert s.tile() == (rows, 9, width)
        s.step(STEPS - 1)
        out.append(_state(s, path))
        s.close()
    assert _same(*out)


@pytest.mark.parametrize("precision", [sbpsat.FP32, sbpsat.FP32_FP16STORE])
def test_tuned_equals_untuned_and_in_place(precision, monkeypatch):
    w = wl.random_box((140, 43, 61), faces=(A, P, M, A, P, M), seed=13, steps=STEPS)
    out = []
    for path, tune in (("onepass", True), ("onepass", False), ("inplace", False)):
        s = _sim(w, path, monkeypatch, precision)
        s.step(3)
        if tune:
            before = [s.field(c) for c in range(6)]
            depth, ms = s.autotune(2)
            assert depth == s.tile()[1] and ms > 0 and s.step_index == 3
            assert _same(before, [s.field(c) for c in range(6)])
        s.step(STEPS - 4)
        out.append(_state(s, path))
        s.close()
    assert _same(out[0], out[1]) and _same(out[0], out[2])


def test_one_pass_step_under_concurrent_load(monkeypatch):
    """The two streams of a one-pass step give the same bits alone and beside other work."""
    w = wl.dielectric(N=64, steps=400)

    def run(load):
        s = _sim(w, "onepass", monkeypatch)
        stop = threading.Event()

        def busy():
            st, x = torch.cuda.Stream(), torch.rand(1 << 24, device="cuda")
            with torch.cuda.stream(st):
                while not stop.is_set():
                    for _ in range(20):
                        x.mul_(1.0000001).add_(1e-9)
                    st.synchronize()

        th = threading.Thread(target=busy)
        if load:
            th.start()
        try:
            s.step(w.steps - 1)
            out = _state(s, "onepass")
        finally:
            stop.set()
            if load:
                th.join()
        s.close()
        return out

    ref = run(False)
    for load in (True, False, True):
        assert _same(run(load), ref)
