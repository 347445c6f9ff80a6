"""Tuning a grid that steps in place: there is no tile to choose, and the time is its own steps'."""
import numpy as np
import pytest

from paper_2206_00638_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2206_00638_gb300 import sbpsat  # noqa: E402


@pytest.mark.parametrize("precision", [sbpsat.FP32, sbpsat.FP32_FP16STORE])
@pytest.mark.parametrize("n", [(150, 61, 43), (70, 100, 90), (230, 40, 33)])
def test_tile_and_state_stay(n, precision):
    """The tile that no step uses is not searched for; trial steps leave fields, probes and step alone."""
    w = wl.random_box(n, seed=8, steps=20)
    tuned, plain = (sbpsat.from_workload(w, precision=precision)[0] for _ in range(2))
    for s in (tuned, plain):
        s.reserve_probes(20)
        s.step(3)
    tile = tuned.tile()
    depth, ms = tuned.autotune(3)
    assert tuned.tile() == tile and depth == tile[1] and ms > 0 and tuned.step_index == 3
    for s in (tuned, plain):
        s.step(17)
    for c in range(6):
        assert np.array_equal(tuned.field(c), plain.field(c)), c
    assert np.array_equal(tuned.probes(), plain.probes())


def test_joined_blocks_that_step_in_place():
    w = wl.two_block(nxy=40, nz=24, steps=10)
    tuned, plain = sbpsat.from_workload(w), sbpsat.from_workload(w)
    for g in (tuned, plain):
        sbpsat.step_group(g, 4)
    tile = tuned[1].tile()
    tuned[1].autotune(3)
    assert tuned[1].tile() == tile
    for g in (tuned, plain):
        sbpsat.step_group(g, 6)
    for a, b in zip(tuned, plain):
        for c in range(6):
            assert np.array_equal(a.field(c), b.field(c)), c
