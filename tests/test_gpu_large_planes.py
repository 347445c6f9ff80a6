"""Grids with few but huge planes: work lists whose counts need more than 32 bits."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2206_00638_gb300 import sbpsat  # noqa: E402

A, M, P = sbpsat.ABSORBING, sbpsat.PMC, sbpsat.PEC


def _corner(n, precision):
    """Probes around a source near the far x, y corner after six steps (the field reaches six cells)."""
    s = sbpsat.Sim(n, (1e-3,) * 3, (P, A, P, M, A, M), precision=precision)
    at = (n[0] - 5, n[1] - 6, n[2] // 2)
    s.add_source(sbpsat.EZ, *at, sbpsat.GAUSS, 100.0, 4e-12, 4e-12)
    for c in range(6):
        for d in ((0, 0, 0), (1, -1, 0), (3, 4, 1), (-2, 0, -1), (4, 5, -2), (-1, 4, 1)):
            s.add_probe(c, *(a + b for a, b in zip(at, d)))
    s.reserve_probes(6)
    s.step(6)
    out = s.probes()
    s.close()
    torch.cuda.empty_cache()            # the workspace leaves the allocator's pool
    return out


@pytest.mark.parametrize("n, precision, need", [((19000, 19000, 4), sbpsat.FP32, 75), ((16384, 16384, 8), sbpsat.FP32, 165),
                                                ((19000, 19000, 4), sbpsat.FP32_FP16STORE, 45)])
def test_corner_of_huge_planes(n, precision, need):
    """The layer planes hold 2.1e9 nodes: the far corner steps as a small grid's does."""
    torch.cuda.empty_cache()
    if torch.cuda.mem_get_info()[0] < need << 30:
        pytest.skip(f"needs {need} GiB of free device memory")
    big, small = _corner(n, precision), _corner((40, 40, n[2]), precision)
    assert np.abs(small[12]).max() > 0          # Ez at the source
    assert np.array_equal(big, small)
