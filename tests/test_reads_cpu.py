"""The step and energy kernels stay inside their arrays: the device code runs on the host with an
unmapped page behind every field and cell array (the arrays are the caller's workspace, and behind
the last one there may be nothing).  Grids: the smallest, rows without padding (nx + 2 a multiple of
8), thin ones, and past each vector remainder."""
import subprocess

import pytest

from tests import host_replay

MAIN = r"""
template <typename T, bool MU> void halves(Host &g, int face)
{
    auto p = g.params<T>(face, MU);
    constexpr int V = sizeof(T) == 8 ? 1 : 4;
    const Dim block = {sbp::kSweepThreads, 1, 1};
    for (int kz : {1, 4}) {
        const sbp::Sweep wh = g.sweep(false, V, kz), we = g.sweep(true, V, kz);
        launch({wh.ctas, 1, 1}, block, [&] { sbp::half_h<unsigned, T, T, MU, V>(p, wh); });
        launch({we.ctas, 1, 1}, block, [&] { sbp::half_e<unsigned, T, T, MU, V>(p, we); });
        launch({we.ctas, 1, 1}, block, [&] { sbp::half_e<long long, T, T, MU, V>(p, we); });
    }
}

void rims(Host &g, int face)
{
    auto p = g.params<float>(face, false);
    const sbp::Sweep wh = g.sweep(false, 1, 4, true), we = g.sweep(true, 1, 4, true);
    const Dim block = {sbp::kSweepThreads, 1, 1};
    float *out[3] = {guarded<float>(g.elems), guarded<float>(g.elems), guarded<float>(g.elems)};
    launch({wh.ctas, 1, 1}, block, [&] { sbp::rim_step<false, float>(p, wh, out[0], out[1], out[2]); });
    launch({we.ctas, 1, 1}, block, [&] { sbp::rim_step<true, float>(p, we, out[0], out[1], out[2]); });
}

template <typename T, bool MU> void energy(Host &g, int face)
{
    auto p = g.params<T>(face, MU);
    const Dim block = {sbp::kBlockX, sbp::kBlockY, 1};
    for (int kc : {3, 8}) {
        const Dim grid = {(g.n[0] + 2 + block.x - 1) / block.x, (g.n[1] + 2 + block.y - 1) / block.y,
                          (unsigned)(g.n[2] + 2 + kc - 1) / kc};
        p.kchunk = kc;
        p.partials = guarded<double>(grid.x * grid.y * grid.z);
        launch(grid, block, [&] { sbp::energy_sum<T, T, MU>(p); });
    }
}

// The slab kernels' nodes (the persistent batch's boundary, one-pass steps with 64-bit indices).
void bands(Host &g, int face)
{
    auto p = g.params<float>(face, false);
    float *out[3] = {guarded<float>(g.elems), guarded<float>(g.elems), guarded<float>(g.elems)};
    for (bool electric : {false, true}) {
        const sbp::Band b = make_band(g.n, electric);
        launch({b.ctas, 1, 1}, {256, 1, 1}, [&] {
            if (electric) sbp::band_e<float, false>(p, b, out[0], out[1], out[2]);
            else sbp::band_h<float, false>(p, b, out[0], out[1], out[2]);
        });
    }
}

int main(int argc, char **argv)
{
    const int n[3] = {std::atoi(argv[2]), std::atoi(argv[3]), std::atoi(argv[4])}, face = std::atoi(argv[5]);
    Host g(n);
    const char what = argv[1][0];
    if (what == 'h') { halves<float, false>(g, face); halves<double, true>(g, face); halves<float, true>(g, face); }
    if (what == 'r') rims(g, face);
    if (what == 'b') bands(g, face);
    if (what == 'e') { energy<float, false>(g, face); energy<double, true>(g, face); }
    return 0;
}
"""
GRIDS = [(4, 4, 4), (6, 5, 7), (14, 8, 9), (13, 9, 11), (256, 6, 6), (400, 10, 10), (1000, 4, 4)]
FACES = [0, 1, 2]    # PEC, PMC, absorbing


@pytest.fixture(scope="module")
def replay(tmp_path_factory):
    exe = host_replay.build(str(tmp_path_factory.mktemp("replay")), MAIN)
    return lambda what, n, face: subprocess.run([exe, what, *map(str, n), str(face)]).returncode


@pytest.mark.parametrize("face", FACES)
@pytest.mark.parametrize("n", GRIDS)
def test_half_steps_stay_inside(replay, n, face):
    assert replay("half", n, face) == 0


@pytest.mark.parametrize("face", FACES)
@pytest.mark.parametrize("n", [m for m in GRIDS if min(m) >= 8])
def test_rim_of_one_pass_steps_stays_inside(replay, n, face):
    assert replay("rim", n, face) == 0


@pytest.mark.parametrize("face", FACES)
@pytest.mark.parametrize("n", GRIDS)
def test_energy_stays_inside(replay, n, face):
    assert replay("energy", n, face) == 0


@pytest.mark.parametrize("face", FACES)
@pytest.mark.parametrize("n", [m for m in GRIDS if min(m) >= 8])
def test_band_kernels_stay_inside(replay, n, face):
    assert replay("band", n, face) == 0
