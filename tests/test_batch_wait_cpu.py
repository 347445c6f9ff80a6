"""A batched half-step whose members are done still waits for the launch before it: what follows (the
chunk's last launches, the step counters, copies of the fields) is ordered behind it alone."""
import subprocess

import pytest

from tests import host_replay

MAIN = r"""
int main(int argc, char **argv)
{
    const int n[3] = {9, 8, 10}, done = std::atoi(argv[2]);
    Host g(n);
    long long counter[2] = {5, 5};
    sbp::BatchHalf grids[2];
    int pre[3] = {0, 0, 0};
    for (int q = 0; q < 2; q++) {
        grids[q].p = g.params<float>(0, false);
        static_cast<sbp::Sweep &>(grids[q].w[0]) = g.sweep(false, 2, 2);
        static_cast<sbp::Sweep &>(grids[q].w[1]) = g.sweep(true, 2, 2);
        grids[q].counter = counter + q;
        grids[q].target = q < done ? 7 : 8;        // the launch below is step 7
        grids[q].probe_base = 0;
        pre[q + 1] = pre[q] + grids[q].w[1].ctas;
    }
    const Dim block = {sbp::kSweepThreads, 1, 1};
    const sbp::Sweep &w = grids[0].w[1];
    if (argv[1][0] == 's')
        launch({(unsigned)pre[2], 1, 1}, block, [&] { sbp::half_batched<true>(grids, pre, 2, 2); });
    else
        launch({w.ctas, 1, 1}, block, [&] { sbp::half_member<true, 2>(grids[0].p, w, counter, grids[0].target, 0, 2); });
    const long long idle = argv[1][0] == 's' ? done * w.ctas : w.ctas;
    return g_waits < idle * sbp::kSweepThreads;    // every thread of a CTA without work
}
"""


@pytest.fixture(scope="module")
def replay(tmp_path_factory):
    return host_replay.build(str(tmp_path_factory.mktemp("wait")), MAIN)


@pytest.mark.parametrize("launch, done", [("shared", 1), ("shared", 2), ("alone", 1)])
def test_done_members_wait(replay, launch, done):
    assert subprocess.run([replay, launch, str(done)]).returncode == 0
