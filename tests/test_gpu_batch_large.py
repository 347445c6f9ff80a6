"""Batch members past the sizes of the small shared launches."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2206_00638_gb300 import sbpsat  # noqa: E402
from paper_2206_00638_gb300 import workloads as wl  # noqa: E402
from tests import parity  # noqa: E402

P, M, A = sbpsat.PEC, sbpsat.PMC, sbpsat.ABSORBING
H = (1e-3,) * 3


def _driven(n, at, probes):
    """A vacuum block driven by a point source, stepped six times as a batch's only member; its
    probes.  In six steps the field reaches six cells, so any two such blocks agree around the source."""
    s = sbpsat.Sim(n, H, (P,) * 6)
    s.add_source(sbpsat.EZ, *at, sbpsat.GAUSS, 100.0, 4e-12, 4e-12)
    for c, i, j, k in probes:
        s.add_probe(c, i, j, k)
    s.reserve_probes(6)
    batch = sbpsat.Batch()
    batch.add(s, 6)
    batch.step(6)
    out = s.probes()
    batch.close()
    s.close()
    torch.cuda.empty_cache()            # the workspace leaves the allocator's pool
    return out


def test_member_of_more_than_2_to_32_elements():
    """Planes past element 2^32 (1024 x 1024 elements a plane, from plane 4096 on) get their own
    update, and the planes 4096 below them keep their zeros."""
    torch.cuda.empty_cache()
    n, high = (1022, 1022, 4128), 4110
    if torch.cuda.mem_get_info()[0] < 235 << 30:
        pytest.skip("needs 235 GiB of free device memory")
    around = [(c, 500 + d, 400 - d, high + e) for c in range(6) for d in (0, 1, 2) for e in (-2, 0, 1)]
    below = [(c, 500, 400, high - 4096 + e) for c in (0, 2, 3) for e in (-1, 0)]
    big = _driven(n, (500, 400, high), around + below)
    small = _driven((40, 40, 40), (20, 20, 20), [(c, i - 480, j - 380, k - high + 20) for c, i, j, k in around])
    assert np.abs(small).max() > 0
    assert np.array_equal(big[: len(around)], small)
    assert not big[len(around):].any()


@pytest.mark.parametrize("use_graphs", [True, False])
def test_one_pass_members_beside_others(use_graphs, monkeypatch):
    """Members that step in one pass, a batch of them alone first, then with members that step in
    place: each gives the bits it gives alone, whichever ends first and inside a chunk."""
    sizes = [((40, 33, 29), 17, "onepass"), ((70, 43, 37), 30, "onepass"), ((33, 20, 17), 21, "inplace"),
             ((64, 48, 40), 40, "inplace")]
    works = [wl.random_box(n, faces=(A, P, M, A, P, M), seed=40 + q, steps=st) for q, (n, st, _) in enumerate(sizes)]
    alone, sims = [], []
    for w, (_, st, path) in zip(works, sizes):
        monkeypatch.setenv("SBP_STEP_PATH", path)
        a = parity.gpu_run(w, st, sbpsat.FP32, energy_every=5)[0]
        alone.append([a.field(c) for c in range(6)] + [a.probes()])
        a.close()
        s = sbpsat.from_workload(w, energy_every=5)[0]
        s.reserve_probes(st)
        sims.append(s)
    batch = sbpsat.Batch(use_graphs=use_graphs)
    for s, (_, st, _) in zip(sims[:2], sizes):
        batch.add(s, st)
    batch.step(7)
    for s, (_, st, _) in zip(sims[2:], sizes[2:]):
        batch.add(s, st)
    for k in (7, 7, 7, 7, 9, 5):
        batch.step(k)
    for s, (_, st, _), ref in zip(sims, sizes, alone):
        assert batch.remaining(s) == 0 and s.step_index == st
        for c in range(6):
            assert np.array_equal(s.field(c), ref[c]), (s.n, c)
        assert np.array_equal(s.probes(), ref[6])
    batch.close()
    for s in sims:
        s.close()


def test_members_take_the_path_they_take_alone():
    """The one-pass kernel's bounded waits, made to run out, are reported from a batch as from
    sbp_step: a member whose steps go through that kernel goes through it in a batch."""
    s = sbpsat.Sim((40, 33, 29), H, (P,) * 6, flags=sbpsat.FLAG_TEST_WAIT_TIMEOUT)
    batch = sbpsat.Batch()
    batch.add(s, 2)
    batch.step(2)
    with pytest.raises(sbpsat.SbpError) as err:
        s.sync()
    assert err.value.code == -5
    batch.close()
    s.close()


def _members():
    """Small members of more than one L2 group, two that step by themselves in vectors of 2, one in
    vectors of 4 (2.5 M nodes), and targets that end inside chunks."""
    sizes = [(33, 20, 17), (88, 88, 86), (86, 90, 88), (91, 85, 87), (87, 89, 90), (84, 92, 88), (101, 100, 99),
             (117, 96, 131), (142, 135, 140), (8, 9, 8)]
    steps = [13, 21, 16, 9, 24, 17, 23, 11, 15, 5]
    rng = np.random.default_rng(7)
    out = []
    for q, (n, st) in enumerate(zip(sizes, steps)):
        faces = tuple(int(v) for v in rng.choice([P, M, A], size=6))
        out.append(wl.random_box(n, faces=faces, seed=60 + q, steps=st))
    return out


@pytest.mark.parametrize("use_graphs", [True, False])
def test_groups_and_lone_members_equal_alone(use_graphs):
    """Shared launches of several groups, members alone in a launch, and members that leave and join
    between chunks: every one with the bits it has alone."""
    works = _members()
    sims = []
    for w in works:
        sims.append(sbpsat.from_workload(w)[0])
        sims[-1].reserve_probes(w.steps)
    batch = sbpsat.Batch(use_graphs=use_graphs)
    late = (2, 8)
    for q, (s, w) in enumerate(zip(sims, works)):
        if q not in late:
            batch.add(s, w.steps)
    batch.step(6)
    for q in late:
        batch.add(sims[q], works[q].steps)
    batch.remove(sims[9])                                  # done: its target was 5
    for k in (8, 8, 8):
        batch.step(k)
    for q, (s, w) in enumerate(zip(sims, works)):
        assert s.step_index == w.steps and (q == 9 or batch.remaining(s) == 0)
        alone = parity.gpu_run(w, w.steps, sbpsat.FP32)[0]
        for c in range(6):
            assert np.array_equal(s.field(c), alone.field(c)), (w.blocks[0].n, c)
        assert np.array_equal(s.probes(), alone.probes())
        alone.close()
    batch.close()


@pytest.mark.parametrize("n", [(48, 40, 33), (117, 96, 131), (142, 135, 140)])
@pytest.mark.parametrize("use_graphs", [True, False])
def test_last_member_ends_one_step_before_the_chunk(n, use_graphs):
    """The chunk's last launches are those of a finished member: fields read right after are whole."""
    w = wl.random_box(n, faces=(A, P, M, A, P, M), seed=71, steps=7)
    alone = parity.gpu_run(w, 7, sbpsat.FP32)[0]
    ref = [alone.field(c) for c in range(6)]
    for _ in range(3):
        s = sbpsat.from_workload(w)[0]
        s.reserve_probes(7)
        batch = sbpsat.Batch(use_graphs=use_graphs)
        batch.add(s, 7)
        batch.step(8)
        for c in range(6):
            assert np.array_equal(s.field(c), ref[c]), c
        batch.close()
        s.close()
    alone.close()


@pytest.mark.parametrize("use_graphs, persistent", [(True, False), (False, False), (True, True)])
def test_members_changed_between_chunks(use_graphs, persistent):
    """A member stepped by itself, given new sources and a new probe buffer, or restored from a checkpoint
    between chunks goes on from that state."""
    def change(s, k):
        if k == 0:
            s.step(3)
        elif k == 1:
            s.reserve_probes(50)
            s.add_source(sbpsat.EX, 5, 6, 7, sbpsat.GAUSS, 50.0, 4e-12, s.dt * s.step_index)
        elif k == 2:
            s.load(s.saved)

    works = [wl.random_box(n, faces=(A, P, M, A, P, M), seed=90 + q) for q, n in enumerate([(20, 17, 23), (40, 33, 29)])]
    batch, sims, refs = sbpsat.Batch(use_graphs=use_graphs, persistent=persistent), [], []
    for w in works:
        for group in (sims, refs):
            group.append(sbpsat.from_workload(w)[0])
            group[-1].reserve_probes(30)
        batch.add(sims[-1], 1000)
    for k in range(4):
        batch.step(5)
        for s in refs:
            s.step(5)
        if k == 1:
            for s in sims + refs:
                s.saved = s.save()
        for s in (sims[1], refs[1]):
            change(s, k)
    for s, r in zip(sims, refs):
        assert s.step_index == r.step_index
        for c in range(6):
            assert np.array_equal(s.field(c), r.field(c)), c
        assert np.array_equal(s.probes(), r.probes())
    batch.close()


@pytest.mark.parametrize("persistent", [False, True])
def test_members_connected_after_joining_are_refused(persistent):
    """A batch steps single blocks: connecting members to each other, before or after its first chunk,
    is refused at the next one (on the host), and the members go on as a group."""
    for early in (True, False):
        w = wl.random_box((20, 17, 23), seed=6)
        sims = [sbpsat.from_workload(w)[0] for _ in range(2)]
        batch = sbpsat.Batch(persistent=persistent)
        for s in sims:
            batch.add(s, 20)
        if not early:
            batch.step(2)
        sims[0].connect(5, sims[1], 4)
        with pytest.raises(sbpsat.SbpError) as err:
            batch.step(2)
        assert err.value.code == -7
        for s in sims:
            batch.remove(s)
        sbpsat.step_group(sims, 2)
        assert [s.step_index for s in sims] == ([2, 2] if early else [4, 4])
        batch.close()


@pytest.mark.parametrize("steps", [6001, 9000])
def test_long_chunk_in_pieces(steps):
    """One call for thousands of steps keeps its graph small (a whole one of 9000 steps of three launches'
    worth of members would hold some 100 MB on the device) and gives the bits of the same steps alone."""
    works = [wl.random_box(n, faces=(A, P, M, A, P, A), seed=80 + q, steps=steps - 700 * q)
             for q, n in enumerate([(8, 9, 8), (14, 11, 12), (101, 100, 20)])]
    sims = [sbpsat.from_workload(w)[0] for w in works]
    batch = sbpsat.Batch()
    for s, w in zip(sims, works):
        batch.add(s, w.steps)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    batch.step(steps)
    torch.cuda.synchronize()
    assert free - torch.cuda.mem_get_info()[0] < 64 << 20
    for s, w in zip(sims, works):
        assert s.step_index == w.steps
        alone = sbpsat.from_workload(w)[0]
        alone.step(w.steps)
        for c in range(6):
            assert np.array_equal(s.field(c), alone.field(c)), c
        alone.close()
    batch.close()


def test_server_requests_in_one_pass(monkeypatch):
    """Served requests that step in one pass, admitted and retired between chunks beside each other,
    give the samples they give alone."""
    monkeypatch.setenv("SBP_STEP_PATH", "onepass")
    reqs = wl.serving_stream(nreq=5, seed=12, n_range=(20, 56), steps_range=(20, 70))
    ref = []
    for spec, steps in reqs:
        s = sbpsat.Sim(spec.n, spec.h, spec.faces, eps_r=spec.eps_r, cfl=0.95)
        for src in spec.sources:
            s.add_source(src.comp, src.i, src.j, src.k, src.kind, src.amp, src.tw, src.t0, src.f)
        for p in spec.probes:
            s.add_probe(p.comp, p.i, p.j, p.k)
        s.reserve_probes(steps)
        s.step(steps)
        ref.append(s.probes())
        s.close()
    srv = sbpsat.Server(stream=torch.cuda.Stream(), max_slots=3, chunk=16)
    tickets = [srv.submit(spec, steps) for spec, steps in reqs]
    srv.drain()
    for t, r, (spec, steps) in zip(tickets, ref, reqs):
        res = srv.poll(t)
        assert res is not None and res.status == 0 and res.steps == steps
        assert np.array_equal(srv.probes(t), r), spec.n
        srv.release(t)
    srv.close()
