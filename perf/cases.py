"""The work that users have this framework do, as cases to be timed and compared.

A case is one chunk of a running simulation: the blocks exist, with materials, initial fields,
sources and probes, and one pass advances them by ``steps`` leapfrog steps through the public
entry points and reads every field into device arrays.  ``exact`` is the same chunk in 64 bits in
plain torch, written from the scheme's definition (operators with closure rows, face penalties,
node materials), without the package's code.
"""
import math

import numpy as np
import torch

from paper_2206_00638_gb300 import sbpsat as sb

C0 = 299792458.0
EPS0 = 8.8541878128e-12
MU0 = 1.25663706212e-6
FACES = {"P": sb.PEC, "M": sb.PMC, "A": sb.ABSORBING, "I": sb.INTERFACE}
PRECISION = {"fp32": sb.FP32, "fp64": sb.FP64, "fp16": sb.FP32_FP16STORE}
ON_PLUS = ((0, 1, 1), (1, 0, 1), (1, 1, 0), (1, 0, 0), (0, 1, 0), (0, 0, 1))
# dC/dt = + D_a0 U0 - D_a1 U1: ((U0, a0), (U1, a1)) per component
CURL = (((5, 1), (4, 2)), ((3, 2), (5, 0)), ((4, 0), (3, 1)), ((1, 2), (2, 1)), ((2, 0), (0, 2)), ((0, 1), (1, 0)))


def listed():
    return [
        # the smallest run: the 1 m cavity in double precision, watched at one probe
        _case("cavity_fp64", 20, 16, 12, faces="PPPPPP", precision="fp64", cfl=0.9, h=0.05, steps=100),
        # one column of the dispersion tool's amplification matrix: write a periodic complex cube,
        # one step, read it back
        _case("dispersion_column", 8, 8, 8, kind="periodic", precision="fp64", cfl=0.99, steps=1, source="none"),
        # one small and one ordinary grid of the serving range (32..192 cells), stepped alone
        _case("lone_small", 61, 47, 38, faces="PAPAAP", eps="boxes", steps=64, source="point"),
        _case("lone_medium", 117, 96, 131, faces="APAAPP", eps="boxes", steps=64, source="point"),
        # a serving batch: grids of 32..192 cells per axis advanced by one chunk
        _case("batch_serving", 192, 192, 192, kind="batch", members=24, sizes=4, faces="random", eps="boxes",
              steps=32, source="point"),
        # two blocks joined by the interface penalty
        _case("two_block", 192, 192, 96, kind="joined", faces="AAAAAA", eps="patches", steps=32, source="sheet"),
        # the dielectric cube workload at full size
        _case("dielectric_256", 256, 256, 256, faces="PPPPPP", eps="cube", steps=32, source="point"),
        # the headline block, single precision and half-precision storage, tuned as its users do
        _case("mixed_512", 512, 512, 512, faces="MMPPAA", eps="spheres", steps=16, source="sheet", tune=True),
        _case("mixed_512_fp16", 512, 512, 512, faces="MMPPAA", eps="spheres", precision="fp16", steps=16,
              source="sheet", tune=True),
        # magnetic materials (mu_r per cell)
        _case("magnetic", 121, 101, 88, faces="MPAPAM", eps="boxes", mu=True, steps=32, source="point"),
        # a long run under the energy monitor, with an energy reading at the end of the chunk
        _case("monitored", 160, 144, 128, faces="PPMMPA", eps="boxes", steps=40, source="sheet", energy_every=10),
        # double precision at an ordinary size
        _case("block_fp64", 96, 75, 88, faces="MPAPAM", eps="boxes", precision="fp64", steps=16, source="point"),
    ]


def _case(name, nx, ny, nz, kind="block", faces="PPPPPP", precision="fp32", eps="vacuum", mu=False, source="point",
          steps=32, cfl=0.95, h=1e-3, members=1, sizes=0, energy_every=0, tune=False):
    c = {"kind": kind, "nx": nx, "ny": ny, "nz": nz, "faces": faces, "precision": precision, "eps": eps, "mu": mu,
         "source": source, "steps": steps, "cfl": cfl, "h": h, "members": members, "sizes": sizes,
         "energy_every": energy_every, "tune": tune}
    return dict(c, name=name) if name else c


def draw(rng):
    """One more case of the same ranges."""
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def faces():
        return "".join(rng.choice("PMA") for _ in range(6))

    kind = rng.choice(["block"] * 6 + ["joined", "batch", "periodic"])
    if kind == "periodic":
        return _case(None, size(4, 24), size(4, 24), size(4, 24), kind=kind, precision=rng.choice(["fp64", "fp32"]),
                     cfl=0.99, steps=rng.choice([1, 1, 4]), source="none")
    if kind == "batch":
        m = rng.randint(96, 192)
        return _case(None, m, m, m, kind=kind, members=rng.randint(3, 24), sizes=rng.randint(1, 9999),
                     faces="random", eps="boxes", steps=rng.randint(8, 32))
    if kind == "joined":
        return _case(None, size(24, 224), size(24, 224), size(24, 160), kind=kind, faces=faces(), eps="patches",
                     precision=rng.choice(["fp32", "fp32", "fp16", "fp64"]) if rng.random() < 0.3 else "fp32",
                     steps=rng.randint(8, 16), source="sheet")
    option = rng.choice(["plain", "plain", "plain", "fp16", "fp64", "mu", "energy"])
    top = 112 if option == "fp64" else 192 if option in ("mu", "energy") else 400
    n = [size(10, top) for _ in range(3)]
    steps = max(4, min(128, int(4e8 / (n[0] * n[1] * n[2] + 1e6))))
    if option in ("fp64", "mu", "energy"):
        steps = min(steps, 32)
    return _case(None, *n, faces=faces(), precision=option if option in ("fp16", "fp64") else "fp32",
                 eps=rng.choice(["vacuum", "boxes", "spheres", "cube"]), mu=option == "mu",
                 source=rng.choice(["point", "sheet"]), steps=steps,
                 energy_every=rng.randint(3, 20) if option == "energy" else 0)


# --- inputs -----------------------------------------------------------------

def _extents(n, c):
    return tuple(n[a] + (1 if ON_PLUS[c][a] else 2) for a in range(3))


def _members(case):
    """Cells of a batch's grids: uniform from 32 to nx per axis."""
    r = np.random.default_rng(case["sizes"])
    return [tuple(int(v) for v in r.integers(32, case["nx"] + 1, size=3)) for _ in range(case["members"])]


def _blocks(case, seed):
    """(cells, faces, seed) of every block of the case."""
    n = (case["nx"], case["ny"], case["nz"])
    if case["kind"] == "batch":
        r = np.random.default_rng(seed)
        return [(nb, "".join("PA"[v] for v in r.integers(0, 2, size=6)), seed * 1000 + m)
                for m, nb in enumerate(_members(case))]
    if case["kind"] == "joined":
        f = case["faces"]
        return [(n, f[:5] + "I", seed * 1000), (n, f[:4] + "I" + f[5], seed * 1000 + 1)]
    if case["kind"] == "periodic":
        return [(n, "PPPPPP", seed * 1000), (n, "PPPPPP", seed * 1000 + 1)]
    return [(n, case["faces"], seed * 1000)]


def _cells(n, kind, seed, lo, hi, gen):
    """Per-cell material (nz, ny, nx) float32 on the GPU."""
    nx, ny, nz = n
    a = torch.ones((nz, ny, nx), dtype=torch.float32, device="cuda")
    if kind == "cube":
        q = [slice(3 * m // 8, max(3 * m // 8 + 1, 5 * m // 8)) for m in (nz, ny, nx)]
        a[q[0], q[1], q[2]] = 4.0
    elif kind in ("boxes", "patches"):
        sub = 16 if kind == "boxes" else 8
        nb = [(m + sub - 1) // sub for m in (nz, ny, nx)]
        v = torch.rand(nb, generator=gen, device="cuda") * (hi - lo) + lo
        for ax in range(3):
            v = v.repeat_interleave(sub, ax)
        a = v[:nz, :ny, :nx].contiguous()
    elif kind == "spheres":
        r = np.random.default_rng(seed)
        m = min(n)
        ax = [torch.arange(k, device="cuda", dtype=torch.float32) + 0.5 for k in (nz, ny, nx)]
        for _ in range(4):
            rad = float(r.uniform(m / 16, 3 * m / 16))
            c = [float(r.uniform(rad, k - rad)) for k in (nz, ny, nx)]
            d2 = ((ax[0] - c[0]) ** 2)[:, None, None] + ((ax[1] - c[1]) ** 2)[None, :, None] + \
                ((ax[2] - c[2]) ** 2)[None, None, :]
            a[d2 <= rad * rad] = float(np.float32(r.uniform(2.0, 8.0)))
    return a


def _fields(n, gen, dtype):
    """Six smooth fields (three standing waves each) with one per cent of noise on every node:
    E of order 1 V/m, H of order 1/377 A/m."""
    out = []
    for c in range(6):
        e = _extents(n, c)
        f = torch.zeros((e[2], e[1], e[0]), dtype=torch.float32, device="cuda")
        for _ in range(3):
            p = torch.rand(6, generator=gen, device="cuda") * 2 * math.pi
            v = [torch.cos(torch.arange(e[a], device="cuda") * (p[a] / 4 / math.pi) + p[3 + a]) for a in range(3)]
            f += v[2][:, None, None] * (v[1][:, None] * v[0][None, :])[None]
        f += 0.02 * (torch.rand(f.shape, generator=gen, device="cuda") - 0.5)
        f *= 0.5 if c < 3 else 0.5 / 377.0
        out.append(f.to(dtype))
    return out


def _inputs(case, seed):
    """What every block starts from."""
    out = []
    dtype = torch.float64 if case["precision"] == "fp64" else torch.float32
    for n, faces, s in _blocks(case, seed):
        gen = torch.Generator(device="cuda").manual_seed(s)
        r = np.random.default_rng(s)
        hi = 4.0 if case["eps"] == "patches" else 6.0
        b = {"n": n, "faces": faces, "eps": None, "mu": None, "sources": [], "probes": []}
        if case["eps"] != "vacuum":
            b["eps"] = _cells(n, case["eps"], s, 1.0, hi, gen)
        if case["mu"]:
            b["mu"] = _cells(n, "boxes", s, 1.0, 2.0, gen)
        b["fields"] = _fields(n, gen, dtype)
        tw = math.sqrt(2.0 / math.pi) / 10e9 * case["h"] / 1e-3     # pulse about 10 GHz at 1 mm
        if case["source"] == "point":
            e = _extents(n, sb.EZ)
            pos = [int(r.integers(3, max(4, e[a] - 3))) for a in range(3)]
            b["sources"] = [(sb.EZ, *pos, sb.GAUSS_DERIV, 100.0, tw, tw)]
        elif case["source"] == "sheet":
            b["sources"] = [(sb.EY, -1, -1, n[2] // 16, sb.GAUSS, 100.0, tw, tw)]
        if case["source"] != "none":
            b["probes"] = [(c, *[int(r.integers(3, max(4, v - 3))) for v in _extents(n, c)]) for c in range(3)]
        out.append(b)
    return out


def _phases(seed):
    return [float(v) for v in np.random.default_rng(seed).uniform(0.1, 1.5, size=3)]


# --- the framework ----------------------------------------------------------

def prepare(case, seed):
    prec = PRECISION[case["precision"]]
    dtype = torch.float64 if prec == sb.FP64 else torch.float32
    sims, fields, outs, flat = [], [], [], []
    for b in _inputs(case, seed):
        f = tuple(FACES[x] for x in b["faces"])
        s = sb.Sim(b["n"], (case["h"],) * 3, f, cfl=case["cfl"], precision=prec, energy_every=case["energy_every"],
                   eps_r=None if b["eps"] is None else b["eps"].cpu().numpy(),
                   mu_r=None if b["mu"] is None else b["mu"].cpu().numpy())
        for src in b["sources"]:
            s.add_source(*src)
        for p in b["probes"]:
            s.add_probe(*p)
        if b["probes"]:
            s.reserve_probes(200000 if case["kind"] == "block" else 50000)
        for c in range(6):
            s.set_field(c, b["fields"][c])
        e = [_extents(b["n"], c) for c in range(6)]
        for part in (range(3), range(3, 6)):        # one array for E and one for H, a view per component
            size = [math.prod(e[c]) for c in part]
            a = torch.empty(sum(size), dtype=dtype, device="cuda")
            flat.append(a)
            outs += [v.view(e[c][2], e[c][1], e[c][0]) for v, c in zip(a.split(size), part)]
        fields.append(b["fields"] if case["kind"] == "periodic" else None)
        sims.append(s)
    batch = energy = None
    if case["kind"] == "joined":
        sims[0].connect(5, sims[1], 4)
    elif case["kind"] == "periodic":
        for axis, alpha in enumerate(_phases(seed)):
            sb.connect_phase(sims[0], sims[1], axis, alpha)
    elif case["kind"] == "batch":
        batch = sb.Batch()
        for s in sims:
            batch.add(s, 10 ** 9)
    if case["energy_every"]:
        energy = torch.zeros(1, dtype=torch.float64, device="cuda")
    if case["tune"]:
        sims[0].autotune()
    return {"case": case, "sims": sims, "fields": fields, "outs": outs, "flat": flat, "batch": batch, "energy": energy}


def run(state):
    sims, steps = state["sims"], state["case"]["steps"]
    if state["fields"][0] is not None:              # the periodic pair is written before each step
        for s, f in zip(sims, state["fields"]):
            for c in range(6):
                s.set_field(c, f[c])
    if state["batch"] is not None:
        state["batch"].step(steps)
    elif len(sims) > 1:
        sb.step_group(sims, steps)
    else:
        sims[0].step(steps)
    for i, s in enumerate(sims):
        for c in range(6):
            s.field(c, out=state["outs"][6 * i + c])
    if state["energy"] is not None:
        sims[0].energy_noalloc(state["energy"])
        return {"fields": state["flat"], "energy": state["energy"]}
    return {"fields": state["flat"]}


def work(case):
    """Per cell and step: six fields read and written and the cell's materials read once; about
    60 operations (two curls, the coefficients and the node's reciprocal)."""
    size = {"fp32": 4, "fp64": 8, "fp16": 2}[case["precision"]]
    if case["kind"] == "batch":
        cells = sum(nx * ny * nz for nx, ny, nz in _members(case))
    else:
        cells = case["nx"] * case["ny"] * case["nz"] * (1 if case["kind"] == "block" else 2)
    per = 12 * size + 4 + (4 if case["mu"] else 0)
    return {"bytes": cells * per * case["steps"], "flops": 60 * cells * case["steps"]}


# --- the same in 64 bits ----------------------------------------------------

def _dminus(u, ax, n):
    """x+ (n+1 values) to x- (n+2 rows) at unit spacing."""
    i = u.unbind(ax)
    rows = u.narrow(ax, 1, n) - u.narrow(ax, 0, n)          # rows 1..n
    out = torch.cat([rows.narrow(ax, 0, 1), rows, rows.narrow(ax, n - 1, 1)], ax)
    out.select(ax, 2).copy_((4 * i[2] - 3 * i[1] - i[0]) / 5)
    out.select(ax, n - 1).copy_((i[n] + 3 * i[n - 1] - 4 * i[n - 2]) / 5)
    return out


def _dplus(v, ax, n):
    """x- (n+2 values) to x+ (n+1 rows) at unit spacing."""
    i = v.unbind(ax)
    out = v.narrow(ax, 1, n + 1) - v.narrow(ax, 0, n + 1)
    out.select(ax, 0).copy_((i[1] + i[2]) / 2 - i[0])
    out.select(ax, 1).copy_(0.75 * i[2] - 0.5 * i[0] - 0.25 * i[1])
    out.select(ax, n - 1).copy_(0.25 * i[n] + 0.5 * i[n + 1] - 0.75 * i[n - 1])
    out.select(ax, n).copy_(i[n + 1] - 0.5 * (i[n - 1] + i[n]))
    return out


def _node(cells, c, n):
    """Mean of the cells that touch each node of component c."""
    if cells is None:
        return torch.ones((1, 1, 1), dtype=torch.float64, device="cuda").expand(*_extents(n, c)[::-1])
    v = cells.double()
    for a in range(3):
        ax = 2 - a
        v = torch.cat([v.narrow(ax, 0, 1), v, v.narrow(ax, n[a] - 1, 1)], ax)
        if ON_PLUS[c][a]:
            v = 0.5 * (v.narrow(ax, 0, n[a] + 1) + v.narrow(ax, 1, n[a] + 1))
    return v


def _wave(kind, t, tw, t0):
    x = (t - t0) / tw
    g = math.exp(-4 * math.pi * x * x)
    return g if kind == sb.GAUSS else -math.sqrt(8 * math.pi) * x * math.exp(0.5) * g


def _half(blocks, F, b, c, h, dt, m, partner):
    """The new values of component c of block b: curl, face penalties, absorbing self terms."""
    B = blocks[b]
    n, electric = B["n"], c < 3
    eps, mu = B["node_eps"][c], B["node_mu"][c]
    coef = dt / ((EPS0 * eps if electric else MU0 * mu) * h)
    acc = gam = None
    for t, (u, a) in enumerate(CURL[c]):
        sg, ax = (1.0, -1.0)[t], 2 - a
        d = (_dplus if electric else _dminus)(F[b][u], ax, n[a])
        acc = sg * d if acc is None else acc.add_(d, alpha=sg)
        for side in (-1, 1):
            here = 0 if side < 0 else acc.shape[ax] - 1      # the face node of c
            there = 0 if side < 0 else F[b][u].shape[ax] - 1  # and of the field it reads
            kind, phi = B["faces"][2 * a + (side > 0)], -sg * side
            pv = F[b][u].select(ax, there)
            if kind == ("M" if electric else "P"):
                acc.select(ax, here).add_(pv, alpha=2 * phi)
            elif kind == "A":
                acc.select(ax, here).add_(pv, alpha=phi)
                eta = math.sqrt(MU0 / EPS0) * torch.sqrt(mu.select(ax, here) / eps.select(ax, here))
                g = 0.5 * coef.select(ax, here) * (1 / eta if electric else eta)
                gam = torch.zeros_like(acc) if gam is None else gam
                gam.select(ax, here).add_(g)
            elif kind == "I":
                acc.select(ax, here).add_(pv - partner(b, u, a, side), alpha=phi)
    acc *= coef
    for s in B["sources"] if electric else ():
        if s[0] == c:
            J = s[5] * _wave(s[4], (m + 0.5) * dt, s[6], s[7])
            at = tuple(slice(None) if v < 0 else slice(v, v + 1) for v in (s[3], s[2], s[1]))
            acc[at] -= dt / EPS0 * J / eps[at]
    old = F[b][c]
    return old + acc if gam is None else ((1 - gam) * old + acc) / (1 + gam)


def _energy(B, F, Hnew, h):
    n, W = B["n"], 0.0
    for c in range(6):
        v = F[c] ** 2 * B["node_eps"][c] * EPS0 if c < 3 else F[c] * Hnew[c - 3] * B["node_mu"][c] * MU0
        for a in range(3):
            w = torch.ones(_extents(n, c)[a], dtype=torch.float64, device="cuda")
            w[0] = w[-1] = 0.5
            if not ON_PLUS[c][a]:
                w[1] = w[-2] = 0.25
                w[2] = w[-3] = 1.25
            v = v * w.view([-1 if 2 - a == q else 1 for q in range(3)])
        W += 0.5 * v.sum() * h ** 3
    return W.reshape(1)


def exact(case, seed):
    blocks, h = _inputs(case, seed), case["h"]
    dt = case["cfl"] * h / (C0 * math.sqrt(3.0))
    for B in blocks:
        B["node_eps"] = [_node(B["eps"], c, B["n"]) for c in range(6)]
        B["node_mu"] = [_node(B["mu"], c, B["n"]) for c in range(6)]
        if case["kind"] == "periodic":
            B["faces"] = "IIIIII"
    F = [[f.double() for f in B["fields"]] for B in blocks]
    phases = _phases(seed)

    def partner(b, u, a, side):
        """What an interface face is compared with: the joined block's face, or the opposite face of
        the complex pair times exp(-j alpha) (high face) or exp(+j alpha) (low face)."""
        end = -1 if side < 0 else 0
        if case["kind"] == "joined":
            return F[1 - b][u].select(2 - a, end)
        c, s = math.cos(phases[a]), math.sin(phases[a]) * side * (1 if b == 0 else -1)
        return c * F[b][u].select(2 - a, end) + s * F[1 - b][u].select(2 - a, end)

    for m in range(case["steps"]):
        for comps in ((3, 4, 5), (0, 1, 2)):
            if case["kind"] == "batch":             # independent blocks
                for b in range(len(blocks)):
                    new = [_half(blocks, F, b, c, h, dt, m, partner) for c in comps]
                    F[b][comps[0]:comps[0] + 3] = new
                continue
            new = [[_half(blocks, F, b, c, h, dt, m, partner) for c in comps] for b in range(len(blocks))]
            for b, v in enumerate(new):
                F[b][comps[0]:comps[0] + 3] = v
    fields = []
    for f in F:
        fields += [torch.cat([v.reshape(-1) for v in f[:3]]), torch.cat([v.reshape(-1) for v in f[3:]])]
    if case["energy_every"]:
        new = [_half(blocks, F, 0, c, h, dt, case["steps"], partner) for c in (3, 4, 5)]
        return {"fields": fields, "energy": _energy(blocks[0], F[0], new, h)}
    return {"fields": fields}
