"""The in-place half-steps' work list on the CPU: the box, layer and end items of a launch, by the
index arithmetic of make_sweep (host) and box / rim placement (device), cover every node of the
padded block exactly once, over grids from the smallest up and past each vector remainder."""
import itertools

import numpy as np
import pytest

THREADS = 128


def fast_div(d):
    sh = 0
    while (1 << sh) < d:
        sh += 1
    mul = ((1 << 32) * ((1 << sh) - d)) // d + 1
    assert mul < 1 << 32
    return lambda n: (((n * mul) >> 32) + n) >> sh


def cover(n, electric, v, kz, onepass=False):
    lo, hi, box = [0] * 3, [0] * 3, [0] * 3
    for a in range(3):
        low, high = (2 if electric else 3), n[a] - 2
        lo[a] = low if a else (low + v - 1) // v * v
        hi[a] = max(high if a else (high + 1) // v * v - 1, lo[a] - 1)
        if onepass:
            lo[a], hi[a] = (3 if electric else 4), n[a] - 3
        box[a] = hi[a] - lo[a] + 1
    nv, planes, rows, xs = box[0] // v, n[2] + 2, n[1] + 2, n[0] + 2
    assert box[0] % v == 0
    vecs, zplanes, ynodes, ends = nv * box[1], planes - box[2], (rows - box[1]) * xs, xs - box[0]
    rim = ynodes + ends * box[1]
    ctas_of = lambda items: (items + THREADS - 1) // THREADS
    cz, cbox = ctas_of(zplanes * rows * xs), 0 if onepass else ctas_of(vecs)
    cchunk = cbox + ctas_of(kz * rim)
    chunks = (planes + kz - 1) // kz
    dnv, dxs, drows = fast_div(max(nv, 1)), fast_div(xs), fast_div(rows)
    dends, drim, dchunk = fast_div(max(ends, 1)), fast_div(max(rim, 1)), fast_div(cchunk)
    hits = np.zeros((planes, rows, xs), dtype=int)
    for cta in range(cz + cchunk * chunks):
        r = 0 if cta < cz else cta - cz
        chunk = dchunk(r)
        q = r - chunk * cchunk
        kb, ke = max(chunk * kz, lo[2]), min(chunk * kz + kz - 1, hi[2])
        if cta >= cz and q < cbox:
            for t in range(q * THREADS, min((q + 1) * THREADS, vecs)):
                row = dnv(t)
                i, j = lo[0] + v * (t - row * nv), lo[1] + row
                assert i % v == 0 and i + v - 1 <= hi[0]
                hits[kb:ke + 1, j, i:i + v] += 1
            continue
        if cta < cz:
            first, count = cta * THREADS, zplanes * rows * xs
        else:
            first, count = (q - cbox) * THREADS, max(ke - kb + 1, 0) * rim
        for t in range(first, min(first + THREADS, count)):
            if cta < cz:
                row = dxs(t)
                pl = drows(row)
                i, j = t - row * xs, row - pl * rows
                k = pl if pl < lo[2] else hi[2] + 1 + (pl - lo[2])
            else:
                pl = drim(t)
                u, k = t - pl * rim, kb + pl
                if u < ynodes:
                    row = dxs(u)
                    i, j = u - row * xs, row if row < lo[1] else hi[1] + 1 + (row - lo[1])
                else:
                    row = dends(u - ynodes)
                    e = u - ynodes - row * ends
                    i, j = e if e < lo[0] else hi[0] + 1 + (e - lo[0]), lo[1] + row
            hits[k, j, i] += 1
    return hits


SIZES = list(itertools.product((4, 5, 6, 7), (4, 5, 6), (4, 5, 7))) + \
    [(n, 9, 8) for n in range(8, 24)] + [(12, n, 6) for n in range(7, 13)] + [(33, 30, 29), (131, 6, 5)]


@pytest.mark.parametrize("v", [1, 2, 4])
@pytest.mark.parametrize("electric", [False, True])
def test_every_node_once(electric, v):
    for n in SIZES:
        for kz in (1, 3, 16):
            hits = cover(n, electric, v, kz)
            assert hits.min() == 1 and hits.max() == 1, (n, kz)


@pytest.mark.parametrize("electric", [False, True])
def test_one_pass_leaves_the_rim(electric):
    """Without box items: every node outside the one-pass box once, none inside."""
    for n in [(8, 8, 8), (9, 8, 11), (12, 17, 8), (34, 9, 10), (21, 30, 26)]:
        hits = cover(n, electric, 1, 4, onepass=True)
        lo, hi = (3 if electric else 4), [m - 3 for m in n]
        inner = hits[lo:hi[2] + 1, lo:hi[1] + 1, lo:hi[0] + 1]
        assert inner.max(initial=0) == 0 and hits.sum() == hits.size - inner.size and hits.max() == 1


def test_fast_division():
    rng = np.random.default_rng(1)
    for d in list(range(1, 300)) + [int(x) for x in rng.integers(1, 2 ** 31, 200)]:
        f = fast_div(d)
        for m in [0, 1, d - 1, d, d + 1, 2 ** 31 - 1] + [int(x) for x in rng.integers(0, 2 ** 31, 20)]:
            if m < 2 ** 31:
                assert f(m) == m // d
