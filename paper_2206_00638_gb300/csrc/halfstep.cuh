// In-place half-steps (sm_103a): one launch updates every node of H, the next
// every node of E.
//
//   half_h  H^{n+1/2} = H^{n-1/2} + dt/mu (D- E^n) + SAT_H      Eqs. (10)-(15), Alg. 2
//   half_e  E^{n+1}   = E^n + dt/eps (D+ H^{n+1/2} - J) + SAT_E Eqs. (7)-(9), (19)-(21), Alg. 1
//
// The nodes of a block are dealt to two kinds of CTAs of one launch.
//   - Box CTAs: the nodes whose rows are two-point rows along every axis and
//     meet no face.  A thread owns V neighbouring x nodes of one row (vector
//     loads and stores) and marches kz planes, carrying the z-neighbours and the
//     eps sums of the previous plane in registers.
//   - Rim CTAs: every node around the box, one per thread, x fastest.  The rows
//     of all three axes are three entries with coefficients, so one short code
//     serves faces, edges and corners; it loads everything a node needs before
//     it computes.  A grid's first wave is over in a few microseconds, and what
//     counts there is the longest chain of a rim thread: rim code that took
//     four nodes per thread, or called its penalties one after the other, made
//     a 61x47x38 half-step 6 us long where the box alone takes 2.
// Threads are dealt over (row, vector) pairs without gaps, so narrow grids fill
// their warps.  The rim of a plane is listed next to the box CTAs of the same
// planes: an end node sits in a DRAM unit that the box part of its row reads as
// well, and so finds it in L2.
#pragma once
#include "fused.cuh"

namespace sbp {

constexpr int kSweepThreads = 128;        // threads of a CTA

// CTAs of a half-step that fit an SM, by registers: 72 a thread in FP32 (76-80 left
// to the compiler cost 8 % at 117 x 96 x 131; E in vectors of 4, which would take
// 96: 1048 us per step at 512^3 in FP16 storage, 997 at 80 registers, 964 at 72),
// 112 and more in FP64.
template <typename T> constexpr int kHalfCtas = sizeof(T) == 8 ? 4 : 7;

// n / d for n < 2^31, with the multiplier of d found on the host.
struct FastDiv { unsigned mul, shift; };
__device__ __forceinline__ unsigned operator/(unsigned n, const FastDiv &d) { return (__umulhi(n, d.mul) + n) >> d.shift; }

// n / d, for counts of rim nodes: 32-bit ones through the multiplier, 64-bit ones
// (steps with 64-bit indices, whose layer planes may hold 2^31 nodes) by division.
__device__ __forceinline__ unsigned quotient(unsigned n, unsigned, const FastDiv &f) { return n / f; }
__device__ __forceinline__ unsigned long long quotient(unsigned long long n, unsigned d, const FastDiv &) { return n / d; }

// Work list of one in-place half-step launch.
struct Sweep {
    int lo[3], hi[3];         // the box, inclusive per axis; empty along an axis when hi < lo
    int kz;                   // planes per z-chunk
    unsigned nv, vecs;        // vectors per row and per plane of the box
    unsigned xs, rows;        // nodes per row and rows of a whole plane
    unsigned ends;            // nodes of a row left and right of the box
    unsigned zplanes;         // planes below and above the box
    unsigned ynodes, rim;     // rim nodes of a box plane: y layers, in all
    unsigned cz;              // CTAs of the planes below and above the box (first in the list)
    unsigned cbox, cchunk;    // box CTAs and all CTAs of a z-chunk
    unsigned flip;            // last chunk when the chunks are taken from the last to the first, else 0
    unsigned ctas;
    FastDiv dnv, dxs, drows, dends, drim, dchunk;
};

// --- programmatic dependent launch -----------------------------------------
// Each half-step lets the next one start as soon as all of its own CTAs run,
// and waits for the previous one before it touches a field: the launch latency
// (about a third of a small grid's half-step) overlaps the running kernel.
__device__ __forceinline__ void pdl_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// --- vector access ----------------------------------------------------------
template <int V, typename S>
__device__ __forceinline__ void ldv(const S *p, compute_t<S> (&v)[V])
{
    constexpr int bytes = V * (int)sizeof(S);
    if constexpr (V == 1) {
        v[0] = ld_s(p);
    } else {
        static_assert(bytes == 8 || bytes == 16, "vector width");
        using W = typename std::conditional<bytes == 16, uint4, uint2>::type;
        union { W w; S s[V]; } u;
        u.w = *reinterpret_cast<const W *>(p);
#pragma unroll
        for (int q = 0; q < V; ++q) {
            if constexpr (std::is_same<S, __half>::value) v[q] = __half2float(u.s[q]);
            else v[q] = u.s[q];
        }
    }
}
// Store v (already rounded to the storage type).
template <int V, typename S, typename T>
__device__ __forceinline__ void stv(S *p, const T (&v)[V])
{
    if constexpr (V == 1) {
        st_s(p, v[0]);
    } else {
        using W = typename std::conditional<V * sizeof(S) == 16, uint4, uint2>::type;
        union { W w; S s[V]; } u;
#pragma unroll
        for (int q = 0; q < V; ++q) {
            if constexpr (std::is_same<S, __half>::value) u.s[q] = __float2half_rn(v[q]);
            else u.s[q] = v[q];
        }
        *reinterpret_cast<W *>(p) = u.w;
    }
}
// Cell values (FP32) in the arithmetic type.
template <int V, typename T>
__device__ __forceinline__ void ldcells(const float *p, T (&v)[V])
{
    float f[V];
    if constexpr (V == 4) {
        const float4 w = __ldg(reinterpret_cast<const float4 *>(p));
        f[0] = w.x; f[1] = w.y; f[2] = w.z; f[3] = w.w;
    } else if constexpr (V == 2) {
        const float2 w = __ldg(reinterpret_cast<const float2 *>(p));
        f[0] = w.x; f[1] = w.y;
    } else {
        f[0] = __ldg(p);
    }
#pragma unroll
    for (int q = 0; q < V; ++q) v[q] = widen<T>(f[q]);
}

// old + increment of two curl terms, in the rounding order of the general path.
// (FP64 too: adding the terms to the old value one by one saves an operation of
// three and rounds twice at the field's size.)
template <typename S, typename T>
__device__ __forceinline__ T advance_plain(T old, const Coef<T> &c0, T d0, const Coef<T> &c1, T d1)
{
    typename AccOf<T, S>::type a;
    a.add(c0, d0);
    a.add(c1, d1, T(-1));
    return old + plain_increment(a);
}

// Step index and probe sample slot of a launch.
struct When { long long step, slot; };

// Sources and probes that some node of a warp may hold: source values (null for
// none) and a bit per probe.
struct Marks { const double *J; unsigned long long pm; };

__device__ __forceinline__ bool meets(const int (&box)[6], int i0, int i1, int j, int k0, int k1)
{
    return i0 <= box[3] && i1 >= box[0] && j <= box[4] && j >= box[1] && k0 <= box[5] && k1 >= box[2];
}

// The marks of a warp whose lanes hold nodes i0..i1 of row j in planes k0..k1.
// Nearly every warp is done after the test against the index boxes around all
// probes and all sources.  Every lane of the warp calls it.
template <bool ELECTRIC, typename T, typename S>
__device__ __forceinline__ Marks find_marks(const Params<T, S> &p, When when, int i0, int i1, int j, int k0, int k1)
{
    Marks r = {nullptr, 0ull};
    const bool near_p = meets(p.pbox[ELECTRIC ? 0 : 1], i0, i1, j, k0, k1);
    const bool near_s = ELECTRIC && meets(p.sbox, i0, i1, j, k0, k1);
    if (!__any_sync(0xffffffffu, near_p || near_s)) return r;
    constexpr int c0 = ELECTRIC ? 0 : 3;
    const int lane = threadIdx.x & 31;
    const int ja = __reduce_min_sync(0xffffffffu, j), jb = __reduce_max_sync(0xffffffffu, j);
    k0 = __reduce_min_sync(0xffffffffu, k0);
    k1 = __reduce_max_sync(0xffffffffu, k1);
    for (int q0 = 0; q0 < p.nprb; q0 += 32) {
        const int q = q0 + lane;
        bool hit = false;
        if (q < p.nprb) {
            const Prb P = p.prb[q];
            hit = P.comp >= c0 && P.comp <= c0 + 2 && P.k >= k0 && P.k <= k1 && P.j >= ja && P.j <= jb;
        }
        r.pm |= (unsigned long long)__ballot_sync(0xffffffffu, hit) << q0;
    }
    if (ELECTRIC) r.J = source_values(p, when.step, lane, k0, k1, ja, jb, 0, INT32_MAX);
    return r;
}

template <int V, typename T, typename S>
__device__ __forceinline__ void vec_probes(const Params<T, S> &p, When t, unsigned long long m, int c0, int i0, int j, int k,
                                           const T (&a)[V], const T (&b)[V], const T (&c)[V])
{
    for (; m; m &= m - 1) {
        const int q = __ffsll((long long)m) - 1;
        const Prb &P = p.prb[q];
        if (P.j != j || P.k != k || t.slot >= p.probe_cap) continue;
#pragma unroll
        for (int e = 0; e < V; ++e)
            if (P.i == i0 + e)
                p.probe_buf[(long long)q * p.probe_cap + t.slot] =
                    (P.comp == c0 ? a[e] : P.comp == c0 + 1 ? b[e] : c[e]) * p.fscale[c0 >= 3];
    }
}

// First x, row and plane range of a box thread.
struct VecPlace { int i0, j, k0, k1; bool valid; };

template <int V>
__device__ __forceinline__ VecPlace vec_place(const Sweep &w, unsigned cta, int chunk)
{
    VecPlace r;
    const unsigned t = cta * (unsigned)kSweepThreads + threadIdx.x;
    r.valid = t < w.vecs;
    const unsigned tc = min(t, w.vecs - 1u), row = tc / w.dnv;
    r.j = w.lo[1] + (int)row;
    r.i0 = w.lo[0] + V * (int)(tc - row * w.nv);
    r.k0 = max(chunk * w.kz, w.lo[2]);
    r.k1 = min(chunk * w.kz + w.kz - 1, w.hi[2]);
    return r;
}

// I: the type of an element index (unsigned, or long long for arrays of 2^32
// elements and more; unsigned sums wrap, so offsets may be negative).  One
// 32-bit addition and one widening multiply-add make an address, where 64-bit
// sums take twice that, and the half-steps of grids that stay in L2 are bound by
// their instructions.
template <typename I, typename T, typename S, bool MUVAR, int V>
__device__ __forceinline__ void box_h(const Params<T, S> &p, const Sweep &w, When when, unsigned cta, int chunk)
{
    const VecPlace r = vec_place<V>(w, cta, chunk);
    if (r.k0 > r.k1) return;
    const unsigned long long pm = find_marks<false>(p, when, r.i0, r.i0 + V - 1, r.j, r.k0, r.k1).pm;
    if (!r.valid) return;
    const I sy = (I)p.sy, sz = (I)p.sz;
    I o = (I)r.k0 * sz + (I)r.j * sy + (I)r.i0;
    const S *const Ex = p.F[0], *const Ey = p.F[1], *const Ez = p.F[2];
    S *const Hx = p.F[3], *const Hy = p.F[4], *const Hz = p.F[5];
    const Coef<T> Bx = p.B[0], By = p.B[1], Bz = p.B[2];
    pdl_wait();
    T exm[V], eym[V], m0[V];
    ldv<V>(Ex + (I)(o - sz), exm);
    ldv<V>(Ey + (I)(o - sz), eym);
    if constexpr (MUVAR) ldcells<V>(p.mu + o, m0);
    for (int k = r.k0; k <= r.k1; ++k, o += sz) {
        T ex[V], ey[V], ez[V], exj[V], ezj[V], hx[V], hy[V], hz[V];
        const S *const pey = Ey + o, *const pez = Ez + o;
        const I oj = o - sy;
        ldv<V>(Ex + o, ex);
        ldv<V>(pey, ey);
        ldv<V>(pez, ez);
        ldv<V>(Ex + oj, exj);
        ldv<V>(Ez + oj, ezj);
        const T eyl = ld_s(pey - 1), ezl = ld_s(pez - 1);
        ldv<V>(Hx + o, hx);
        ldv<V>(Hy + o, hy);
        ldv<V>(Hz + o, hz);
        T mj[V], mk[V], mr = T(0);
        if constexpr (MUVAR) {
            ldcells<V>(p.mu + (I)(o + sy), mj);
            ldcells<V>(p.mu + (I)(o + sz), mk);
            mr = widen<T>(__ldg(p.mu + o + V));
        }
#pragma unroll
        for (int q = 0; q < V; ++q) {
            const T eyi = q ? ey[q - 1] : eyl, ezi = q ? ez[q - 1] : ezl;
            const T d0 = ey[q] - eym[q], d1 = ez[q] - ezj[q];       // Hx: Bz dEy/dz - By dEz/dy
            const T d2 = ez[q] - ezi, d3 = ex[q] - exm[q];          // Hy: Bx dEz/dx - Bz dEx/dz
            const T d4 = ex[q] - exj[q], d5 = ey[q] - eyi;          // Hz: By dEx/dy - Bx dEy/dx
            if constexpr (MUVAR) {
                const T mi = q + 1 < V ? m0[q + 1 < V ? q + 1 : q] : mr;
                typename AccOf<T, S>::type a, b, c;
                a.add(Bz, d0); a.add(By, d1, T(-1));
                b.add(Bx, d2); b.add(Bz, d3, T(-1));
                c.add(By, d4); c.add(Bx, d5, T(-1));
                hx[q] = quant<S>(hx[q] + scaled_increment(a, m0[q] + mi));
                hy[q] = quant<S>(hy[q] + scaled_increment(b, m0[q] + mj[q]));
                hz[q] = quant<S>(hz[q] + scaled_increment(c, m0[q] + mk[q]));
            } else {
                hx[q] = quant<S>(advance_plain<S>(hx[q], Bz, d0, By, d1));
                hy[q] = quant<S>(advance_plain<S>(hy[q], Bx, d2, Bz, d3));
                hz[q] = quant<S>(advance_plain<S>(hz[q], By, d4, Bx, d5));
            }
        }
        stv<V>(Hx + o, hx);
        stv<V>(Hy + o, hy);
        stv<V>(Hz + o, hz);
        if (pm) vec_probes<V>(p, when, pm, 3, r.i0, r.j, k, hx, hy, hz);
#pragma unroll
        for (int q = 0; q < V; ++q) {
            exm[q] = ex[q];
            eym[q] = ey[q];
            if constexpr (MUVAR) m0[q] = mk[q];
        }
    }
}

// Pair sums of the eps cells (j, j+1; i, i+1) of one plane, from which the node
// sums of cell_sum are built in its association.
template <int V, typename I, typename T>
__device__ __forceinline__ void eps_pairs(const float *eps, I o, I sy, T (&a)[V], T (&b)[V], T (&c)[V])
{
    T f[V], g[V];
    const float *const pf = eps + o, *const pg = eps + (I)(o + sy);
    ldcells<V>(pf, f);
    ldcells<V>(pg, g);
    const T fr = widen<T>(__ldg(pf + V)), gr = widen<T>(__ldg(pg + V));
#pragma unroll
    for (int q = 0; q < V; ++q) {
        const int n = q + 1 < V ? q + 1 : q;
        a[q] = f[q] + g[q];
        b[q] = f[q] + (q + 1 < V ? f[n] : fr);
        c[q] = g[q] + (q + 1 < V ? g[n] : gr);
    }
}

// The current density of the warp's sources on V nodes of the three components.
template <int V, typename T, typename S, typename A>
__device__ __forceinline__ void vec_sources(const Params<T, S> &p, const double *J, int i0, int j, int k, A (&a)[V],
                                            A (&b)[V], A (&c)[V])
{
    for (int s = 0; s < p.nsrc; ++s) {
        const Src &P = p.src[s];
        if ((P.k >= 0 && P.k != k) || (P.j >= 0 && P.j != j)) continue;
        const T v = T(J[s]);
#pragma unroll
        for (int q = 0; q < V; ++q) {
            if (P.i >= 0 && P.i != i0 + q) continue;
            if (P.comp == 0) a[q].add(p.AJ, v, T(-1));
            else if (P.comp == 1) b[q].add(p.AJ, v, T(-1));
            else c[q].add(p.AJ, v, T(-1));
        }
    }
}

template <typename I, typename T, typename S, int V>
__device__ __forceinline__ void box_e(const Params<T, S> &p, const Sweep &w, When when, unsigned cta, int chunk)
{
    const VecPlace r = vec_place<V>(w, cta, chunk);
    if (r.k0 > r.k1) return;
    const Marks marks = find_marks<true>(p, when, r.i0, r.i0 + V - 1, r.j, r.k0, r.k1);
    if (!r.valid) return;
    const I sy = (I)p.sy, sz = (I)p.sz;
    I o = (I)r.k0 * sz + (I)r.j * sy + (I)r.i0;
    S *const Ex = p.F[0], *const Ey = p.F[1], *const Ez = p.F[2];
    const S *const Hx = p.F[3], *const Hy = p.F[4], *const Hz = p.F[5];
    const Coef<T> Ax = p.A[0], Ay = p.A[1], Az = p.A[2];
    pdl_wait();
    T qa[V], qb[V], qc[V];
    eps_pairs<V>(p.eps, o, sy, qa, qb, qc);
    T hx[V], hy[V];
    ldv<V>(Hx + o, hx);
    ldv<V>(Hy + o, hy);
    T hyr = ld_s(Hy + o + V);
    for (int k = r.k0; k <= r.k1; ++k, o += sz) {
        T hxn[V], hyn[V], hz[V], hzj[V], hxj[V], ex[V], ey[V], ez[V], na[V], nb[V], nc[V];
        const I oz = o + sz, oj = o + sy;
        const S *const phy = Hy + oz, *const phz = Hz + o;
        ldv<V>(Hx + oz, hxn);
        ldv<V>(phy, hyn);
        const T hyrn = ld_s(phy + V), hzr = ld_s(phz + V);
        ldv<V>(phz, hz);
        ldv<V>(Hz + oj, hzj);
        ldv<V>(Hx + oj, hxj);
        ldv<V>(Ex + o, ex);
        ldv<V>(Ey + o, ey);
        ldv<V>(Ez + o, ez);
        eps_pairs<V>(p.eps, oz, sy, na, nb, nc);
        typename AccOf<T, S>::type a[V], b[V], c[V];
#pragma unroll
        for (int q = 0; q < V; ++q) {
            const int n = q + 1 < V ? q + 1 : q;
            const T hyi = q + 1 < V ? hy[n] : hyr, hzi = q + 1 < V ? hz[n] : hzr;
            a[q].add(Ay, hzj[q] - hz[q]); a[q].add(Az, hyn[q] - hy[q], T(-1));
            b[q].add(Az, hxn[q] - hx[q]); b[q].add(Ax, hzi - hz[q], T(-1));
            c[q].add(Ax, hyi - hy[q]);    c[q].add(Ay, hxj[q] - hx[q], T(-1));
        }
        if (marks.J) vec_sources<V>(p, marks.J, r.i0, r.j, k, a, b, c);
#pragma unroll
        for (int q = 0; q < V; ++q) {
            ex[q] = quant<S>(ex[q] + scaled_increment(a[q], qa[q] + na[q]));
            ey[q] = quant<S>(ey[q] + scaled_increment(b[q], qb[q] + nb[q]));
            ez[q] = quant<S>(ez[q] + scaled_increment(c[q], qb[q] + qc[q]));
        }
        stv<V>(Ex + o, ex);
        stv<V>(Ey + o, ey);
        stv<V>(Ez + o, ez);
        if (marks.pm) vec_probes<V>(p, when, marks.pm, 0, r.i0, r.j, k, ex, ey, ez);
#pragma unroll
        for (int q = 0; q < V; ++q) {
            hx[q] = hxn[q]; hy[q] = hyn[q];
            qa[q] = na[q]; qb[q] = nb[q]; qc[q] = nc[q];
        }
        hyr = hyrn;
    }
}

// --- rim CTAs ----------------------------------------------------------------
// One axis of a rim node: its D row there (offset of the first entry from the
// node, coefficients) and the face it lies on (side -1 / +1, 0 for none).
template <typename I, typename T> struct RimAxis {
    I off, st;
    T k[3];
    bool closure;             // a closure row: its third entry counts
    int side, type;
};

template <bool ELECTRIC, typename I, typename T, typename S>
__device__ __forceinline__ RimAxis<I, T> rim_axis(const Params<T, S> &p, int a, int r)
{
    const int n = p.n[a], last = n + (ELECTRIC ? 0 : 1);
    RimAxis<I, T> x;
    x.st = a == 0 ? I(1) : a == 1 ? (I)p.sy : (I)p.sz;
    if constexpr (ELECTRIC) dplus_coefs(r, n, x.k);
    else dminus_coefs(r, n, x.k);
    // (asked of the index, not of the coefficient: an FP64 comparison goes through the FP64 pipe)
    x.closure = ELECTRIC ? r <= 1 || r >= n - 1 : r == 2 || r == n - 1 || r == n + 1;
    x.off = (I)((ELECTRIC ? dplus_start(r, n) : dminus_start(r, n)) - r) * x.st;
    x.side = r == 0 ? -1 : r == last ? 1 : 0;
    x.type = x.side ? p.face[2 * a + (x.side > 0)] : (ELECTRIC ? kPEC : kPMC);   // the type without a penalty
    return x;
}

// The row on its entries.  A two-point row gives the same bits either way; FP64,
// whose pipe is the narrow one, takes the single subtraction.
template <typename I, typename T>
__device__ __forceinline__ T rim_row(const RimAxis<I, T> &x, const Tri<T> &v)
{
    if constexpr (std::is_same<T, double>::value)
        if (!x.closure) return v.b - v.a;
    return row_chain(x.k, v.a, v.b, v.c);
}

// Absorbing self term along axis a from the sums of the node's cells.  One copy,
// called: roots and divisions inlined at the six sites of the rim code made its
// warps wait for instruction fetch (cavity in FP64 21.3 -> 12.4 us per step,
// 121 x 101 x 88 with mu_r 20.8 -> 18.8, 512^3 in FP16 storage 1114 -> 1064).
template <typename T, typename S, bool ELECTRIC, bool MUVAR>
__device__ __noinline__ T rim_gamma(const Params<T, S> &p, int a, T se, T sm)
{
    if constexpr (ELECTRIC) {
        const T mr = MUVAR ? sm * T(0.25) : T(1);
        return abs_gamma_e(T(p.A[a].hi) * p.uA, se, node_eta(p.eta0, mr, se * T(0.25)));
    } else {
        const T er = se * T(0.5), mr = MUVAR ? sm * T(0.5) : T(1);
        const T ba = (MUVAR ? T(p.B[a].hi) * T(0.5) / mr : T(p.B[a].hi)) * p.uB;
        return abs_gamma_h(ba, node_eta(p.eta0, mr, er));
    }
}
// New value of component C at a rim node, in the operation order of h_apply /
// e_apply.  v[t]: the entries of the two curl terms; nv[t]: the partner's values on
// interface faces; se: sum of the node's eps cells (4 for E, 2 for H, there only
// read on an absorbing face).
template <typename T, int C, bool MUVAR, typename I, typename S>
__device__ __forceinline__ T rim_apply(const Params<T, S> &p, const RimAxis<I, T> (&ax)[3], const int (&idx)[3], T old,
                                       const Tri<T> (&v)[2], const T (&nv)[2], T se, T sm, const double *J)
{
    constexpr bool electric = C < 3;
    typename AccOf<T, S>::type acc;
    T gam = T(0);
#pragma unroll
    for (int t = 0; t < 2; ++t) {
        const int a = curl_axis(C, t), sg = curl_sign(t);
        const Coef<T> &cf = electric ? p.A[a] : p.B[a];
        acc.add(cf, rim_row(ax[a], v[t]), T(sg));
        if (ax[a].type == (electric ? kPEC : kPMC)) continue;
        const bool up = sg * ax[a].side < 0;           // phi = -sg * side
        T pv = ax[a].side < 0 ? v[t].a : v[t].c;
        if (ax[a].type == kIFACE) pv = pv - nv[t];
        acc.add(cf, pv, ax[a].type == (electric ? kPMC : kPEC) ? (up ? T(2) : T(-2)) : (up ? T(1) : T(-1)));
        if (ax[a].type == kABS) gam += rim_gamma<T, S, electric, MUVAR>(p, a, se, sm);
    }
    if (electric && J) {
        for (int s = 0; s < p.nsrc; ++s) {
            const Src &P = p.src[s];
            if (P.comp == C && (P.i < 0 || P.i == idx[0]) && (P.j < 0 || P.j == idx[1]) && (P.k < 0 || P.k == idx[2]))
                acc.add(p.AJ, T(J[s]), T(-1));
        }
    }
    const T inc = electric ? scaled_increment(acc, se) : MUVAR ? scaled_increment(acc, sm) : plain_increment(acc);
    return quant<S>(sat_finish(old, inc, gam));
}

// The entries of component C's two curl terms (a third entry only on closure rows).
template <int C, typename I, typename T, typename S>
__device__ __forceinline__ void rim_gather(const Params<T, S> &p, const RimAxis<I, T> (&ax)[3], I o, Tri<T> (&v)[2])
{
#pragma unroll
    for (int t = 0; t < 2; ++t) {
        const RimAxis<I, T> &x = ax[curl_axis(C, t)];
        const S *const F = p.F[curl_comp(C, t)];
        const I q = o + x.off;
        v[t].a = ld_s(F + q);
        v[t].b = ld_s(F + (I)(q + x.st));
        v[t].c = x.closure ? ld_s(F + (I)(q + x.st + x.st)) : T(0);
    }
}

// The partner's values of component C's two curl fields, where the term's axis
// faces an interface.  on: offsets of the node on the partner's faces per axis.
template <int C, typename I, typename T, typename S>
__device__ __forceinline__ void rim_partners(const Params<T, S> &p, const RimAxis<I, T> (&ax)[3], const long long (&on)[3],
                                             T (&nv)[2])
{
#pragma unroll
    for (int t = 0; t < 2; ++t) {
        const int a = curl_axis(C, t);
        if (ax[a].type == kIFACE)
            nv[t] = link_value<false, T, S>(p.link[2 * a + (ax[a].side > 0)], curl_comp(C, t), on[a]);
    }
}

// Sums of the cells around a node of the three E components (four cells each) or
// the three H components (two each), in the association of cell_sum.
template <bool ELECTRIC, typename I, typename T>
__device__ __forceinline__ void rim_cells(const float *m, I o, I sy, I sz, T &x, T &y, T &z)
{
    const float *const py = m + (I)(o + sy), *const pz = m + (I)(o + sz);
    const T c = widen<T>(__ldg(m + o)), cx = widen<T>(__ldg(m + o + 1)), cy = widen<T>(__ldg(py));
    const T cz = widen<T>(__ldg(pz));
    if constexpr (ELECTRIC) {
        const T cxy = widen<T>(__ldg(py + 1)), cxz = widen<T>(__ldg(pz + 1));
        const T cyz = widen<T>(__ldg(m + (I)(o + sy + sz)));
        x = (c + cy) + (cz + cyz);
        y = (c + cx) + (cz + cxz);
        z = (c + cx) + (cy + cxy);
    } else {
        x = c + cx;
        y = c + cy;
        z = c + cz;
    }
}

// One rim node of a half-step, its new values to `out` (in place, or the new set
// of a one-pass step).  One code for every rim node: variants for the
// row ends and for the layers took a quarter fewer instructions and 15 % more
// time, waiting for instruction fetch.
template <typename I, typename T, typename S, bool ELECTRIC, bool MUVAR>
__device__ __forceinline__ void rim_node(const Params<T, S> &p, S *const (&out)[3], When when, int i, int j, int k,
                                         Marks marks)
{
    constexpr int c0 = ELECTRIC ? 0 : 3;
    const int idx[3] = {i, j, k};
    const RimAxis<I, T> ax[3] = {rim_axis<ELECTRIC, I, T>(p, 0, i), rim_axis<ELECTRIC, I, T>(p, 1, j),
                                 rim_axis<ELECTRIC, I, T>(p, 2, k)};
    const I sy = (I)p.sy, sz = (I)p.sz, o = (I)k * sz + (I)j * sy + (I)i;
    const int nx = p.n[0], ny = p.n[1], nz = p.n[2];
    const bool abs = ax[0].type == kABS || ax[1].type == kABS || ax[2].type == kABS;
    pdl_wait();
    Tri<T> vx[2], vy[2], vz[2];
    rim_gather<c0>(p, ax, o, vx);
    rim_gather<c0 + 1>(p, ax, o, vy);
    rim_gather<c0 + 2>(p, ax, o, vz);
    T x = ld_s(p.F[c0] + o), y = ld_s(p.F[c0 + 1] + o), z = ld_s(p.F[c0 + 2] + o);
    // partner values with the other loads: fetched one by one where each is used,
    // they were most of a small periodic pair's half-step
    T nx2[2] = {T(0), T(0)}, ny2[2] = {T(0), T(0)}, nz2[2] = {T(0), T(0)};
    if (ax[0].type == kIFACE || ax[1].type == kIFACE || ax[2].type == kIFACE) {
        long long on[3] = {0, 0, 0};
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            if (ax[a].type != kIFACE) continue;
            const Link &L = p.link[2 * a + (ax[a].side > 0)];
            const int nidx = L.side < 0 ? 0 : ELECTRIC ? L.n_norm + 1 : L.n_norm;
            on[a] = (long long)(a == 0 ? nidx : i) + (long long)(a == 1 ? nidx : j) * L.sy +
                    (long long)(a == 2 ? nidx : k) * L.sz;
        }
        rim_partners<c0>(p, ax, on, nx2);
        rim_partners<c0 + 1>(p, ax, on, ny2);
        rim_partners<c0 + 2>(p, ax, on, nz2);
    }
    T ex = T(0), ey = T(0), ez = T(0), mx = T(0), my = T(0), mz = T(0);
    // the last plane repeats its own cells: no component there spans two cells along z,
    // and the arrays' slack plane does not hold a step along y and z together
    const I dz = k <= nz ? sz : I(0);
    if (ELECTRIC || abs) rim_cells<ELECTRIC>(p.eps, o, sy, dz, ex, ey, ez);
    if (MUVAR && (!ELECTRIC || abs)) rim_cells<ELECTRIC>(p.mu, o, sy, dz, mx, my, mz);
    x = rim_apply<T, c0, MUVAR>(p, ax, idx, x, vx, nx2, ex, mx, marks.J);
    y = rim_apply<T, c0 + 1, MUVAR>(p, ax, idx, y, vy, ny2, ey, my, marks.J);
    z = rim_apply<T, c0 + 2, MUVAR>(p, ax, idx, z, vz, nz2, ez, mz, marks.J);
    // nodes of each component (Table I); the others are not stored and hold no probe
    const int e = ELECTRIC ? 1 : 0;
    if (i <= nx + e && j <= ny + 1 - e && k <= nz + 1 - e) st_s(out[0] + o, x);
    if (i <= nx + 1 - e && j <= ny + e && k <= nz + 1 - e) st_s(out[1] + o, y);
    if (i <= nx + 1 - e && j <= ny + 1 - e && k <= nz + e) st_s(out[2] + o, z);
    if (marks.pm) {
        const T a[1] = {x}, b[1] = {y}, c[1] = {z};
        vec_probes<1>(p, when, marks.pm, c0, i, j, k, a, b, c);
    }
}

// Rim CTAs: the planes below and above the box first, then per z-chunk the y
// layers and the row ends of its box planes.
template <typename I, typename T, typename S, bool ELECTRIC, bool MUVAR>
__device__ __forceinline__ void sweep_rim(const Params<T, S> &p, const Sweep &w, S *const (&out)[3], When when, unsigned cta,
                                          unsigned q, int chunk)
{
    using N = typename std::conditional<std::is_same<I, unsigned>::value, unsigned, unsigned long long>::type;
    N t, count;
    int i, j, k;
    if (cta < w.cz) {
        t = (N)cta * (N)kSweepThreads + threadIdx.x;
        count = (N)w.zplanes * w.rows * w.xs;
        if ((t & ~(N)31) >= count) return;
        const N tc = min(t, count - 1), row = quotient(tc, w.xs, w.dxs), pl = quotient(row, w.rows, w.drows);
        i = (int)(tc - row * w.xs);
        j = (int)(row - pl * w.rows);
        k = (int)pl < w.lo[2] ? (int)pl : w.hi[2] + 1 + ((int)pl - w.lo[2]);
    } else {
        const int kb = max(chunk * w.kz, w.lo[2]), ke = min(chunk * w.kz + w.kz - 1, w.hi[2]);
        if (kb > ke) return;
        t = (N)(q - w.cbox) * (N)kSweepThreads + threadIdx.x;
        count = (N)(ke - kb + 1) * w.rim;
        if ((t & ~(N)31) >= count) return;
        const N tc = min(t, count - 1), pl = quotient(tc, w.rim, w.drim), u = tc - pl * w.rim;
        k = kb + (int)pl;
        if (u < w.ynodes) {
            const N row = quotient(u, w.xs, w.dxs);
            i = (int)(u - row * w.xs);
            j = (int)row < w.lo[1] ? (int)row : w.hi[1] + 1 + ((int)row - w.lo[1]);
        } else {
            const N row = quotient(u - w.ynodes, w.ends, w.dends), e = u - w.ynodes - row * w.ends;
            i = (int)e < w.lo[0] ? (int)e : w.hi[0] + 1 + ((int)e - w.lo[0]);
            j = w.lo[1] + (int)row;
        }
    }
    const Marks marks = find_marks<ELECTRIC>(p, when, i, i, j, k, k);
    if (t < count) rim_node<I, T, S, ELECTRIC, MUVAR>(p, out, when, i, j, k, marks);
}

// CTA `cta` of a half-step's work list.
template <bool ELECTRIC, bool MUVAR, int V, typename I, typename T, typename S>
__device__ __forceinline__ void half_cta(const Params<T, S> &p, const Sweep &w, When when, unsigned cta)
{
    const unsigned r = cta < w.cz ? 0u : cta - w.cz, c = r / w.dchunk, q = r - c * w.cchunk;
    const unsigned chunk = w.flip ? w.flip - c : c;
    if (cta >= w.cz && q < w.cbox) {
        if constexpr (ELECTRIC) box_e<I, T, S, V>(p, w, when, q, (int)chunk);
        else box_h<I, T, S, MUVAR, V>(p, w, when, q, (int)chunk);
    } else {
        constexpr int c0 = ELECTRIC ? 0 : 3;
        S *const out[3] = {p.F[c0], p.F[c0 + 1], p.F[c0 + 2]};
        sweep_rim<I, T, S, ELECTRIC, MUVAR>(p, w, out, when, cta, q, (int)chunk);
    }
}

// The nodes of a half-step that the one-pass kernel leaves out (a work list
// without box CTAs), from the old set to the new one.
//
// One node per thread with every load first, where the slab kernels (band_h,
// band_e) took a warp's nodes through code for its slab with 64-bit addresses: at
// 512^3 130 + 140 us a step alone (157 + 170 before), beside the one-pass kernel
// the step takes 1423 us (1471).
template <bool ELECTRIC, typename S>
__global__ void __launch_bounds__(kSweepThreads, 7)
    rim_step(const __grid_constant__ Params<float, S> p, const __grid_constant__ Sweep w, S *x, S *y, S *z)
{
    const unsigned cta = blockIdx.x, r = cta < w.cz ? 0u : cta - w.cz, chunk = r / w.dchunk, q = r - chunk * w.cchunk;
    S *const out[3] = {x, y, z};
    sweep_rim<unsigned, float, S, ELECTRIC, false>(p, w, out, {p.step, p.probe_slot}, cta, q, (int)chunk);
}

template <typename I, typename T, typename S, bool MUVAR, int V>
__global__ void __launch_bounds__(kSweepThreads, kHalfCtas<T>)
    half_h(const __grid_constant__ Params<T, S> p, const __grid_constant__ Sweep w)
{
    pdl_release();
    half_cta<false, MUVAR, V, I>(p, w, {p.step, p.probe_slot}, blockIdx.x);
}

template <typename I, typename T, typename S, bool MUVAR, int V>
__global__ void __launch_bounds__(kSweepThreads, kHalfCtas<T>)
    half_e(const __grid_constant__ Params<T, S> p, const __grid_constant__ Sweep w)
{
    pdl_release();
    half_cta<true, MUVAR, V, I>(p, w, {p.step, p.probe_slot}, blockIdx.x);
}

// ---------------------------------------------------------------------------
// Batched half-steps: one launch advances every grid of a group of a batch.  A
// CTA finds its grid in a prefix table of CTA counts and copies the grid's
// parameters to shared memory (one round trip, before it waits for the launch
// before it); the step index comes from a device counter, so a captured chunk
// of K steps can be replayed (its launches carry offsets 0..K-1, batch_advance
// adds the steps taken).  Grids that reached their target step skip their work,
// so a chunk may end a grid early; their CTAs wait all the same, since what comes
// after the launch is ordered behind the launch before it by that wait alone.
//
// The grids of a batch are independent, so a chunk need not take every grid
// through a step before the next: it takes a group of grids, as many as stay in
// L2 together, through all its steps, then the next group.
// ---------------------------------------------------------------------------
struct alignas(16) BatchSweep : Sweep {};
static_assert(sizeof(BatchSweep) % 16 == 0, "copied in 16-byte units");

struct alignas(16) BatchHalf {
    alignas(16) Params<float> p;  // the member's fields, in place (step and probe slot come from the counter)
    BatchSweep w[2];              // work lists of H and E
    const long long *counter;     // steps taken (device)
    long long target;             // the grid stops when the counter reaches this
    long long probe_base;
};

// Vectors of 2: a member of the 2.5 M nodes from which vectors of 4 pay steps alone.
constexpr int kBatchV = 2;

template <bool ELECTRIC>
__global__ void __launch_bounds__(kSweepThreads, kHalfCtas<float>)
    half_batched(const BatchHalf *grids, const int *pre, int n, int offset)
{
    __shared__ __align__(16) Params<float> p;
    __shared__ BatchSweep w;
    pdl_release();
    // the tables and counters were written before the chunk's first launch, which
    // waited for them whole: they can be read while the launch before runs
    const int first = pre[0], g = find_slot(pre, n, (int)blockIdx.x + first);
    const BatchHalf &B = grids[g];
    auto copy = [](void *dst, const void *src, int bytes) {
        for (int q = threadIdx.x; q < bytes / 16; q += kSweepThreads)
            static_cast<uint4 *>(dst)[q] = __ldg(static_cast<const uint4 *>(src) + q);
    };
    copy(&p, &B.p, ((int)offsetof(Params<float>, link) + 15) / 16 * 16);   // members have no links
    copy(&w, &B.w[ELECTRIC], sizeof(w));
    const long long step = *B.counter + offset;
    if (step >= B.target) { pdl_wait(); return; }
    __syncthreads();
    half_cta<ELECTRIC, false, kBatchV, unsigned>(p, w, {step, step - B.probe_base}, (unsigned)((int)blockIdx.x + first - pre[g]));
}

// One member of a batch alone: its parameters are the launch's, which cost a CTA
// no copy (a grid that fills the GPU by itself steps 1.3 times faster so).
template <bool ELECTRIC, int V>
__global__ void __launch_bounds__(kSweepThreads, kHalfCtas<float>)
    half_member(const __grid_constant__ Params<float> p, const __grid_constant__ Sweep w, const long long *counter,
                long long target, long long probe_base, int offset)
{
    pdl_release();
    const long long step = *counter + offset;
    if (step >= target) { pdl_wait(); return; }
    half_cta<ELECTRIC, false, V, unsigned>(p, w, {step, step - probe_base}, blockIdx.x);
}

// The members' step counters after a chunk of k steps.
__global__ void batch_advance(long long *counters, const long long *targets, int n, long long k)
{
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= n) return;
    const long long c = counters[g], t = targets[g];
    counters[g] = c + k < t ? c + k : (c < t ? t : c);
}

}  // namespace sbp
