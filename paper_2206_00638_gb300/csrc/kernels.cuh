// Device code of the GB300 SBP-SAT FDTD library (arXiv 2206.00638).
//
// This file holds what every kernel shares: the operator rows (Appendix) with
// their closure rows, the SAT penalties of the face types (PEC / PMC /
// absorbing / interface), node materials, sources and the arithmetic of one
// node, and the kernels that do not step: the energy, the copies of a field in
// and out of the padded layout, the coefficient build.  halfstep.cuh steps in
// place, one launch per half-step; fused.cuh steps the deep interior in one
// pass between two field sets.
//
// FP32 arithmetic keeps its coefficients exact to ~1e-14: every material
// coefficient dt/(eps h) is carried as an unevaluated sum hi + lo of two
// floats, and the node's 1/sum(eps_r) as a Newton-corrected reciprocal pair,
// so rounding of a coefficient does not bias the phase velocity; only the
// per-step rounding of the field update (unbiased) remains.
#pragma once
#include <cuda_fp16.h>

#include <cstdint>
#include <type_traits>

namespace sbp {

constexpr int kMaxSources = 16;
constexpr int kMaxProbes = 64;
constexpr int kBlockX = 32;
constexpr int kBlockY = 8;

enum : int { kPEC = 0, kPMC = 1, kABS = 2, kIFACE = 3 };

// Table I: component c lives on the plus grid (n+1 nodes) along axis a.
__host__ __device__ constexpr bool on_plus(int c, int a)
{
    return c == 0 ? a != 0 : c == 1 ? a != 1 : c == 2 ? a != 2
         : c == 3 ? a == 0 : c == 4 ? a == 1 : a == 2;
}

// Eqs. (7)-(12): dC/dt = (+1) D^{axis0} C0 + (-1) D^{axis1} C1.
__host__ __device__ constexpr int curl_comp(int c, int t)
{
    // Ex: Hz, Hy   Ey: Hx, Hz   Ez: Hy, Hx   Hx: Ey, Ez   Hy: Ez, Ex   Hz: Ex, Ey
    return t == 0 ? (c == 0 ? 5 : c == 1 ? 3 : c == 2 ? 4 : c == 3 ? 1 : c == 4 ? 2 : 0)
                  : (c == 0 ? 4 : c == 1 ? 5 : c == 2 ? 3 : c == 3 ? 2 : c == 4 ? 0 : 1);
}
__host__ __device__ constexpr int curl_axis(int c, int t)
{
    // Ex: y, z   Ey: z, x   Ez: x, y   Hx: z, y   Hy: x, z   Hz: y, x
    return t == 0 ? (c == 0 ? 1 : c == 1 ? 2 : c == 2 ? 0 : c == 3 ? 2 : c == 4 ? 0 : 1)
                  : (c == 0 ? 2 : c == 1 ? 0 : c == 2 ? 1 : c == 3 ? 1 : c == 4 ? 2 : 0);
}
__host__ __device__ constexpr int curl_sign(int t) { return t == 0 ? 1 : -1; }

template <typename T> struct Coef { T hi, lo; };

struct Link {               // interface partner of one face
    const void *F[6];       // partner block's padded fields
    const void *G[6];       // second partner (phase-shifted periodic face of a complex pair), or null
    double w[2];            // partner value = w[0] F + w[1] G (used when G is set)
    long long sy, sz;       // partner strides (elements)
    int n_norm;             // partner cell count along the face normal
    int side;               // partner face side: -1 low, +1 high
};

struct Src { int comp, i, j, k, wf; double amp, tw, t0, f; };
struct Prb { int comp, i, j, k; };

// Field storage type S and the arithmetic type of its values: FP16 storage
// is computed in FP32.
template <typename S> struct Compute { using type = S; };
template <> struct Compute<__half> { using type = float; };
template <typename S> using compute_t = typename Compute<S>::type;

// T: arithmetic type; S: storage type of the six fields (T, or __half with
// T = float).  Stored FP16 values are field / scale, one scale for E and one
// for H; the curl coefficients below carry the ratio of the two scales, so a
// kernel only converts on load and store.
// What every node needs comes first, the lists that few nodes look at after it.
template <typename T, typename S = T>
struct Params {
    S *F[6];                // padded fields Ex..Hz: element (i,j,k) at k*sz + j*sy + i
    const float *eps;       // ghost-padded cell eps_r on the same layout: cell (cx,cy,cz) at (cx+1,cy+1,cz+1)
    const float *mu;        // same for mu_r (only read when MUVAR)
    long long sy, sz;
    int n[3];
    int face[6];
    Coef<T> B[3];           // H: dt/(mu0 h_a) (uniform mu) or 2 dt/(mu0 h_a) (scaled by 1/sum2 mu_r)
    Coef<T> A[3];           // E: 4 dt/(eps0 h_a), scaled by 1/sum4 eps_r of the node
    Coef<T> AJ;             // 4 dt/eps0, source term
    T fscale[2];                       // physical value = stored value * fscale[E=0 / H=1]
    T uB, uA;                          // fscale[H]/fscale[E] and its inverse: B and A carry the
                                       // scale ratio; the absorbing-SAT gamma needs them without
    int nsrc, nprb;
    int pbox[2][6], sbox[6];           // index boxes (low, high per axis) around the probes of E, of H, and the sources
    T *probe_buf;
    long long probe_cap, probe_slot;   // sample slot of this step (skip if >= cap)
    long long step;                    // n: the E half-step injects J(t^{n+1/2})
    double dt, eta0, eps0, mu0;
    double h[3];
    double *partials;                  // energy partial sums, one per CTA of energy_sum
    int kchunk;
    int fdtd;                          // 1: plain Yee FDTD comparator (band kernels only)
    Src src[kMaxSources];
    Prb prb[kMaxProbes];
    Link link[6];
};

// ---------------------------------------------------------------------------
// small arithmetic helpers
// ---------------------------------------------------------------------------
template <typename T> struct Acc;
template <> struct Acc<float> {
    float hi = 0.f, lo = 0.f;
    __device__ __forceinline__ void add(const Coef<float> &c, float x, float scale = 1.f)
    {
        hi = fmaf(scale * c.hi, x, hi);
        lo = fmaf(scale * c.lo, x, lo);
    }
};
template <> struct Acc<double> {
    double hi = 0.0;
    __device__ __forceinline__ void add(const Coef<double> &c, double x, double scale = 1.0)
    {
        hi = fma(scale * c.hi, x, hi);
    }
};

// Reciprocal of s as hi + lo (hardware approximation + one Newton residual).
__device__ __forceinline__ void recip_pair(float s, float &rh, float &rl)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(s));
    float e = fmaf(-s, r, 1.0f);
    rh = r;
    rl = r * e;
}

// A positive normal float as T.  The FP64 form moves the bits with integer
// operations: the FP64 pipe, which converts too, takes 2 lanes per clock and SM.
template <typename T> __device__ __forceinline__ T widen(float f);
template <> __device__ __forceinline__ float widen<float>(float f) { return f; }
template <> __device__ __forceinline__ double widen<double>(float f)
{
    const unsigned b = __float_as_uint(f);
    return __hiloint2double((int)((b >> 3) + (896u << 20)), (int)(b << 29));
}

// Any float as a double (exactly), without the FP64 pipe: a subnormal is scaled
// into the normal range first, infinities and NaN get the FP64 exponent.
__device__ __forceinline__ double to_double(float f)
{
    const unsigned b = __float_as_uint(f);
    unsigned m = b & 0x7fffffffu, bias = 896u << 20;
    if (m < 0x00800000u) {
        m = __float_as_uint(__uint_as_float(m) * 16777216.f);
        bias = m ? (896u - 24u) << 20 : 0u;
    }
    unsigned hi = (m >> 3) + bias;
    if (m >= 0x7f800000u) hi |= 0x7ff00000u;
    return __hiloint2double((int)(hi | (b & 0x80000000u)), (int)(m << 29));
}
__device__ __forceinline__ double to_double(double f) { return f; }

// FP32 approximation of 1/s (relative error below 2^-21) from s's leading bits,
// widened; false outside [2^-100, 2^100), FP32's comfortable range.
__device__ __forceinline__ bool recip_seed(double s, double &r)
{
    const int hi = __double2hiint(s);
    const float f = __uint_as_float(__funnelshift_l((unsigned)__double2loint(s), (unsigned)(hi - (896 << 20)), 3));
    float q;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(q) : "f"(f));
    r = widen<double>(q);
    return (unsigned)(hi - (923 << 20)) < (unsigned)(200 << 20);
}

// a/s for a positive s: a times a reciprocal good to 2^-42, corrected by the
// remainder of that quotient (Markstein, IBM J. Res. Dev. 34, 1990), which leaves
// one rounding as a division does.  Five FP64 operations; a division takes about
// ten, at 2 lanes per clock and SM.  (A rounded reciprocal, multiplied inside the
// sum with the old value, takes two fewer: 96 x 75 x 88 at 1474 instead of 1599 us
// per 16 steps, and an error 10 % above the quotient's, since a node's reciprocal
// is off the same way at every step.)
__device__ __noinline__ double quot64_any(double a, double s) { return a / s; }
__device__ __forceinline__ double quot64(double a, double s)
{
    double r;
    if (!recip_seed(s, r)) return quot64_any(a, s);
    r = fma(r, fma(-s, r, 1.0), r);
    const double q = a * r;
    if ((__double2hiint(q) & 0x7ff00000) == 0x7ff00000) return q;    // infinite or NaN: no remainder
    return fma(fma(-s, q, a), r, q);
}

// increment = r * acc with r = 1/s (E nodes, or H nodes with varying mu)
__device__ __forceinline__ float scaled_increment(const Acc<float> &a, float s)
{
    float rh, rl;
    recip_pair(s, rh, rl);
    return fmaf(rh, a.hi, fmaf(rh, a.lo, rl * a.hi));
}
__device__ __forceinline__ double scaled_increment(const Acc<double> &a, double s)
{
    return quot64(a.hi, s);
}
__device__ __forceinline__ float plain_increment(const Acc<float> &a) { return a.hi + a.lo; }
__device__ __forceinline__ double plain_increment(const Acc<double> &a) { return a.hi; }

// FP32 arithmetic on FP16-stored fields: the coefficients' rounding residue
// (lo, about 6e-8 relative) is far below the storage rounding (4.9e-4), so
// the increment is accumulated from the rounded coefficients alone.
struct AccLite {
    float hi = 0.f;
    __device__ __forceinline__ void add(const Coef<float> &c, float x, float scale = 1.f)
    {
        hi = fmaf(scale * c.hi, x, hi);
    }
};
__device__ __forceinline__ float scaled_increment(const AccLite &a, float s)
{
    float rh, rl;
    recip_pair(s, rh, rl);
    return fmaf(rh, a.hi, rl * a.hi);
}
__device__ __forceinline__ float plain_increment(const AccLite &a) { return a.hi; }

// The accumulator of arithmetic type T for fields stored as S.
template <typename T, typename S> struct AccOf { using type = Acc<T>; };
template <> struct AccOf<float, __half> { using type = AccLite; };

// Rows of the Appendix operators at unit spacing.  Every row reads at most
// three consecutive entries of its line; they are gathered first (no branch
// before the loads, so all of a node's loads are in flight together) and the
// row formula is then applied to them.  The line holds entries 0..n+1 of the
// padded layout, so the gathered triple is always in bounds.
template <typename T> struct Tri { T a, b, c; };

// Field loads and stores in the storage type, values in the arithmetic type.
template <typename S>
__device__ __forceinline__ compute_t<S> ld_s(const S *p)
{
    if constexpr (std::is_same<S, __half>::value) return __half2float(*p);
    else return *p;
}
template <typename S>
__device__ __forceinline__ compute_t<S> ldg_s(const S *p)
{
    if constexpr (std::is_same<S, __half>::value) return __half2float(__ldg(p));
    else return __ldg(p);
}
// CG = true reads through L2 only (ld.global.cg), for values this kernel
// itself wrote earlier (coherent across the threads of a CTA after a
// barrier, never served stale from L1 or the read-only path).
template <bool CG, typename S>
__device__ __forceinline__ compute_t<S> ldf(const S *p)
{
    if constexpr (CG) {
        if constexpr (std::is_same<S, __half>::value) return __half2float(__ldcg(p));
        else return __ldcg(p);
    } else {
        return ld_s(p);
    }
}
// The value a store of v keeps (round to nearest for FP16 storage).
template <typename S, typename T>
__device__ __forceinline__ T quant(T v)
{
    if constexpr (std::is_same<S, __half>::value) return __half2float(__float2half_rn(v));
    else return v;
}
template <typename S, typename T>
__device__ __forceinline__ void st_s(S *p, T v)
{
    if constexpr (std::is_same<S, __half>::value) *p = __float2half_rn(v);
    else *p = v;
}

// entries s0, s0+1, s0+2 of the line starting at `line` with stride s
template <bool CG, typename S>
__device__ __forceinline__ Tri<compute_t<S>> tri_load(const S *line, long long s, int s0)
{
    const S *q = line + (long long)s0 * s;
    return {ldf<CG>(q), ldf<CG>(q + s), ldf<CG>(q + 2 * s)};
}

// FMA in the arithmetic type.
__device__ __forceinline__ float fma_t(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double fma_t(double a, double b, double c) { return fma(a, b, c); }

// A row of either operator reads at most three consecutive entries u_a, u_b,
// u_c of its line, with coefficients k0, k1, k2 (unit spacing).  Every kernel
// evaluates a row as the same chain, entries in increasing index order:
//   d = k0 u_a;  d = fma(k1, u_b, d);  d = fma(k2, u_c, d).
// A zero coefficient leaves d unchanged, and an interior row (-1, 1, 0)
// gives u_b - u_a exactly as a subtraction does, so the interior fast paths
// (plain differences), the one-pass kernel's x-end windows (four entries,
// zeros outside the row) and the general path all produce the same bits.
template <typename T>
__device__ __forceinline__ T row_chain(const T k[3], T a, T b, T c)
{
    T d = k[0] * a;
    d = fma_t(k[1], b, d);
    return fma_t(k[2], c, d);
}

// D- : x+ (n+1 values) -> x- (n+2 rows).  First entry read by row r.
__device__ __forceinline__ int dminus_start(int r, int n)
{
    return (r == 0 || r == 2) ? 0 : (r == n - 1 || r == n + 1) ? n - 2 : r - 1;
}
// Coefficients of row r of D- on the entries at dminus_start(r, n) (Appendix).
template <typename T>
__device__ __forceinline__ void dminus_coefs(int r, int n, T k[3])
{
    if (r == 2) { k[0] = T(-0.2); k[1] = T(-0.6); k[2] = T(0.8); }              // (4u2 - 3u1 - u0) / 5
    else if (r == n - 1) { k[0] = T(-0.8); k[1] = T(0.6); k[2] = T(0.2); }      // (u_n + 3u_{n-1} - 4u_{n-2}) / 5
    else if (r == n + 1) { k[0] = T(0); k[1] = T(-1); k[2] = T(1); }            // u_n - u_{n-1}
    else { k[0] = T(-1); k[1] = T(1); k[2] = T(0); }                            // rows 0 (u1 - u0), 1, 3..n-2, n
}
// Row r of D- from the entries gathered at dminus_start(r, n).
template <typename T>
__device__ __forceinline__ T dminus_eval(const Tri<T> &u, int r, int n)
{
    T k[3];
    dminus_coefs(r, n, k);
    return row_chain(k, u.a, u.b, u.c);
}

// D+ : x- (n+2 values) -> x+ (n+1 rows).  First entry read by row r.
__device__ __forceinline__ int dplus_start(int r, int n) { return r <= 1 ? 0 : r >= n - 1 ? n - 1 : r; }
// Coefficients of row r of D+ on the entries at dplus_start(r, n) (Appendix).
template <typename T>
__device__ __forceinline__ void dplus_coefs(int r, int n, T k[3])
{
    if (r == 0) { k[0] = T(-1); k[1] = T(0.5); k[2] = T(0.5); }                 // (v1 + v2)/2 - v0
    else if (r == 1) { k[0] = T(-0.5); k[1] = T(-0.25); k[2] = T(0.75); }       // 3v2/4 - v0/2 - v1/4
    else if (r == n - 1) { k[0] = T(-0.75); k[1] = T(0.25); k[2] = T(0.5); }    // v_n/4 + v_{n+1}/2 - 3v_{n-1}/4
    else if (r == n) { k[0] = T(-0.5); k[1] = T(-0.5); k[2] = T(1); }           // v_{n+1} - (v_{n-1} + v_n)/2
    else { k[0] = T(-1); k[1] = T(1); k[2] = T(0); }                            // rows 2..n-2: v_{r+1} - v_r
}
// Row r of D+ from the entries gathered at dplus_start(r, n).
template <typename T>
__device__ __forceinline__ T dplus_eval(const Tri<T> &v, int r, int n)
{
    T k[3];
    dplus_coefs(r, n, k);
    return row_chain(k, v.a, v.b, v.c);
}

// SAT helpers shared by every kernel that evaluates a face node, so that all
// of them round alike.
// Penalty value of an interface face: the partner's field at its face node,
// or e^{-+j alpha} times the complex partner (real and imaginary simulations).
template <bool CG, typename T, typename S>
__device__ __forceinline__ T link_value(const Link &L, int u, long long on)
{
    T nv = ldf<CG>(static_cast<const S *>(L.F[u]) + on);
    if (L.G[u]) nv = fma_t(T(L.w[1]), T(ldf<CG>(static_cast<const S *>(L.G[u]) + on)), T(L.w[0]) * nv);
    return nv;
}
// Characteristic impedance eta0 sqrt(mu_r / eps_r) at the node.
template <typename T>
__device__ __forceinline__ T node_eta(double eta0, T mr, T er) { return T(eta0) * sqrt(mr / er); }
// Absorbing penalty, H side: gamma = dt eta / (2 mu h) = (1/2) ba eta, ba = dt / (mu h) in stored units.
template <typename T>
__device__ __forceinline__ T abs_gamma_h(T ba, T eta) { return T(0.5) * ba * eta; }
// Absorbing penalty, E side: gamma = dt / (2 eta eps h) = (a / se) / (2 eta), a = 4 dt / (eps0 h) in
// stored units and se = 4 eps_r of the node.
template <typename T>
__device__ __forceinline__ T abs_gamma_e(T a, T se, T eta) { return a / se / (T(2) * eta); }
// New value with the absorbing self term averaged over the two time levels
// (pointwise semi-implicit): ((1 - gamma) old + inc) / (1 + gamma).
template <typename T>
__device__ __forceinline__ T sat_finish(T old, T inc, T gam)
{
    if (gam != T(0)) {
        if constexpr (std::is_same<T, double>::value) return quot64(fma_t(T(1) - gam, old, inc), T(1) + gam);
        return fma_t(T(1) - gam, old, inc) / (T(1) + gam);
    }
    return old + inc;
}

// 1D norm weight (unit spacing) of node r: P+ = diag(1/2,1,...,1,1/2),
// P- = diag(1/2,1/4,5/4,1,...,1,5/4,1/4,1/2)  (Appendix).
// A product of three is exact in FP32.
__device__ __forceinline__ float norm_weight(bool plus, int r, int n)
{
    if (plus) return (r == 0 || r == n) ? 0.5f : 1.0f;
    if (r == 0 || r == n + 1) return 0.5f;
    if (r == 1 || r == n) return 0.25f;
    if (r == 2 || r == n - 1) return 1.25f;
    return 1.0f;
}

__device__ __forceinline__ int extent(const int n[3], int c, int a) { return n[a] + (on_plus(c, a) ? 1 : 2); }

// (m[o] + m[o+a]) + (m[o+b] + m[o+a+b])
template <typename S>
__device__ __forceinline__ S pair_sum(const float *__restrict__ m, long long o, long long a, long long b)
{
    return (widen<S>(__ldg(m + o)) + widen<S>(__ldg(m + o + a))) +
           (widen<S>(__ldg(m + o + b)) + widen<S>(__ldg(m + o + a + b)));
}

// Sum of the ghost-padded cell values around a node of component c: the
// closed-box cell set of the node, always 2x2 (E) or 2x1 (H) entries after
// ghost padding (duplicates stand for clipped cells, so the mean is the mean
// over the distinct cells).
template <int C, typename S = float>
__device__ __forceinline__ S cell_sum(const float *__restrict__ m, long long o, long long sy, long long sz)
{
    // ghost-padded index of the node's first cell is the node index itself;
    // a plus-grid axis spans two cells (offset 0 and +1), a minus-grid axis one.
    // Summed pairwise, (a + b) + (c + d): exact whenever the cells agree, and
    // the same order in the fast and the general path.
    constexpr bool px = on_plus(C, 0), py = on_plus(C, 1), pz = on_plus(C, 2);
    if (px && py) return pair_sum<S>(m, o, 1, sy);
    if (px && pz) return pair_sum<S>(m, o, 1, sz);
    if (py && pz) return pair_sum<S>(m, o, sy, sz);
    const long long d = px ? 1 : py ? sy : sz;
    return widen<S>(__ldg(m + o)) + widen<S>(__ldg(m + o + d));
}
// Pair sums of the cells (j, j+1; i, i+1) of one plane of the cell array at m:
// the node sums of cell_sum are sums of two of them.
__device__ __forceinline__ void eps_pair_sums(const float *__restrict__ m, long long sy, double &a, double &b, double &c)
{
    const double f = widen<double>(__ldg(m)), fx = widen<double>(__ldg(m + 1));
    const double g = widen<double>(__ldg(m + sy)), gx = widen<double>(__ldg(m + sy + 1));
    a = f + g;
    b = f + fx;
    c = g + gx;
}

// Source waveforms (Sec. VI-B, VI-C): t and t0, tw in seconds.  A call, not
// inlined: a few lanes of a launch reach it, and its code would sit between the
// instructions that every warp fetches.
__device__ __noinline__ double waveform(int wf, double t, double tw, double t0, double f)
{
    const double x = (t - t0) / tw;
    const double g = exp(-4.0 * 3.14159265358979323846 * x * x);
    if (wf == 0) return g;
    if (wf == 1) return -5.0132565492620005 * x * 1.6487212707001282 * g;   // -sqrt(8 pi) x e^{1/2} g
    double ph = f * t;
    ph -= floor(ph);
    return sin(6.283185307179586 * ph) * g;
}

// J(t^{n+1/2}) of the sources that reach the index box of a warp, in the
// warp's slots of shared memory (entry q for source q), or null when none
// does.  One lane evaluates each source, once for the warp: the FP64 waveform
// costs about as much as a whole node.  Every lane of the warp calls it.
template <typename T, typename S>
__device__ __forceinline__ const double *source_values(const Params<T, S> &p, long long step, int lane, int k0, int k1,
                                                       int j0, int j1, int i0, int i1)
{
    static_assert(kMaxSources <= 32, "one lane per source");
    __shared__ double sJ[8][kMaxSources];
    if (!p.nsrc) return nullptr;
    bool hit = false;
    if (lane < p.nsrc) {
        const Src &Sr = p.src[lane];
        hit = (Sr.i < 0 || (Sr.i >= i0 && Sr.i <= i1)) && (Sr.j < 0 || (Sr.j >= j0 && Sr.j <= j1)) &&
              (Sr.k < 0 || (Sr.k >= k0 && Sr.k <= k1));
    }
    if (!__any_sync(0xffffffffu, hit)) return nullptr;
    double *const J = sJ[(threadIdx.x >> 5) & 7];
    __syncwarp();                                     // reads of an earlier use are done
    if (hit) {
        const Src &Sr = p.src[lane];
        J[lane] = Sr.amp * waveform(Sr.wf, ((double)step + 0.5) * p.dt, Sr.tw, Sr.t0, Sr.f);
    }
    __syncwarp();
    return J;
}

// Block-wide deterministic sum of one double per thread (fixed tree).
__device__ __forceinline__ void block_sum_to(double v, double *dst)
{
    __shared__ double red[kBlockX * kBlockY / 32];
    const int lane = threadIdx.x, warp = threadIdx.y;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (lane == 0) red[warp] = v;
    __syncthreads();
    if (warp == 0) {
        v = lane < (int)blockDim.y ? red[lane] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if (lane == 0) *dst = v;
    }
}

// ---------------------------------------------------------------------------
// H half-step: general path for one component at one node
// ---------------------------------------------------------------------------
// Entries of E read by the two curl terms of H component C at node idx.
// G: bit a set when the node may lie on a closure row or face along axis a;
// along the other axes the node is interior and the row is u_r - u_{r-1}.
// CG: read through L2 only (fields another CTA of the same launch wrote).
template <typename T, int C, int G = 7, bool CG = false, typename S = T>
__device__ __forceinline__ void h_gather(const Params<T, S> &p, const int idx[3], long long o, Tri<T> v[2])
{
#pragma unroll
    for (int t = 0; t < 2; ++t) {
        const int u = curl_comp(C, t), a = curl_axis(C, t);
        const long long st = a == 0 ? 1 : a == 1 ? p.sy : p.sz;
        if ((G >> a) & 1) {
            v[t] = tri_load<CG>(p.F[u] + (o - idx[a] * st), st, dminus_start(idx[a], p.n[a]));
        } else {
            v[t].a = ldf<CG>(p.F[u] + o - st);
            v[t].b = ldf<CG>(p.F[u] + o);
            v[t].c = v[t].b;
        }
    }
}

// H^{n+1/2} of component C at node idx from H^{n-1/2} (hold) and the gathered E.
template <typename T, int C, bool MUVAR, int G = 7, typename S = T>
__device__ __forceinline__ T h_apply(const Params<T, S> &p, const int idx[3], long long o, T hold, const Tri<T> v[2])
{
    typename AccOf<T, S>::type acc;
    T gam = T(0);
#pragma unroll
    for (int t = 0; t < 2; ++t) {
        const int u = curl_comp(C, t), a = curl_axis(C, t), sg = curl_sign(t);
        const bool gen = (G >> a) & 1;
        const T d = gen ? dminus_eval(v[t], idx[a], p.n[a]) : v[t].b - v[t].a;
        acc.add(p.B[a], d, T(sg));
        // H on the minus grid along a: face nodes at 0 and n+1 carry the SAT
        if (gen && (idx[a] == 0 || idx[a] == p.n[a] + 1)) {
            const int side = idx[a] == 0 ? -1 : 1;
            const int f = 2 * a + (side > 0);
            const int type = p.face[f];
            if (type != kPMC) {
                const T phi = T(-sg * side);
                const T pv = side < 0 ? v[t].a : v[t].c;      // E on the face: entry 0 or n
                if (type == kPEC) {
                    acc.add(p.B[a], pv, T(2) * phi);
                } else if (type == kABS) {
                    acc.add(p.B[a], pv, phi);
                    const T er = cell_sum<C, T>(p.eps, o, p.sy, p.sz) * T(0.5);
                    const T mr = MUVAR ? cell_sum<C, T>(p.mu, o, p.sy, p.sz) * T(0.5) : T(1);
                    // B holds dt/(mu0 h_a) (x2 when mu varies)
                    const T ba = (MUVAR ? T(p.B[a].hi) * T(0.5) / mr : T(p.B[a].hi)) * p.uB;
                    gam += abs_gamma_h(ba, node_eta(p.eta0, mr, er));
                } else {   // interface: (phi/2)(E^A - E^B) / (mu w), w = h/2
                    const Link &L = p.link[f];
                    const int nidx = L.side < 0 ? 0 : L.n_norm;      // partner E on its plus grid along a
                    long long on = 0;
                    const long long ost[3] = {1, L.sy, L.sz};
                    for (int b = 0; b < 3; ++b) on += (long long)(b == a ? nidx : idx[b]) * ost[b];
                    acc.add(p.B[a], pv - link_value<false, T, S>(L, u, on), phi);
                }
            }
        }
    }
    T inc;
    if (MUVAR) {
        inc = scaled_increment(acc, cell_sum<C, T>(p.mu, o, p.sy, p.sz));
    } else {
        inc = plain_increment(acc);
    }
    return sat_finish(hold, inc, gam);
}

// H half-step, general path, one component at one node (Eqs. (10)-(15)).
template <typename T, int C, bool MUVAR, typename S = T>
__device__ __forceinline__ T h_node(const Params<T, S> &p, const int idx[3], long long o, T hold)
{
    Tri<T> v[2];
    h_gather<T, C, 7>(p, idx, o, v);
    return h_apply<T, C, MUVAR, 7>(p, idx, o, hold, v);
}

// Entries of H read by the two curl terms of E component C at node idx.
// G as for h_gather; interior rows of D+ are v_{r+1} - v_r.
template <typename T, int C, bool CG = false, int G = 7, typename S = T>
__device__ __forceinline__ void e_gather(const Params<T, S> &p, const int idx[3], long long o, Tri<T> v[2])
{
#pragma unroll
    for (int t = 0; t < 2; ++t) {
        const int u = curl_comp(C, t), a = curl_axis(C, t);
        const long long st = a == 0 ? 1 : a == 1 ? p.sy : p.sz;
        if ((G >> a) & 1) {
            v[t] = tri_load<CG>(p.F[u] + (o - idx[a] * st), st, dplus_start(idx[a], p.n[a]));
        } else {
            v[t].a = ldf<CG>(p.F[u] + o);
            v[t].b = ldf<CG>(p.F[u] + o + st);
            v[t].c = v[t].b;
        }
    }
}

// E^{n+1} of component C at node idx from E^n (eold), se = sum4 eps_r of the
// node and the gathered H.
template <typename T, int C, bool MUVAR, bool CG = false, int G = 7, typename S = T>
__device__ __forceinline__ T e_apply(const Params<T, S> &p, const int idx[3], long long o, T eold, T se, const Tri<T> v[2],
                                     unsigned smask, const double *J)
{
    typename AccOf<T, S>::type acc;
    T gam = T(0);
#pragma unroll
    for (int t = 0; t < 2; ++t) {
        const int u = curl_comp(C, t), a = curl_axis(C, t), sg = curl_sign(t);
        const bool gen = (G >> a) & 1;
        const T d = gen ? dplus_eval(v[t], idx[a], p.n[a]) : v[t].b - v[t].a;
        acc.add(p.A[a], d, T(sg));
        // E on the plus grid along a: face nodes at 0 and n carry the SAT
        if (gen && (idx[a] == 0 || idx[a] == p.n[a])) {
            const int side = idx[a] == 0 ? -1 : 1;
            const int f = 2 * a + (side > 0);
            const int type = p.face[f];
            if (type != kPEC) {
                const T phi = T(-sg * side);
                const T pv = side < 0 ? v[t].a : v[t].c;      // H on the face: entry 0 or n+1
                if (type == kPMC) {
                    acc.add(p.A[a], pv, T(2) * phi);
                } else if (type == kABS) {
                    acc.add(p.A[a], pv, phi);
                    const T er = se * T(0.25);
                    const T mr = MUVAR ? cell_sum<C, T>(p.mu, o, p.sy, p.sz) * T(0.25) : T(1);
                    gam += abs_gamma_e(T(p.A[a].hi) * p.uA, se, node_eta(p.eta0, mr, er));
                } else {
                    const Link &L = p.link[f];
                    const int nidx = L.side < 0 ? 0 : L.n_norm + 1;  // partner H on its minus grid along a
                    long long on = 0;
                    const long long ost[3] = {1, L.sy, L.sz};
                    for (int b = 0; b < 3; ++b) on += (long long)(b == a ? nidx : idx[b]) * ost[b];
                    acc.add(p.A[a], pv - link_value<CG, T, S>(L, u, on), phi);
                }
            }
        }
    }
    // current-density sources: eps dE/dt = ... - J
    unsigned m = smask;
    while (m) {
        const int q = __ffs(m) - 1;
        m &= m - 1;
        const Src &Sr = p.src[q];
        if (Sr.comp == C && (Sr.k < 0 || Sr.k == idx[2])) acc.add(p.AJ, T(J[q]), T(-1));
    }
    const T inc = scaled_increment(acc, se);
    return sat_finish(eold, inc, gam);
}

// ---------------------------------------------------------------------------
// Kernels
// ---------------------------------------------------------------------------

// Terms of the energy sums: weight times the squared E, or times H^{n-1/2}
// H^{n+1/2} and mu_r (sum of the two cells).
template <typename T>
__device__ __forceinline__ double energy_e(double weight, T e, double sum)
{
    return fma(weight, to_double(e) * to_double(e), sum);
}
template <typename T, typename S, int C, bool MUVAR>
__device__ __forceinline__ double energy_h(const Params<T, S> &p, long long o, float w, T ho, T hn, double sum)
{
    double a = to_double(ho);
    if (MUVAR) a *= cell_sum<C, double>(p.mu, o, p.sy, p.sz);
    if (w != 1.f) a *= widen<double>(w);
    return fma(a, to_double(hn), sum);
}

// Leapfrog energy of Eq. (16) (FP64) over every node, one partial sum per CTA
// in p.partials: H^{n+1/2} is formed on the fly, no field is changed.
//
// Bound by the FP64 pipe (2 lanes per clock and SM).  Per thread the sums of
// eps E^2 and mu H H are kept apart, so the constants leave the loop; a node's
// eps sums come from pair sums carried from plane to plane (six additions for
// three components); the norm weights multiply as FP32, where their products
// are exact, and FP32 values and cells widen by integer operations.  That is 15
// FP64 operations for an interior node and about 24 at the boundary, where 78
// were: 165 us for 160 x 144 x 128 cells with the final sum, 475 before.
template <typename T, typename S, bool MUVAR>
__global__ void __launch_bounds__(kBlockX *kBlockY) energy_sum(const Params<T, S> p)
{
    const int j = blockIdx.y * kBlockY + threadIdx.y;
    const int nx = p.n[0], ny = p.n[1], nz = p.n[2];
    // x nodes in the order 3 .. nx-2, then the six ends: all but the last warps of a
    // row then hold two-point rows only (at 160 cells 4 of 6 warps, 3 in the plain order)
    const int at = blockIdx.x * kBlockX + threadIdx.x, inner = nx - 4, end = at - inner;
    const int i = at < inner ? at + 3 : end < 3 ? end : nx - 4 + end;
    const int k0 = blockIdx.z * p.kchunk;
    const int k1 = min(k0 + p.kchunk, nz + 2);
    double se = 0.0, sh = 0.0;
    if (at < nx + 2 && j < ny + 2) {
        const S *__restrict__ Hx = p.F[3];
        const S *__restrict__ Hy = p.F[4];
        const S *__restrict__ Hz = p.F[5];
        const S *__restrict__ Ex = p.F[0];
        const S *__restrict__ Ey = p.F[1];
        const S *__restrict__ Ez = p.F[2];
        const long long sy = p.sy, sz = p.sz;
        long long o = (long long)k0 * sz + (long long)j * sy + i;
        // the warp's row lies inside the box of two-point rows along x and y
        const bool inside = (int)blockIdx.x * kBlockX + kBlockX <= inner && j >= 3 && j <= ny - 2;
        const Coef<T> Bx = p.B[0], By = p.B[1], Bz = p.B[2];
        double qa, qb, qc;
        eps_pair_sums(p.eps + o, sy, qa, qb, qc);
        for (int k = k0; k < k1; ++k, o += sz) {
            const T ex = ldg_s(Ex + o), ey = ldg_s(Ey + o), ez = ldg_s(Ez + o);
            const T hx = ldg_s(Hx + o), hy = ldg_s(Hy + o), hz = ldg_s(Hz + o);
            double na, nb, nc;
            // (the last plane again at the end: no E node there spans two cells along z)
            eps_pair_sums(p.eps + o + (k <= nz ? sz : 0), sy, na, nb, nc);
            if (inside && k >= 3 && k <= nz - 2) {
                const T exj = ldg_s(Ex + o - sy), exk = ldg_s(Ex + o - sz), eyi = ldg_s(Ey + o - 1);
                const T eyk = ldg_s(Ey + o - sz), ezi = ldg_s(Ez + o - 1), ezj = ldg_s(Ez + o - sy);
                typename AccOf<T, S>::type a, b, c;
                a.add(Bz, ey - eyk); a.add(By, ez - ezj, T(-1));
                b.add(Bx, ez - ezi); b.add(Bz, ex - exk, T(-1));
                c.add(By, ex - exj); c.add(Bx, ey - eyi, T(-1));
                if constexpr (MUVAR) {
                    sh = energy_h<T, S, 3, MUVAR>(p, o, 1.f, hx, quant<S>(hx + scaled_increment(a, cell_sum<3, T>(p.mu, o, sy, sz))), sh);
                    sh = energy_h<T, S, 4, MUVAR>(p, o, 1.f, hy, quant<S>(hy + scaled_increment(b, cell_sum<4, T>(p.mu, o, sy, sz))), sh);
                    sh = energy_h<T, S, 5, MUVAR>(p, o, 1.f, hz, quant<S>(hz + scaled_increment(c, cell_sum<5, T>(p.mu, o, sy, sz))), sh);
                } else {
                    sh = energy_h<T, S, 3, MUVAR>(p, o, 1.f, hx, quant<S>(hx + plain_increment(a)), sh);
                    sh = energy_h<T, S, 4, MUVAR>(p, o, 1.f, hy, quant<S>(hy + plain_increment(b)), sh);
                    sh = energy_h<T, S, 5, MUVAR>(p, o, 1.f, hz, quant<S>(hz + plain_increment(c)), sh);
                }
                se = energy_e(qa + na, ex, se);
                se = energy_e(qb + nb, ey, se);
                se = energy_e(qb + qc, ez, se);
            } else {
                // nodes of each component (Table I) with their norm weights
                const int idx[3] = {i, j, k};
                if (i <= nx && j <= ny + 1 && k <= nz + 1)
                    sh = energy_h<T, S, 3, MUVAR>(p, o, norm_weight(true, i, nx) * norm_weight(false, j, ny) * norm_weight(false, k, nz), hx,
                                                   quant<S>(h_node<T, 3, MUVAR>(p, idx, o, hx)), sh);
                if (i <= nx + 1 && j <= ny && k <= nz + 1)
                    sh = energy_h<T, S, 4, MUVAR>(p, o, norm_weight(false, i, nx) * norm_weight(true, j, ny) * norm_weight(false, k, nz), hy,
                                                   quant<S>(h_node<T, 4, MUVAR>(p, idx, o, hy)), sh);
                if (i <= nx + 1 && j <= ny + 1 && k <= nz)
                    sh = energy_h<T, S, 5, MUVAR>(p, o, norm_weight(false, i, nx) * norm_weight(false, j, ny) * norm_weight(true, k, nz), hz,
                                                   quant<S>(h_node<T, 5, MUVAR>(p, idx, o, hz)), sh);
                if (i <= nx + 1 && j <= ny && k <= nz)
                    se = energy_e(widen<double>(norm_weight(false, i, nx) * norm_weight(true, j, ny) * norm_weight(true, k, nz)) * (qa + na), ex, se);
                if (i <= nx && j <= ny + 1 && k <= nz)
                    se = energy_e(widen<double>(norm_weight(true, i, nx) * norm_weight(false, j, ny) * norm_weight(true, k, nz)) * (qb + nb), ey, se);
                if (i <= nx && j <= ny && k <= nz + 1)
                    se = energy_e(widen<double>(norm_weight(true, i, nx) * norm_weight(true, j, ny) * norm_weight(false, k, nz)) * (qb + qc), ez, se);
            }
            qa = na;
            qb = nb;
            qc = nc;
        }
    }
    // eps_r is a quarter of the four cells' sum, mu_r half of the two cells'
    const double cE = p.eps0 * 0.25 * (double)p.fscale[0] * (double)p.fscale[0];
    const double cH = p.mu0 * (MUVAR ? 0.5 : 1.0) * (double)p.fscale[1] * (double)p.fscale[1];
    const double hvol = p.h[0] * p.h[1] * p.h[2];
    block_sum_to((cE * se + cH * sh) * hvol,
                 p.partials + ((long long)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x);
}

// Fixed-order sum of the per-CTA energy partials (one CTA, deterministic).
__global__ void __launch_bounds__(256) energy_finalize(const double *__restrict__ partials, long long n,
                                                        double *__restrict__ out)
{
    __shared__ double red[256];
    double v = 0.0;
    for (long long q = threadIdx.x; q < n; q += 256) v += partials[q];
    red[threadIdx.x] = v;
    __syncthreads();
    for (int s = 128; s > 0; s >>= 1) {
        if ((int)threadIdx.x < s) red[threadIdx.x] += red[threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x == 0) *out = 0.5 * red[0];
}

// One component between its dense array (natural extents e0 x e1 x e2, x
// fastest) and the padded layout (row pitch sy, plane pitch sz), converting
// between the stored type and the caller's: out = in * scale (FP16 storage;
// scale is 1 and left out otherwise).  TO_PADDED: dense in, padded out.
//
// Bound by memory.  One warp takes a row: the row's place is decoded once
// (one division per row, not per element), and the lanes walk it in 128-byte
// segments, four loads in flight each.  Dense rows start at any element, so
// the accesses stay one element wide; 32 lanes still cover whole sectors.
// 5.2 TB/s out of a 512^3 FP32 grid (205 us per component; the pitched copy
// call took 617 us, 1.74 TB/s; the FP16 form with a division per element 815).
template <bool TO_PADDED, typename In, typename Out>
__global__ void __launch_bounds__(256) move_field(const In *__restrict__ src, Out *__restrict__ dst, int e0, int e1,
                                                  long long rows, long long sy, long long sz, float scale)
{
    const int lane = threadIdx.x & 31;
    for (long long r = blockIdx.x * 8ll + (threadIdx.x >> 5); r < rows; r += gridDim.x * 8ll) {
        const long long k = r / e1, j = r - k * e1;
        const long long dense = r * e0, padded = k * sz + j * sy;
        const In *s = src + (TO_PADDED ? dense : padded);
        Out *d = dst + (TO_PADDED ? padded : dense);
        for (int i0 = lane; i0 < e0; i0 += 128) {
            In v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (i0 + 32 * u < e0) v[u] = s[i0 + 32 * u];
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (i0 + 32 * u < e0) {
                    if constexpr (std::is_same<In, Out>::value) d[i0 + 32 * u] = v[u];
                    else if constexpr (TO_PADDED) d[i0 + 32 * u] = __float2half_rn(v[u] * scale);
                    else d[i0 + 32 * u] = __half2float(v[u]) * scale;
                }
        }
    }
}

// Ghost-padded cell array (coefficient build, once per grid): padded (cx+1,
// cy+1, cz+1) holds cell (cx, cy, cz); ghost layers repeat the nearest cell.
__global__ void pad_cells(const float *__restrict__ cells, int nx, int ny, int nz, float fill,
                          float *__restrict__ out, long long sy, long long sz)
{
    const long long total = (long long)(nx + 2) * (ny + 2) * (nz + 2);
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < total;
         q += (long long)gridDim.x * blockDim.x) {
        const int i = (int)(q % (nx + 2));
        const int j = (int)((q / (nx + 2)) % (ny + 2));
        const int k = (int)(q / ((long long)(nx + 2) * (ny + 2)));
        float v = fill;
        if (cells) {
            const int cx = min(max(i - 1, 0), nx - 1);
            const int cy = min(max(j - 1, 0), ny - 1);
            const int cz = min(max(k - 1, 0), nz - 1);
            v = cells[((long long)cz * ny + cy) * nx + cx];
        }
        out[(long long)k * sz + (long long)j * sy + i] = v;
    }
}

}  // namespace sbp
