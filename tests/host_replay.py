"""The device code of the step kernels compiled for the host and run thread by thread.

``build`` takes the kernels' source as it stands (kernels.cuh, fused.cuh, halfstep.cuh and the work
lists of sbpsat.cu), replaces inline PTX, and compiles it with g++ (unoptimised: every load stays) behind the small CUDA shim below:
the threads of a CTA are contexts that switch at warp and CTA synchronisation.  ``programs`` then
run single launches on arrays of exactly the library's sizes with an unmapped page behind each, so a
read or write past an array ends the process."""
import os
import re
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2206_00638_gb300", "csrc")

SHIM = r"""
#include <sys/mman.h>
#include <ucontext.h>
#include <unistd.h>
#include <algorithm>
#include <climits>
#include <cmath>
#include <cstddef>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <type_traits>
#include <vector>
#define __device__
#define __host__
#define __global__ static
#define __shared__ static
#define __forceinline__ inline
#define __noinline__ __attribute__((noinline))
#define __launch_bounds__(...)
#define __maxnreg__(...)
#define __grid_constant__
#define __align__(n) __attribute__((aligned(n)))
struct Dim { unsigned x, y, z; };
static Dim threadIdx, blockIdx, blockDim, gridDim;
struct uint2 { unsigned x, y; };
struct uint4 { unsigned x, y, z, w; };
struct float2 { float x, y; };
struct float4 { float x, y, z, w; };
struct __half { _Float16 v; };
struct CUtensorMap { char bytes[128]; };
inline float __half2float(__half h) { return (float)h.v; }
inline __half __float2half_rn(float f) { return {(_Float16)f}; }
template <typename T> T __ldg(const T *p) { return *p; }
template <typename T> T __ldcg(const T *p) { return *p; }
template <typename A, typename B> A bits(B b) { A a; static_assert(sizeof(A) == sizeof(B)); std::memcpy(&a, &b, sizeof(a)); return a; }
inline unsigned __float_as_uint(float f) { return bits<unsigned>(f); }
inline float __uint_as_float(unsigned u) { return bits<float>(u); }
inline int __double2hiint(double d) { return (int)(bits<uint64_t>(d) >> 32); }
inline int __double2loint(double d) { return (int)bits<uint64_t>(d); }
inline double __hiloint2double(int h, int l) { return bits<double>((uint64_t)(unsigned)h << 32 | (unsigned)l); }
inline unsigned __funnelshift_l(unsigned lo, unsigned hi, unsigned s) { return (unsigned)(((uint64_t)hi << 32 | lo) << (s & 31) >> 32); }
inline unsigned __umulhi(unsigned a, unsigned b) { return (unsigned)((uint64_t)a * b >> 32); }
inline int __ffs(int v) { return __builtin_ffs(v); }
inline int __ffsll(long long v) { return __builtin_ffsll(v); }
using std::max; using std::min;
// never run here: the one-pass and the persistent kernel
namespace sbp { __align__(128) unsigned char smem_raw[1]; }
inline void __nanosleep(unsigned) {}
inline void __threadfence() {}
inline int __syncthreads_or(int v) { return v; }
inline size_t __cvta_generic_to_shared(const void *) { return 0; }
template <typename T> T atomicAdd(T *p, T v) { T o = *p; *p += v; return o; }
template <typename T> T atomicExch(T *p, T v) { T o = *p; *p = v; return o; }

// --- threads of a CTA ---------------------------------------------------------
struct Group { int alive = 0, arrived = 0; unsigned gen = 0; long long in[256], out[256]; };
struct Fiber { ucontext_t ctx; bool done; Dim id; int lane; Group *warp; std::vector<char> stack; };
static std::vector<Fiber> g_fibers(256);
static Group g_warps[8], g_block;
static ucontext_t g_main;
static Fiber *g_me;
static std::function<void()> g_kernel;
static long long g_waits;               // threads that executed griddepcontrol.wait
inline void pdl_wait_hook() { g_waits++; }
static void release(Group &g) { std::memcpy(g.out, g.in, sizeof(g.in)); g.arrived = 0; g.gen++; }
// Deposit v, wait for every live member, return the values deposited.
static const long long *meet_group(Group &g, int slot, long long v)
{
    const unsigned gen = g.gen;
    g.in[slot] = v;
    if (++g.arrived == g.alive) release(g);
    while (g.gen == gen) { Fiber *me = g_me; swapcontext(&me->ctx, &g_main); }
    return g.out;
}
static void fiber_main()
{
    g_kernel();
    Fiber &f = *g_me;
    f.done = true;
    for (Group *g : {f.warp, &g_block}) {
        g->in[g == &g_block ? (int)(&f - &g_fibers[0]) : f.lane] = LLONG_MIN;    // gone
        g->alive--;
        if (g->alive && g->arrived == g->alive) release(*g);
    }
    swapcontext(&f.ctx, &g_main);
}
static void launch(Dim grid, Dim block, std::function<void()> kernel)
{
    g_kernel = kernel;
    gridDim = grid; blockDim = block;
    const int n = (int)(block.x * block.y);
    for (unsigned c = 0; c < grid.x * grid.y * grid.z; c++) {
        blockIdx = {c % grid.x, c / grid.x % grid.y, c / (grid.x * grid.y)};
        g_block = Group();
        for (Group &w : g_warps) w = Group();
        for (int t = 0; t < n; t++) {
            Fiber &f = g_fibers[t];
            f.done = false;
            f.id = {t % block.x, t / block.x, 0};
            f.lane = t & 31;
            f.warp = &g_warps[t >> 5];
            f.warp->alive++;
            g_block.alive++;
            if (f.stack.empty()) f.stack.resize(64 << 10);
            getcontext(&f.ctx);
            f.ctx.uc_stack.ss_sp = f.stack.data();
            f.ctx.uc_stack.ss_size = f.stack.size();
            f.ctx.uc_link = &g_main;
            makecontext(&f.ctx, fiber_main, 0);
        }
        for (int left = n; left;) {
            left = 0;
            for (int t = 0; t < n; t++) {
                Fiber &f = g_fibers[t];
                if (f.done) continue;
                g_me = &f;
                threadIdx = f.id;
                swapcontext(&g_main, &f.ctx);
                left += !f.done;
            }
        }
    }
}
inline void __syncthreads() { const Dim t = threadIdx; meet_group(g_block, (int)(g_me - &g_fibers[0]), 0); threadIdx = t; }
template <typename F> auto over_warp(long long v, F f)
{
    const Dim t = threadIdx;
    const long long *all = meet_group(*g_me->warp, g_me->lane, v);
    threadIdx = t;
    return f(all);
}
inline void __syncwarp() { over_warp(0, [](const long long *) { return 0; }); }
inline unsigned __ballot_sync(unsigned, int v)
{
    return over_warp(v != 0, [](const long long *a) { unsigned m = 0; for (int l = 0; l < 32; l++) m |= (unsigned)(a[l] == 1) << l; return m; });
}
inline int __any_sync(unsigned m, int v) { return __ballot_sync(m, v) != 0; }
inline int __reduce_min_sync(unsigned, int v)
{
    return over_warp(v, [](const long long *a) { long long r = INT_MAX; for (int l = 0; l < 32; l++) if (a[l] != LLONG_MIN) r = min(r, a[l]); return (int)r; });
}
inline int __reduce_max_sync(unsigned, int v)
{
    return over_warp(v, [](const long long *a) { long long r = INT_MIN; for (int l = 0; l < 32; l++) r = max(r, a[l]); return (int)max(r, (long long)INT_MIN); });
}
inline double __shfl_down_sync(unsigned, double v, int o)
{
    const int at = g_me->lane + o < 32 ? g_me->lane + o : g_me->lane;
    return over_warp(bits<long long>(v), [at](const long long *a) { return bits<double>(a[at]); });
}

// An array that ends where the mapped memory does.
template <typename T> T *guarded(size_t n)
{
    const size_t page = (size_t)sysconf(_SC_PAGESIZE), bytes = (n * sizeof(T) + page - 1) / page * page;
    char *m = (char *)mmap(nullptr, bytes + page, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS, -1, 0);
    if (m == MAP_FAILED || mprotect(m + bytes, page, PROT_NONE)) std::abort();
    T *a = (T *)(m + bytes - n * sizeof(T));
    for (size_t q = 0; q < n; q++) a[q] = T();
    return a;
}
"""

HELPERS = r"""
// A grid's band, arrays and parameters as the library lays them out.
sbp::Band make_band(const int n[3], bool electric)
{
    sbp::Band b;
    b.lo = electric ? 3 : 4;
    for (int a = 0; a < 3; a++) b.hi[a] = n[a] - 3;
    b.segs = b.hi[0] / 32 + 1;
    b.zplanes = b.lo + (n[2] + 1 - b.hi[2]);
    b.yrows = b.lo + (n[1] + 1 - b.hi[1]);
    b.jin = b.hi[1] - b.lo + 1;
    b.xgroups = (n[1] + 2 + 7) / 8;
    b.wz = b.zplanes * b.jin * b.segs;
    b.wy = (n[2] + 2) * b.yrows * b.segs;
    b.wx = (n[2] + 2) * b.xgroups * 2;
    b.ctas = (b.wz + b.wy + b.wx + 7) / 8;
    return b;
}

struct Host {
    int n[3];
    long long sy, sz;
    size_t elems;
    Host(const int m[3])
    {
        for (int a = 0; a < 3; a++) n[a] = m[a];
        sy = (n[0] + 2 + 7) / 8 * 8;
        sz = sy * (n[1] + 2);
        elems = (size_t)sz * (n[2] + 3);
    }
    template <typename T> sbp::Params<T> params(int face, bool mu)
    {
        sbp::Params<T> p;
        std::memset(&p, 0, sizeof(p));
        for (int c = 0; c < 6; c++) p.F[c] = guarded<T>(elems);
        float *cells[2] = {guarded<float>(elems), mu ? guarded<float>(elems) : nullptr};
        for (float *m : cells)
            for (size_t q = 0; m && q < elems; q++) m[q] = 1.f + (float)(q % 7);
        p.eps = cells[0];
        p.mu = cells[1];
        p.sy = sy; p.sz = sz;
        for (int a = 0; a < 3; a++) {
            p.n[a] = n[a];
            p.face[2 * a] = p.face[2 * a + 1] = face;
            p.B[a] = {T(0.25), T(0)};
            p.A[a] = {T(0.5), T(0)};
        }
        p.eta0 = p.uA = p.uB = 1;
        p.fscale[0] = p.fscale[1] = 1;
        for (int *box : {p.pbox[0], p.pbox[1], p.sbox})
            for (int a = 0; a < 3; a++) { box[a] = INT_MAX; box[3 + a] = -1; }
        return p;
    }
    sbp::Sweep sweep(bool electric, int v, int kz, bool onepass = false)
    {
        sbp::Sweep w;
        if (make_sweep(n, electric, v, kz, w, onepass)) std::abort();
        return w;
    }
};
"""


def _device(name):
    """A source file with its inline PTX replaced."""
    text = open(os.path.join(CSRC, name)).read()
    text = re.sub(r"^#(include|pragma once).*$", "", text, flags=re.M)
    text = text.replace("extern __shared__", "extern")
    text = re.sub(r'asm\s+volatile\("griddepcontrol\.wait;".*?\);', "pdl_wait_hook();", text, flags=re.S)
    text = re.sub(r'asm\("rcp\.approx\.ftz\.f32 %0, %1;" : "=f"\((\w+)\) : "f"\((\w+)\)\);', r"\1 = 1.0f / \2;", text)
    assert "rcp.approx" not in text
    text = re.sub(r"asm\s*(volatile)?\s*\((?:[^()\"]|\"(?:[^\"\\]|\\.)*\"|\((?:[^()\"]|\([^()]*\))*\))*\)\s*;", ";", text)
    assert not re.search(r"\basm\b", re.sub(r"//.*", "", text))
    return text


def _work_lists():
    """fast_div and make_sweep of sbpsat.cu."""
    text = open(os.path.join(CSRC, "sbpsat.cu")).read()
    start, end = text.index("// Multiplier and shift of FastDiv"), text.index("// Vector width (V) and planes per z-chunk")
    return text[start:end]


def build(tmp, main):
    """Compile the device code with ``main`` (C++ source of a program); its path."""
    src, exe = os.path.join(tmp, "replay.cpp"), os.path.join(tmp, "replay")
    with open(src, "w") as f:
        f.write(SHIM)
        f.write("enum { SBP_OK = 0, SBP_EINVAL = -1 };\n")
        for name in ("kernels.cuh", "fused.cuh", "halfstep.cuh"):
            f.write(_device(name))
        f.write(_work_lists() + HELPERS + main)
    subprocess.run(["g++", "-std=c++17", "-O0", "-w", "-o", exe, src], check=True)
    return exe
