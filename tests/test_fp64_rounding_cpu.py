"""FP64 half-steps round the increment at its own size and the new field value once.

H: the device code runs on the host (host_replay) on fields whose differences are exact and with curl
coefficients of 2^-12 times an odd mantissa, so an interior node's increment is 2^-10 of the field:
its two roundings are below 2^-9 of the new value's half ulp, and the sum adds half an ulp.  Adding
each curl term to the field by itself rounds twice at the field's size.

E: on random fields and materials, interior nodes equal old + (sum of the curl terms) / (sum of the
cells) with a plain division, bit for bit."""
import subprocess

from tests import host_replay

MAIN = r"""
int main()
{
    const int n[3] = {12, 11, 10};
    Host g(n);
    auto p = g.params<double>(0, false);
    for (int a = 0; a < 3; a++) p.B[a] = {std::ldexp(1.0 + (2 * a + 1) / 7.0, -12), 0.0};
    unsigned seed = 1;
    for (int c = 0; c < 6; c++)
        for (size_t q = 0; q < g.elems; q++) {
            seed = seed * 1664525u + 1013904223u;
            p.F[c][q] = c < 3 ? (double)(int)(seed >> 20) / 4096 : 1.0 + (seed >> 8) * 0x1p-24 + (seed >> 12) * 0x1p-50;
        }
    std::vector<double> old[3];
    for (int c = 0; c < 3; c++) old[c].assign(p.F[3 + c], p.F[3 + c] + g.elems);
    const sbp::Sweep w = g.sweep(false, 1, 2);
    launch({w.ctas, 1, 1}, {sbp::kSweepThreads, 1, 1}, [&] { sbp::half_h<unsigned, double, double, false, 1>(p, w); });
    // (53-bit coefficients times 13-bit differences: within 2^-64 of the increment in long double)
    double worst = 0;
    for (int k = 3; k <= n[2] - 2; k++)
        for (int j = 3; j <= n[1] - 2; j++)
            for (int i = 3; i <= n[0] - 2; i++) {
                const long long o = k * g.sz + j * g.sy + i, st[3] = {1, g.sy, g.sz};
                for (int c = 3; c < 6; c++) {
                    long double v = old[c - 3][o];
                    for (int t = 0; t < 2; t++) {
                        const double *u = p.F[sbp::curl_comp(c, t)];
                        const int a = sbp::curl_axis(c, t);
                        v += (long double)sbp::curl_sign(t) * p.B[a].hi * (u[o] - u[o - st[a]]);
                    }
                    const double got = p.F[c][o], ulp = std::ldexp(1.0, std::ilogb((double)v) - 52);
                    worst = std::max(worst, std::abs((double)(got - v)) / ulp);
                }
            }
    std::printf("%g\n", worst);
}
"""


MAIN_E = r"""
template <int C> void check(const sbp::Params<double> &p, const std::vector<double> &old, long long o, int &bad)
{
    const long long st[3] = {1, p.sy, p.sz};
    sbp::Acc<double> a;
    for (int t = 0; t < 2; t++) {
        const double *u = p.F[sbp::curl_comp(C, t)];
        const int x = sbp::curl_axis(C, t);
        a.add(p.A[x], u[o + st[x]] - u[o], sbp::curl_sign(t));
    }
    bad += p.F[C][o] != old[o] + a.hi / sbp::cell_sum<C, double>(p.eps, o, p.sy, p.sz);
}
int main()
{
    const int n[3] = {22, 19, 20};
    Host g(n);
    auto p = g.params<double>(0, false);
    std::srand(3);
    auto uniform = [] { return (std::rand() + std::rand() / (RAND_MAX + 1.0)) / RAND_MAX; };
    for (int a = 0; a < 3; a++) p.A[a] = {1.0 + uniform(), 0.0};
    std::vector<double> old[3];
    for (int c = 0; c < 6; c++)
        for (size_t q = 0; q < g.elems; q++) p.F[c][q] = uniform() - 0.5;
    for (size_t q = 0; q < g.elems; q++) const_cast<float *>(p.eps)[q] = (float)(1 + 5 * uniform());
    for (int c = 0; c < 3; c++) old[c].assign(p.F[c], p.F[c] + g.elems);
    const sbp::Sweep w = g.sweep(true, 1, 2);
    launch({w.ctas, 1, 1}, {sbp::kSweepThreads, 1, 1}, [&] { sbp::half_e<unsigned, double, double, false, 1>(p, w); });
    int bad = 0;
    for (int k = 2; k <= n[2] - 2; k++)
        for (int j = 2; j <= n[1] - 2; j++)
            for (int i = 2; i <= n[0] - 2; i++) {
                const long long o = k * g.sz + j * g.sy + i;
                check<0>(p, old[0], o, bad);
                check<1>(p, old[1], o, bad);
                check<2>(p, old[2], o, bad);
            }
    std::printf("%d\n", bad);
}
"""


def test_interior_e_divides(tmp_path):
    exe = host_replay.build(str(tmp_path), MAIN_E)
    assert int(subprocess.run([exe], capture_output=True, check=True, text=True).stdout) == 0


def test_interior_h_rounds_once_at_the_field(tmp_path):
    exe = host_replay.build(str(tmp_path), MAIN)
    worst = float(subprocess.run([exe], capture_output=True, check=True, text=True).stdout)
    assert 0.4 < worst <= 0.5 * (1 + 2.0 ** -8)
