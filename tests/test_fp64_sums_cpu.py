"""The integer sums of the FP64 flow collision, host-compiled.

* Conversions: fx_load, fx_double and fx_store give the doubles that the compiler's own
  conversions give (to nearest even), and fx_corr keeps every bit of a correction down to 2^-33.
* One collision against quadruple precision, over states near the rest weights with a share of
  solid and mushy nodes: errors in ulps of f* no larger than those of FP64 sums.
* The largest moments that populations in range can have do not overflow 64 bits.
* Mass of a periodic box with buoyancy and melting: rounding to nearest changes the sum of the
  populations of a node by 0.29 ulp rms each, 2^-54 for f_0 and less for the others, in either
  direction, so steps over N nodes move the mean by 0.29 x 2^-54 sqrt(steps / N).
"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HARNESS = r"""
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "lbpc_host.h"
#include "lbpc_kernels.cuh"
using namespace lbpc;
#if defined(__SIZEOF_FLOAT128__)
typedef __float128 Quad;
#else
typedef long double Quad;  // 113 bits where there is no __float128
#endif
static uint64_t st = 20170309;
static uint64_t bits() { return st = st * 6364136223846793005ULL + 1442695040888963407ULL; }
static double rnd() { return ((bits() >> 11) * (1.0 / 9007199254740992.0)) * 2 - 1; }  // [-1, 1)
static const double w[19] = {1. / 3, 1. / 18, 1. / 18, 1. / 18, 1. / 18, 1. / 18, 1. / 18,
                             1. / 36, 1. / 36, 1. / 36, 1. / 36, 1. / 36, 1. / 36,
                             1. / 36, 1. / 36, 1. / 36, 1. / 36, 1. / 36, 1. / 36};
static Args a;
static void setup(int n, double Pr, int wall, double rate) {
    lbpc_params p;
    std::memset(&p, 0, sizeof p);
    p.flow_model = LBPC_FLOW_MRT; p.enth_model = LBPC_ENTH_MRT; p.precision = LBPC_FP64;
    for (int f = 0; f < 6; f++) p.bc[f] = wall;
    p.Ra = 1e5; p.Pr = Pr; p.St = 0.5; p.Ma = 0.1; p.s_e = p.s_eps = rate;
    p.Th = 1; p.Tref = 0.3; p.Cp_s = p.Cp_l = p.Cp_ref = 1; p.omega_T = 0.25; p.h0 = -1;
    Derived d; std::string e;
    if (!validate_and_map(n, n, n, &p, d, e)) { puts(e.c_str()); exit(2); }
    double* Tw[6] = {};
    fill_args(a, n, n, n, p, d, Tw);
}
// the same collision coefficients in quadruple precision
static Coef<Quad> quad(const Coef<double>& k) {
    Coef<Quad> q{};
    q.gbeta = k.gbeta; q.Tref = k.Tref; q.frho = k.frho;
    q.r_e = k.r_e; q.r_eps = k.r_eps; q.r_q = k.r_q; q.r_nu9 = k.r_nu9; q.r_pi10 = k.r_pi10;
    q.r_nu11 = k.r_nu11; q.r_pi12 = k.r_pi12; q.r_nu13 = k.r_nu13; q.r_t = k.r_t;
    q.c_e = k.c_e; q.c_eps = k.c_eps; q.c_q = k.c_q; q.c_nu9 = k.c_nu9; q.c_pi10 = k.c_pi10;
    q.c_nu11 = k.c_nu11; q.c_pi12 = k.c_pi12; q.c_nu13 = k.c_nu13;
    return q;
}
static Quad value(FxCorr c) { return (Quad)(long long)c.h * (Quad)0x1p24 + c.l; }  // units of 2^-85
static int conversions() {
    long bad = 0;
    for (int t = 0; t < 2000000; t++) {
        bool ok = true;
        const double f = std::ldexp(1 + (rnd() + 1) / 2, -6 + (int)(bits() >> 40) % 5);
        const long long F = fx_load(f, ok);
        if (f < 0.5) bad += !ok || (double)F * 0x1p-58 != f;
        const long long x = (long long)bits() >> ((bits() >> 40) % 64);
        const unsigned long long ax = x < 0 ? 0ull - (unsigned long long)x : (unsigned long long)x;
        Quad half = 0.5;  // unit of the last of its 53 bits
        for (int n = 53; n < 64 && ax >> n; n++) half *= 2;
        const Quad err = (Quad)fx_double(x) * (Quad)0x1p58 - (Quad)x;
        bad += ax >> 53 ? err > half || err < -half : err != 0;
        ok = true;
        const double d = std::ldexp(rnd(), -4 - (int)((bits() >> 40) % 28));
        const FxCorr c = fx_corr(d, ok);
        if (std::fabs(d) >= 0x1p-33) bad += !ok || value(c) != (Quad)d * (Quad)0x1p85;
        const double small = std::ldexp(rnd(), -33 - (int)((bits() >> 40) % 90));
        const Quad off = value(fx_corr(small, ok)) - (Quad)small * (Quad)0x1p85;
        bad += !ok || off > (Quad)0.5 || off < (Quad)-0.5;
        // stores: sums of corrections of every size, ties made by clearing the low bits
        FxCorr v = 3 * c - fx_corr(small, ok);
        if (t % 3 != 0) v.l = (int)((bits() >> 33) % 3) << 24;
        if (t % 3 == 2) v.h &= ~0x7ull;
        bool in = true;
        const double s = fx_store(F, v, in);
        const Quad sum = (Quad)F * (Quad)0x1p27 + value(v);
        if (sum >= (Quad)0x1p78) bad += !in || s != (double)sum * 0x1p-85;
        else bad += in;
    }
    bool ok = true;
    bad += value(fx_corr(0.0, ok)) != 0 || value(fx_corr(-0.0, ok)) != 0 || fx_double(0) != 0.0 || !ok;
    fx_corr(0x1p-4, ok);
    bad += ok;
    printf("%ld\n", bad);
    return 0;
}
// rms and largest error of a collision in ulps of f*: integer sums, FP64 sums
static void errors(double Pr) {
    setup(32, Pr, LBPC_ADIABATIC, 0);
    const Coef<Quad> kq = quad(a.cd);
    double s2[2] = {}, mx[2] = {};
    long n = 0, out = 0;
    for (int t = 0; t < 40000; t++) {
        double f[2][19];
        Quad r[19];
        for (int q = 0; q < 19; q++) f[0][q] = f[1][q] = w[q] * (1 + 0.05 * rnd());
        for (int q = 0; q < 19; q++) r[q] = f[0][q];
        const double T = rnd(), fl = t % 4 == 0 ? 0 : t % 4 == 1 ? 0.5 + 0.5 * rnd() : 1;
        double u[3], m[4];
        Quad uq[3], mq[4];
        long long F[19];
        if (!flow_fx_load(f[0], F) || !collide_flow_fx(F, f[0], a.cd, T, fl, u[0], u[1], u[2], m[0], m[1], m[2], m[3])) { out++; continue; }
        collide_flow<false>(f[1], a.cd, T, fl, u[0], u[1], u[2], m[0], m[1], m[2], m[3]);
        collide_flow<false>(r, kq, (Quad)T, (Quad)fl, uq[0], uq[1], uq[2], mq[0], mq[1], mq[2], mq[3]);
        for (int q = 0; q < 19; q++)
            for (int i = 0; i < 2; i++) {
                int ex;
                std::frexp((double)r[q], &ex);
                const double e = std::fabs((double)((Quad)f[i][q] - r[q])) * std::ldexp(1.0, 53 - ex);
                s2[i] += e * e;
                mx[i] = e > mx[i] ? e : mx[i];
                n += i == 0;
            }
    }
    printf("%g %g %g %g %ld\n", std::sqrt(s2[0] / n), mx[0], std::sqrt(s2[1] / n), mx[1], out);
}
// change of the mean density of an n^3 periodic box
static void drift(int n, int steps) {
    setup(n, 0.7, LBPC_PERIODIC, 0);
    const int N = n * n * n;
    std::vector<double> f[2], g[2], hp(N), Qf(19 * N), h(N);
    for (int i = 0; i < 2; i++) { f[i].resize(19 * N); g[i].resize(6 * N); }
    for (int m = 0; m < N; m++) {
        h[m] = a.hs + a.L * (1 + 0.8 * rnd());
        for (int q = 0; q < 19; q++) Qf[q * N + m] = w[q] * (1 + 0.02 * rnd());
    }
#define EACH(call) for (int z = 0; z < n; z++) for (int y = 0; y < n; y++) for (int x = 0; x < n; x++) call
    EACH((init_node<LBPC_FP64, LAYOUT_PULL, true, true>(a, x, y, z, Qf.data(), nullptr, h.data(),
                                                        f[0].data(), g[0].data(), hp.data())));
    auto mass = [&](const std::vector<double>& v) { Quad s = 0; for (double x : v) s += x; return s; };
    const Quad before = mass(f[0]);
    for (int s = 0; s < steps; s++)
        EACH((step_node<LBPC_FP64, STEP_PULL, 1>(a, x, y, z, f[s & 1].data(), f[1 - (s & 1)].data(),
                                                 g[s & 1].data(), g[1 - (s & 1)].data(), hp.data())));
    printf("%g\n", (double)((mass(f[steps & 1]) - before) / N));
}
// moving populations at the upper bound, f_0 small: m2 = 9 f_0 - 7 sum f_1..6 - 2 sum f_7..18 is
// near -33; low relaxation rates, so that the correction stays in range whatever the moment is
static void largest_moments() {
    setup(32, 0.7, LBPC_ADIABATIC, 0.01);
    const Coef<Quad> kq = quad(a.cd);
    double worst = 0;
    for (double f0 = 0x1p-6; f0 < 0.5; f0 += 0x1p-8)
        for (double top : {std::nextafter(0.5, 0.0), 0.45, 0.3, 0.2}) {
            double f[19], u[3], m[4];
            Quad r[19], uq[3], mq[4];
            long long F[19];
            for (int q = 0; q < 19; q++) r[q] = f[q] = q ? top : f0;
            if (!flow_fx_load(f, F) || !collide_flow_fx(F, f, a.cd, 0.3, 1.0, u[0], u[1], u[2], m[0],
                                                        m[1], m[2], m[3]))
                continue;  // FP64 sums take it
            collide_flow<false>(r, kq, (Quad)0.3, (Quad)1, uq[0], uq[1], uq[2], mq[0], mq[1], mq[2], mq[3]);
            for (int q = 0; q < 19; q++) worst = std::fmax(worst, std::fabs((double)((Quad)f[q] - r[q])));
        }
    printf("%g\n", worst);
}
int main(int argc, char** argv) {
    if (argv[1][0] == 'c') return conversions();
    if (argv[1][0] == 'e') errors(atof(argv[2]));
    if (argv[1][0] == 'm') largest_moments();
    if (argv[1][0] == 'd') drift(atoi(argv[2]), atoi(argv[3]));
    return 0;
}
"""


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    # by g++ alone: nvcc takes no quadruple precision in functions that are also device code
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc) or not shutil.which("g++"):
        pytest.skip("no CUDA headers or no g++")
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    d = tmp_path_factory.mktemp("fp64_sums")
    src, exe = d / "fx.cpp", d / "fx"
    src.write_text(HARNESS)
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-I", cuda, "-I",
                    os.path.join(ROOT, "include"), "-I",
                    os.path.join(ROOT, "paper_1703_02652_gb300", "csrc"), str(src), "-o", str(exe)],
                   check=True, capture_output=True)

    def run(*args):
        out = subprocess.run([str(exe), *map(str, args)], check=True, capture_output=True, text=True)
        return [float(v) for v in out.stdout.split()]
    return run


def test_conversions_round_once_to_nearest_even(harness):
    assert harness("conversions") == [0]


@pytest.mark.parametrize("Pr", [0.02, 0.7, 50.0])
def test_error_of_a_collision_is_no_larger_than_with_fp64_sums(harness, Pr):
    rms, largest, rms64, largest64, rejected = harness("errors", Pr)
    assert rejected == 0
    assert rms <= rms64 and largest <= largest64
    # half an ulp from the store, the rest from the products of the corrections
    assert rms <= 0.35 and largest <= 1.0


def test_moments_do_not_overflow(harness):
    # populations below 1, moments up to 33: a few roundings of f* and of the corrections
    assert harness("moments")[0] <= 4 * 2.0 ** -53


def test_mass_does_not_drift(harness):
    n, steps = 8, 3000
    sigma = 0.29 * 2.0 ** -54 * (steps / n ** 3) ** 0.5
    assert abs(harness("drift", n, steps)[0]) <= 6 * sigma
