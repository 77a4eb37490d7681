"""The pair kernels' 32-bit offsets at the largest lattices that the dispatch hands to them.

The pair paths form element offsets in int (pairs_fit() in lbpc_kernels.cuh); the per-node path
forms them in 64 bits.  The header is compiled as host code with wrapping integers, as on the
device, and both run on the last node pairs, the x-face pairs and the first ones of lattices
just inside the limits, in reserved address space of which only the slots around those nodes
are touched.  Gathers have to return equal values; the AA and the reverse step equal stores up
to rounding of the collision.  An offset that wraps reads gigabytes away.
"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HARNESS = r"""
#include <sys/mman.h>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include "lbpc_host.h"
#include "lbpc_kernels.cuh"
using namespace lbpc;
constexpr int P = LBPC_FP32;
template <class T> T* reserve(size_t n) {
    void* p = mmap(nullptr, n * sizeof(T), PROT_READ | PROT_WRITE,
                   MAP_PRIVATE | MAP_ANONYMOUS | MAP_NORESERVE, -1, 0);
    if (p == MAP_FAILED) { puts("no address space"); exit(3); }
    return (T*)p;
}
static float hashed(size_t i, unsigned salt) {  // in (-1, 1), never zero
    uint64_t h = (i + 1) * 0x9e3779b97f4a7c15ull + salt * 0xbf58476d1ce4e5b9ull;
    h ^= h >> 31; h *= 0x94d049bb133111ebull; h ^= h >> 29;
    return (float)((int)(h >> 41) | 1) * (1.f / 8388608.f) * 2 - 1;
}
static Args a;
static long bad = 0;
static void near(double v, double w, double tol, const char* what, int q) {
    if (!(std::fabs(v - w) <= tol)) { bad++; if (bad < 20) printf("%s %d: %g %g\n", what, q, v, w); }
}
template <class F> void around(int x0, int y, int z, F fn) {  // the pair and its neighbours
    for (int dz = -1; dz <= 1; dz++)
        for (int dy = -1; dy <= 1; dy++)
            for (int dx = -1; dx <= 2; dx++) {
                const int x = (x0 + dx + a.nx) % a.nx, yy = (y + dy + a.ny) % a.ny,
                          zz = (z + dz + a.nz) % a.nz;
                fn((size_t)x + (size_t)a.nx * (yy + (size_t)a.ny * zz));
            }
}
int main(int argc, char** argv) {
    const int nx = atoi(argv[1]), ny = atoi(argv[2]), nz = atoi(argv[3]);
    lbpc_params p;
    std::memset(&p, 0, sizeof p);
    p.flow_model = LBPC_FLOW_MRT; p.enth_model = LBPC_ENTH_MRT; p.precision = P;
    for (int f = 0; f < 6; f++) p.bc[f] = atoi(argv[4 + f]);
    p.Ra = 1e6; p.Pr = 0.7; p.St = 0.1; p.Ma = 0.1;
    p.Th = 1; p.Tref = 0.5; p.Cp_s = p.Cp_l = p.Cp_ref = 1; p.omega_T = 0.25; p.h0 = -1;
    Derived d; std::string e;
    if (!validate_and_map(nx, ny, nz, &p, d, e)) { puts(e.c_str()); return 1; }
    const size_t N = (size_t)nx * ny * nz;
    double* Tw[6];
    for (int f = 0; f < 6; f++) {
        const size_t m = f < 2 ? (size_t)ny * nz : f < 4 ? (size_t)nx * nz : (size_t)nx * ny;
        Tw[f] = reserve<double>(m);
    }
    fill_args(a, nx, ny, nz, p, d, Tw);
    if (!pairs_fit(a)) { puts("not a pair lattice"); return 4; }
    float *f = reserve<float>(19 * N), *g = reserve<float>(6 * N), *lam = reserve<float>(26 * N);
    float *f2 = reserve<float>(19 * N), *g2 = reserve<float>(6 * N);
    float *lo = reserve<float>(26 * N), *lo2 = reserve<float>(26 * N);
    float *te = reserve<float>(N), *tm = reserve<float>(4 * N);
    double *hp = reserve<double>(N), *hp2 = reserve<double>(N);
    double *gt = reserve<double>((size_t)ny * nz), *gt2 = reserve<double>((size_t)ny * nz);
    const int xs[3] = {0, nx / 2 / 2 * 2, nx - 2};
    for (int x0 : xs)
        for (int y : {0, 1, ny - 2, ny - 1})
            for (int z : {0, 1, nz - 2, nz - 1}) {
                around(x0, y, z, [&](size_t m) {
                    for (int q = 0; q < 19; q++) f[q * N + m] = f2[q * N + m] = 0.01f * hashed(q * N + m, 1);
                    for (int q = 0; q < 6; q++) g[q * N + m] = g2[q * N + m] = 0.1f * hashed(q * N + m, 2);
                    for (int q = 0; q < 26; q++) lam[q * N + m] = hashed(q * N + m, 3);
                    hp[m] = hp2[m] = hashed(m, 4);
                    te[m] = hashed(m, 5);
                    for (int q = 0; q < 4; q++) tm[q * N + m] = 0.05f * hashed(q * N + m, 6);
                });
                const bool inner = inner_row(a, y, z);
                const int n0 = x0 + nx * (y + ny * z);
                // pull gathers, as the row takes them
                float fa[2][19], ga[2][7], fb[19], gb[7];
                double2 ep;
                if (inner)
                    gather_pair_pull<P, true>(a, NbInterior{nx, nx * ny}, x0, y, z, f, g, hp, fa[0],
                                              fa[1], ga[0], ga[1], ep);
                else
                    gather_pair_pull<P, true>(a, make_nb(a, x0, y, z), x0, y, z, f, g, hp, fa[0],
                                              fa[1], ga[0], ga[1], ep);
                for (int i = 0; i < 2; i++) {
                    const Nb b = make_nb(a, x0 + i, y, z);
                    gather_f<P, LAYOUT_PULL, false>(a, b, n0 + i, f, fb);
                    gather_g<P, LAYOUT_PULL, false>(a, b, n0 + i, x0 + i, y, z, g, gb);
                    for (int q = 0; q < 19; q++) near(fa[i][q], fb[q], 0, "f", q);
                    for (int q = 1; q < 7; q++) near(ga[i][q], gb[q], 0, "g", q);
                }
                // reverse step
                if (inner)
                    adj_reverse_pair<P, true>(a, NbInterior{nx, nx * ny}, x0, y, z, lam, lo, te, tm, 0, gt);
                else
                    adj_reverse_pair<P, true>(a, make_nb(a, x0, y, z), x0, y, z, lam, lo, te, tm, 0, gt);
                for (int i = 0; i < 2; i++)
                    adj_reverse_node<P, true>(a, make_nb(a, x0 + i, y, z), x0 + i, y, z, lam, lo2,
                                              te, tm, 0, gt2);
                for (int q = 0; q < 26; q++)
                    for (int i = 0; i < 2; i++)
                        near(lo[q * N + n0 + i], lo2[q * N + n0 + i], 2e-4, "lambda", q);
                if (!inner) continue;
                // AA odd step, in place
                step_pair_aa<P, 1, true>(a, x0, y, z, f, g, hp);
                for (int i = 0; i < 2; i++)
                    step_node<P, STEP_AA_ODD, 1>(a, x0 + i, y, z, f2, f2, g2, g2, hp2);
                around(x0, y, z, [&](size_t m) {
                    for (int q = 0; q < 19; q++) near(f[q * N + m], f2[q * N + m], 1e-6, "AA f", q);
                    for (int q = 0; q < 6; q++) near(g[q * N + m], g2[q * N + m], 1e-6, "AA g", q);
                });
            }
    printf("%ld differences\n", bad);
    return bad != 0;
}
"""


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    d = tmp_path_factory.mktemp("pair_offsets")
    src, exe = d / "pairs.cu", d / "pairs"
    src.write_text(HARNESS)
    subprocess.run([nvcc, "-std=c++17", "-O1", "-Xcompiler", "-fwrapv,-ffp-contract=off", "-I",
                    os.path.join(ROOT, "include"), "-I",
                    os.path.join(ROOT, "paper_1703_02652_gb300", "csrc"), str(src), "-o", str(exe)],
                   check=True, capture_output=True)
    return str(exe)


# walls: 2^29 nodes at most (here and in the last one, one plane below), (2^31 - 1) / 3 without;
# ISOTHERMAL, ADIABATIC and PERIODIC as in lbpc.h
@pytest.mark.parametrize("shape,bc", [((1024, 1024, 511), (1, 2, 2, 2, 2, 2)),
                                      ((1024, 1024, 511), (0, 0, 1, 1, 2, 2)),
                                      ((1024, 1024, 511), (0, 0, 0, 0, 1, 2)),
                                      ((1024, 1024, 682), (0, 0, 0, 0, 0, 0)),
                                      ((6, 4, 5), (1, 2, 2, 2, 2, 1))])
def test_pair_and_node_paths_read_the_same_slots(harness, shape, bc):
    r = subprocess.run([harness, *map(str, shape), *map(str, bc)], capture_output=True, text=True)
    if r.returncode == 3:
        pytest.skip("no address space to reserve")
    assert r.returncode == 0, (r.returncode, r.stdout)


def test_the_dispatch_sends_larger_lattices_to_the_node_path(harness):
    for shape, bc in (((1024, 1024, 512), (1, 2, 2, 2, 2, 2)), ((1024, 1024, 600), (0, 0, 0, 0, 1, 2)),
                      ((1024, 1024, 683), (0,) * 6), ((7, 4, 5), (0,) * 6)):
        r = subprocess.run([harness, *map(str, shape), *map(str, bc)], capture_output=True, text=True)
        assert r.returncode == 4, (shape, r.returncode, r.stdout)
