"""The solver's tables on the host (no GPU): csrc/setup.cpp compiled into a small
program that checks what it builds against 113-bit arithmetic.

- the pressure response to a unit wall datum, which the wall correction is made
  of, is rounded once (2^-52 of its largest value, however close to singular the
  matrix is);
- the multipliers of the two-sided factorisation are rounded once, to 2^-58, and
  the reciprocals of its diagonal to 2^-54 of each;
- the space that contexts reserve and report for the tables holds either form;
- which grids the integer solver takes: every unstretched one of 21 to 768
  radial points at any Reynolds number, time step and length, and no other size;
  stretched ones by their row sums."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include "csrc/setup.cpp"
#include <cstdio>
#include <cstdlib>
using namespace pnop;
#ifdef __SIZEOF_FLOAT128__
typedef __float128 quad;
#else
typedef long double quad;
#endif
static quad mag(quad x) { return x < 0 ? -x : x; }

static HostOps build(int nr, int M, int K, double Lz, double Re, double dt, double stretch) {
    HostOps h;
    h.d.nr = nr;
    h.d.M = M;
    h.d.K = K;
    h.d.nm = 2 * M + 1;
    h.d.nk = K + 1;
    h.d.nth = 3 * (M + 1);
    h.d.nzp = 3 * (K + 1);
    h.d.Lz = Lz;
    h.d.stretch = stretch;
    h.ph = {Re, 8.0, 1.0, dt, 0.0};
    std::string err;
    if (!build_grid(h, err) || !build_operators(h, err)) {
        std::printf("%s\n", err.c_str());
        std::exit(2);
    }
    return h;
}
static long long units(double word) {
    long long v;
    std::memcpy(&v, &word, sizeof v);
    return ((long long)(int)(v >> 32) << 32) + (int)(unsigned)(v & 0xFFFFFFFFll);
}
int main(int argc, char** argv) {
    const std::string what = argv[1];
    if (what == "response") {
        double worst = 0;
        for (int nr : {24, 48, 64})
            for (double Lz : {8.0, 100.0, 1000.0}) {
                const HostOps h = build(nr, 2, 3, Lz, 2000.0, 0.005, 0.0);
                for (int m = 0; m <= 2; ++m)
                    for (int k = 1; k <= 3; k += 2) {
                        const Band A = pressure_band(h, m, 2.0 * M_PI * k / Lz);
                        std::vector<std::vector<quad>> a(nr, std::vector<quad>(nr + 1, 0));
                        for (int i = 0; i < nr; ++i)
                            for (int j = std::max(0, i - kLo); j <= std::min(nr - 1, i + kUp); ++j) a[i][j] = A.get(i, j);
                        a[0][nr] = 1;
                        for (int c = 0; c < nr; ++c) {
                            int p = c;
                            for (int i = c + 1; i < nr; ++i)
                                if (mag(a[i][c]) > mag(a[p][c])) p = i;
                            std::swap(a[p], a[c]);
                            for (int i = c + 1; i < nr; ++i) {
                                const quad f = a[i][c] / a[c][c];
                                for (int j = c; j <= nr; ++j) a[i][j] -= f * a[c][j];
                            }
                        }
                        quad top = 0, off = 0;
                        for (int i = nr - 1; i >= 0; --i) {
                            for (int j = i + 1; j < nr; ++j) a[i][nr] -= a[i][j] * a[j][nr];
                            a[i][nr] /= a[i][i];
                            top = std::max(top, mag(a[i][nr]));
                            off = std::max(off, mag(a[i][nr] - (quad)h.phi[((size_t)m * h.d.nk + k) * nr + i]));
                        }
                        worst = std::max(worst, (double)(off / top));
                    }
            }
        std::printf("%.3g\n", worst);
        return worst <= std::ldexp(1.0, -52) ? 0 : 1;
    }
    if (what == "multipliers") {
        double worst = 0, inverse = 0;
        for (int nr : {24, 41, 64}) {
            const HostOps h = build(nr, 2, 3, 25.0, 2000.0, 0.005, 0.0);
            const FxShape f = fx_shape(nr);
            for (int m = 0; m <= 2; ++m)
                for (int k = 1; k <= 3; ++k)
                    for (int helm = 0; helm < 2; ++helm) {
                        const FixedTable& t = helm ? h.fxH : h.fxP;
                        if (!t.ok) return 3;
                        const double kz = 2.0 * M_PI * k / 25.0;
                        const Band A = helm ? helmholtz_band(h, m, kz) : pressure_band(h, m, kz);
                        std::vector<std::vector<quad>> a(nr, std::vector<quad>(nr, 0));
                        for (int i = 0; i < nr; ++i)
                            for (int j = std::max(0, i - kLo); j <= std::min(nr - 1, i + kUp); ++j) a[i][j] = A.get(i, j);
                        for (int c = 0; c < f.h - 4; ++c) {  // side 0 is plain elimination from row 0
                            const size_t out = (size_t)m * f.tile + f.out[0] + (size_t)(c / 4) * 20 * kTileX + 16 * kTileX + k;
                            const long long d = units(t.direct[out + (size_t)(c % 4) * kTileX]);
                            int code = (int)(d & 0xFF);
                            if (c >= 4)
                                for (int r = code = 0; r < 4; ++r)
                                    code |= (int)(units(t.direct[out + (size_t)r * kTileX]) & 3) << 2 * r;
                            const quad off = (quad)d * a[c][c] * (quad)std::ldexp(1.0, code - 128 - 60) - 1;
                            inverse = std::max(inverse, (double)mag(off));
                            for (int i = c + 1; i <= c + 4; ++i) {
                                const quad l = a[i][c] / a[c][c];
                                for (int j = c; j < nr; ++j) a[i][j] -= l * a[c][j];
                                const size_t at = (size_t)m * f.tile + f.in[0] +
                                                  (((size_t)i * 2 + (c - i + 4) / 2) * kTileX + k) * 2 + (c - i + 4) % 2;
                                const quad want = -l * (quad)std::ldexp(1.0, kFxBits - (c == 0 ? t.shift : 0));
                                worst = std::max(worst, (double)mag((quad)units(t.direct[at]) - want));
                            }
                        }
                    }
        }
        std::printf("%.3g units, 1/D %.3g\n", worst, inverse);
        if (!(inverse <= std::ldexp(1.0, -54))) return 1;
        return worst <= 2.0 ? 0 : 1;  // one to nearest, one where the low digit is kept above -2^31
    }
    if (what == "grids") {
        for (int nr : {9, 16, 20, 21, 22, 23, 24, 25, 27, 32, 41, 48, 64, 81, 100, 128, 200, 400, 768, 769})
            for (double Lz : {0.5, 8.0, 1000.0})
                for (double Re : {1.0, 2000.0, 1.0e5})
                    for (double dt : {1e-5, 0.005, 1.0}) {
                        if (nr > 200 && (Lz != 8.0 || Re != 2000.0 || dt != 0.005)) continue;
                        const HostOps h = build(nr, nr > 200 ? 2 : 7, 3, Lz, Re, dt, 0.0);
                        const bool want = nr >= 21 && nr <= 768;
                        if (h.fxP.ok != want || h.fxH.ok != want) {
                            std::printf("nr %d Lz %g Re %g dt %g: pressure %d Helmholtz %d\n", nr, Lz, Re, dt, h.fxP.ok, h.fxH.ok);
                            return 1;
                        }
                    }
        const HostOps s = build(32, 2, 5, 8.0, 1800.0, 0.005, 0.1);  // wide stencils: sums above kFxRowSum
        return s.fxP.ok || !s.fxH.ok || s.facP.empty() || !s.facH.empty();
    }
    if (what == "sizes") {
        for (int nr = 9; nr <= 800; ++nr)
            for (int nk : {2, 16, 17, 32, 33, 128, 129})
                if (factor_words(nr, nk) < (nk + kTileX - 1) / kTileX * fx_shape(nr).tile ||
                    factor_words(nr, nk) < (size_t)((nk + kTileK - 1) / kTileK) * nr * kBand * kTileK)
                    return 1;
        const HostOps h = build(21, 2, 31, 8.0, 1800.0, 0.005, 0.0);
        return !(h.fxP.direct.size() <= 3 * factor_words(21, 32) && h.fxH.transposed.size() <= 4 * factor_words(21, 32));
    }
    return 4;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("tables")
    src, exe = d / "tables.cpp", d / "tables"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-O2", "-std=c++17", "-pthread", "-I", os.path.join(ROOT, "paper_2509_10103_gb300"), str(src), "-o", str(exe)],
                   check=True)
    return str(exe)


@pytest.mark.parametrize("what", ["response", "multipliers", "grids", "sizes"])
def test_tables(program, what):
    p = subprocess.run([program, what], stdout=subprocess.PIPE, text=True, timeout=600)
    assert p.returncode == 0, p.stdout
