"""The unit and the range of the double-float mode's force split (df_split in
csrc/lsm_internal.h), on the CPU."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")

HARNESS = r"""
#include "lsm_internal.h"
#include <cstdio>
#include <random>
using namespace lsm;
static std::mt19937_64 rg(5);
static double uni(double a, double b) { return a + (b - a) * (double)(rg() >> 11) * 0x1p-53; }

struct Mat { double k, e; };
// [phase][phase][shell] of nphase materials, interfaces the two half springs in series
static std::vector<SpringType> table(const std::vector<Mat> &m, double a, double k2, double diag)
{
    std::vector<SpringType> t;
    for (const Mat &p : m)
        for (const Mat &q : m)
            for (int s = 0; s < 2; s++) {
                const double k = p.k + q.k > 0 ? 2 * p.k * q.k / (p.k + q.k) : 0.0, r0 = s ? a * diag : a;
                const double rc = r0 * (1 + 0.5 * (p.e + q.e));
                t.push_back(SpringType{s ? k * k2 : k, r0, rc * rc, 0.0});
            }
    return t;
}

// The strain, positive or negative, at which type t leaves the plain sums' range
static double strain_of(const SpringType &t, double cmax, int sign)
{
    return sign > 0 ? (cmax < t.k ? cmax / (t.k - cmax) : INFINITY) : cmax / (t.k + cmax);
}

int main()
{
    long bad = 0;
#define CHECK(x) do { if (!(x)) { bad++; std::printf("%s (line %d)\n", #x, __LINE__); } } while (0)
    // any spacing: the range in strains is the same up to the unit's power of two
    const int springs[3][2] = {{4, 4}, {2, 4}, {6, 12}};
    const double diag[3] = {std::sqrt(2.0), 1.0, std::sqrt(2.0)};
    for (int d = 0; d < 3; d++)
        for (double a = 0x1p-20; a < 2e6; a *= d == 1 ? 3.0 : 2.0) {
            const auto t = table({{1.0, 0.05}, {0.1, 0.3}}, a, 1.0, diag[d]);
            const DfSplit s = df_split(t, springs[d][0], springs[d][1]);
            // a contrast of ten: the stiff phase stays in the range up to its critical
            // strain on the square lattice, to half of that (a unit of any rounding) on
            // the packing; 3D: 2^24 units of 2^-26 over forces of 6 + 12 sqrt 2 lengths, 0.0109
            // less a tenth (a soft spring has the same factor at a greater length)
            const double in_range[3] = {0.05, 0.025, 0.009};
            CHECK(strain_of(t[0], s.cmax, 1) > in_range[d]);
            CHECK(strain_of(t[0], s.cmax, -1) > 0.96 * in_range[d]);
            if (d != 1) {
                const DfSplit one = df_split(table({{1.0, 0.05}, {0.1, 0.3}}, 1.0, 1.0, diag[d]), springs[d][0], springs[d][1]);
                CHECK(s.unit == a * one.unit && std::fabs(s.cmax / one.cmax - 1) < 1e-9);
            }
        }
    for (int i = 0; i < 20000; i++) {
        const int d = (int)(rg() % 3), np = 1 + (int)(rg() % 3);
        std::vector<Mat> m;
        for (int p = 0; p < np; p++)
            m.push_back({rg() % 8 == 0 ? 0.0 : std::exp(uni(-14, 14)), rg() % 8 == 0 ? INFINITY : std::exp(uni(-6, 7)) - 0.5 * (rg() % 8 == 0)});
        const double a = std::exp(uni(-10, 10));
        const auto t = table(m, a, uni(0.3, 1.5), diag[d]);
        const DfSplit s = df_split(t, springs[d][0], springs[d][1]);
        CHECK(std::isfinite(s.unit) && s.unit > 0 && std::isfinite(s.cmax) && s.cmax >= 0);
        int e;
        CHECK(std::frexp(s.unit, &e) == 0.5);
        double soft = INFINITY;
        for (const SpringType &q : t)
            if (q.k > 0) soft = std::fmin(soft, q.k * q.r0);
        CHECK(s.unit <= soft * std::exp2(d == 2 ? -22.0 : -21.5));
        if (std::isfinite(soft)) CHECK(s.cmax > 0);
        // intact springs of one particle with |c| <= cmax never leave the range
        for (int rep = 0; rep < 20; rep++) {
            const int p = (int)(rg() % np);
            double sum = 0;
            for (int sh = 0; sh < 2; sh++)
                for (int n = 0; n < springs[d][sh]; n++) {
                    const int q = (int)(rg() % np);
                    const SpringType &y = t[(size_t)(rg() % 2 ? p * np + q : q * np + p) * 2 + sh];
                    if (!(y.k > 0)) continue;
                    double lo = y.r0 * y.k / (y.k + s.cmax), hi = std::sqrt(y.rc2);
                    if (s.cmax < y.k) hi = std::fmin(hi, y.r0 * y.k / (y.k - s.cmax));
                    CHECK(hi < INFINITY || std::isinf(s.cmax));
                    if (!(lo <= hi && hi < INFINITY)) continue;  // broken before its factor is small
                    const double r = rep < 4 ? (rep & 1 ? lo : hi) : uni(lo, hi);
                    if (r <= std::sqrt(y.rc2)) sum += std::fabs(y.k * (r - y.r0));
                }
            CHECK(sum <= s.unit * 0x1p24);
        }
    }
    std::printf("%ld\n", bad);
    return bad != 0;
}
"""


def test_split_unit_and_range(tmp_path):
    """For random tables (contrasts up to e^28, spacings e^-10 to e^10, unbreakable
    and zero springs, the three lattices' spring counts): the unit is a power of
    two below its line, and whatever intact springs with factors up to cmax a
    particle has, their forces sum within the exact range. Two-phase tables: the
    range covers the strains in use at every lattice spacing."""
    gxx = shutil.which("g++")
    if gxx is None or not os.path.exists(os.path.join(CUDA, "cuda_runtime.h")):
        pytest.skip("no g++ or no CUDA headers")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(HARNESS)
    subprocess.check_call([gxx, "-O2", "-std=c++17", "-I", os.path.join(ROOT, "paper_2201_04565_gb300", "csrc"),
                           "-I", CUDA, "-c", "-o", str(tmp_path / "t.o"), str(src)])
    subprocess.check_call([gxx, "-o", str(exe), str(tmp_path / "t.o"), "-Wl,--unresolved-symbols=ignore-all"])
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0 and out.stdout.strip() == "0", out.stdout[-2000:]
