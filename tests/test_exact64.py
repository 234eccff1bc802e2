"""The FP64 operations that the EXACT64 kernels evaluate on the integer and
FP32 pipes (csrc/exact64.cuh), bit for bit: on the CPU against the C
operators, with the hardware estimate replaced by one that is off by up to
2^-22 in either direction, and on the GPU, in the spring kernels, against the
oracle at units where their range checks hand over to the FP64 pipe."""
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HARNESS = r"""
#include "exact64.cuh"
#include <cstdio>
#include <random>
using namespace lsm;
static std::mt19937_64 rg(12345);
static float estimate(float m, int k)
{
    const double u = k == 0 ? 1.0 : k == 1 ? -1.0 : 2.0 * (double)(rg() >> 11) * 0x1p-53 - 1.0;
    return (float)((1.0 + u * 0x1p-22) / std::sqrt((double)m));
}
// significands at the edges: all zeros, all ones, few bits set, random
static uint64_t sig(int k)
{
    const uint64_t full = 0xFFFFFFFFFFFFFull;
    if (k == 0) return rg() % 4;
    if (k == 1) return full - rg() % 4;
    if (k == 2) return (rg() & 0x7FFFFFFull) << 25;
    return rg() & full;
}
int main()
{
    long bad = 0;
    for (long i = 0; i < 2000000; i++) {
        // the whole normal range, and the lengths of a lattice
        const uint64_t e = i % 2 ? 1 + rg() % 2046 : 1010 + rg() % 30;
        uint64_t x = (e << 52) | sig((int)(i % 7));
        if (i % 5 == 0) {  // neighbours of squares: roots next to a representable number
            const double d = (double)((rg() >> 11) | 0x10000000000000ull);
            x = e64_bits(d * d) + rg() % 5 - 2;
        }
        const double xd = e64_double(x), ref = std::sqrt(xd);
        const Root64 r = e64_sqrt(x, estimate(e64_sqrt_arg(x), (int)(i % 9)));
        bad += e64_bits(e64_root(r)) != e64_bits(ref);
        uint64_t a = rg();
        if (i % 3 == 0) a = (a & 0xFFF0000000000000ull) | ((r.R + rg() % 3 - 1) & 0xFFFFFFFFFFFFFull);
        if (i % 4 == 0) a = e64_bits(ref * e64_double(0x3FF0000000000000ull | sig(2))) + rg() % 3 - 1;
        if (e64_div_ok(a, r)) bad += e64_bits(e64_div(a, r)) != e64_bits(e64_double(a) / ref);
        const uint64_t b = (rg() & 0xFFF0000000000000ull) | sig((int)(i % 6));
        a = (rg() & 0xFFF0000000000000ull) | sig((int)(i % 4));  // 27-bit factors: ties
        bool ok = true;
        const uint64_t za = i % 11 ? a : a & 0x8000000000000000ull;
        double p = e64_mul(za, b, ok);
        if (ok) bad += e64_bits(p) != e64_bits(e64_double(za) * e64_double(b));
        ok = true;
        p = e64_sqr(za, ok);
        if (ok) bad += e64_bits(p) != e64_bits(e64_double(za) * e64_double(za));
        const double g[6] = {0.0, xd, e64_double(b & 0x7FFFFFFFFFFFFFFFull), INFINITY, NAN, -NAN};
        for (int s = 0; s < 6; s++)
            for (int t = 0; t < 4; t++) bad += !std::isnan(g[t]) && e64_gt(g[s], g[t]) != (g[s] > g[t]);
        bad += e64_zero(x) || !e64_zero(0) || !e64_zero(0x8000000000000000ull);
    }
    std::printf("%ld\n", bad);
    return bad != 0;
}
"""


def test_operations_are_correctly_rounded(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(HARNESS)
    subprocess.check_call([gxx, "-O2", "-std=c++17", "-ffp-contract=off", "-I",
                           os.path.join(ROOT, "paper_2201_04565_gb300", "csrc"), "-o", str(exe), str(src)])
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0 and out.stdout.strip() == "0", out.stdout


@pytest.mark.gpu
@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("unit", [1.0, 1e-3, 1e-100, 1e-160, 1e150])
def test_spring_kernel_matches_oracle_at_every_scale(oracle_mod, dim, unit):
    """Random networks with lengths from where the squares underflow to where
    they come near overflow, unit and other spring constants and masses,
    springs at rest and zero components: states equal to the oracle's."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2201_04565_gb300 import lsm
    rng = np.random.default_rng(7 + dim)
    n = 300
    X = rng.integers(0, 4, (dim, n)).astype(float) + 6.0 * np.arange(n) / n
    X[:, 1] = X[:, 0] + 1.0
    X[-1, 2] = X[-1, 1]
    X *= unit
    si, sj = np.triu_indices(40, 1)
    keep = rng.random(si.size) < 0.4
    keep[0] = True
    si, sj = si[keep], sj[keep]
    si, sj = np.concatenate([si, np.arange(40, n - 1)]), np.concatenate([sj, np.arange(41, n)])
    r = np.sqrt(((X[:, sj] - X[:, si]) ** 2).sum(0))
    live = r > 0
    si, sj, r = si[live], sj[live], r[live]
    r0 = np.where(rng.random(r.size) < 0.2, r, unit * rng.choice([0.5, 1.0, 2.0], r.size))
    k = rng.choice([1.0, 0.1, 3.7], r.size)
    rc2 = np.where(rng.random(r.size) < 0.1, (1.0001 * r) ** 2, np.inf)
    mass = rng.choice([1.0, 2.0, 2.5], n)
    kw = dict(mass=mass, dt=0.01, damping=0.1)
    o = oracle_mod.Oracle.from_network(X, si, sj, k, r0, rc2, **kw)
    g = lsm.Specimen.from_network(X, si, sj, k, r0, rc2, precision="exact64", **kw)
    for s in (o, g):
        s.step(7)
        s.step(5)
    xo, vo, _ = o.state()
    if not (np.isfinite(xo).all() and np.isfinite(vo).all()):  # a length whose square underflows to 0
        with pytest.raises(lsm.LsmError) as err:
            g.state()
        assert err.value.status == lsm.LSM_ENONFINITE
        return
    xg, vg = g.state()
    assert np.array_equal(xg, xo) and np.array_equal(vg, vo)
    assert np.array_equal(g.broken()[0], o.broken()[0])
