"""The multi-step tile kernel of small images (path 0) against the one-step
tile kernel (path 2)."""
import numpy as np
import pytest

from gen.images import inclusion_image, two_phase_materials

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2201_04565_gb300 import lsm
    lsm.load_library()
    return lsm


def _voided(nx, ny, seed):
    return np.random.default_rng(seed).integers(0, 3, size=(ny, nx)).astype(np.uint8)


# sizes on both sides of the rule's lines (16 x 4 tiles up to 161, 32 x 8 up to
# 304; in the exact mode 16 x 4 up to 76, 32 x 4 up to 152), ragged in both
# directions, narrower than a tile, one row high, with voids, clamped grips
CASES = [((64, 64), {}, None), ((100, 77), {"grip_mode": 1}, None), ((31, 9), {"a": 1.3}, None),
         ((40, 1), {}, None), ((257, 3), {}, None), ((2, 50), {}, None), ((70, 45), {}, 5),
         ((112, 92), {}, None), ((113, 92), {}, 7), ((64, 76), {}, None), ((65, 76), {}, None), ((608, 128), {}, None),
         ((250, 203), {"grip_mode": 1}, 9), ((609, 121), {}, None), ((128, 152), {}, None), ((129, 121), {}, None)]


@pytest.mark.parametrize("precision", ["df64", "f32", "exact64"])
@pytest.mark.parametrize("size,kw,voids", CASES)
def test_multi_step_kernel_agrees_with_one_step(L, precision, size, kw, voids):
    """Same positions, velocities, broken springs and break steps through
    fracture, affine increments and a constant strain rate, whatever the number
    of steps per call (a multiple of the kernel's steps per launch or not).
    Samples: the sums are grouped per tile of each kernel, so the double-float
    sums agree to 1e-10 and the FP64 ones to 1e-12; the kinetic terms of the
    fixed-point modes are float statistics (2^-24 a particle), the residual (a
    maximum) is equal."""
    nx, ny = size
    img = _voided(nx, ny, voids) if voids else inclusion_image(nx, ny, 2.0, 6.0, 0.3, nx)
    img[0, :2] = 1
    k, e, m = two_phase_materials()
    outs = []
    for path in (0, 2):
        g = L.Specimen.from_image(img, k, e, m, precision=precision, path=path, **kw)
        for i, n in enumerate((1, 2, 3, 4, 5, 7, 20, 6, 9, 13)):
            g.apply_strain(0.013 * (i + 1))
            g.step(n)
        g.set_strain_rate(0.2)
        for n in (3, 8):
            g.step(n)
        outs.append((g.state(), g.broken(), g.break_steps(), g.samples()))
        g.close()
    (sa, ba, ta, ma), (sb, bb, tb, mb) = outs
    assert np.array_equal(sa[0], sb[0]) and np.array_equal(sa[1], sb[1])
    assert np.array_equal(ba[0], bb[0]) and ba[1] == bb[1]
    assert np.array_equal(ta, tb)
    if nx > 60 and ny > 40:
        assert ba[0].sum() > 0, "the schedule must reach fracture"
    rel = 1e-12 if precision == "exact64" else 1e-10
    for p, q in zip(ma, mb):
        for key in ("eps", "n_broken", "step", "residual"):
            assert p[key] == q[key], key
        scale = max(abs(q["sigma_vir"]), 1e-3)  # sums of terms of both signs
        for key in ("sigma_vir", "sigma_grip"):
            assert abs(p[key] - q[key]) <= rel * scale, key
        assert p["pe"] == pytest.approx(q["pe"], rel=rel, abs=1e-300)
        assert p["ke"] == pytest.approx(q["ke"], rel=rel if precision == "exact64" else 1e-6, abs=1e-300)
