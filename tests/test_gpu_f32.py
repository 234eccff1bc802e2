"""F32 steps on both sides of the tile height's line (456 tiles of 32 x 16) and
of the strips' (two thirds of the resident warps), and foams with their springs
two at a time."""
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


@pytest.mark.parametrize("nx,ny,a", [(672, 345, 1.0), (671, 335, 1.3), (700, 690, 1.0), (600, 610, 0.5)])
def test_tile_heights_and_strips_agree_bitwise(L, nx, ny, a):
    """The automatic choice, the tile kernel and the strip kernel give the same
    states and broken springs, affine and at a constant strain rate."""
    k, e, m = two_phase_materials()
    img = inclusion_image(nx, ny, 3.0, 12.0, 0.3, 5)
    img[ny // 3:ny // 3 + 5, 40:90] = 0
    outs = []
    for path in (0, 2, 3):
        g = L.Specimen.from_image(img, k, e, m, precision="f32", path=path, a=a)
        for i in range(1, 6):
            g.apply_strain(i * 8e-3)
            g.step(4)
        g.set_strain_rate(0.05)
        g.step(3)
        outs.append((*g.state(), g.broken(), g.break_steps()))
        g.close()
    assert outs[0][2][0].sum() > 0
    for o in outs[1:]:
        assert np.array_equal(outs[0][0], o[0]) and np.array_equal(outs[0][1], o[1])
        assert np.array_equal(outs[0][2][0], o[2][0]) and np.array_equal(outs[0][3], o[3])


@pytest.mark.parametrize("shape,rate", [((9, 17, 33), 0.0), ((8, 8, 16), 0.0), ((20, 24, 21), 0.2)])
def test_foam_pairs_agree_with_the_sample_step(L, shape, rate):
    """A 3D step without a sample (springs two at a time) against steps of one,
    which all sample (one spring at a time): the same forces up to the order of
    the error-compensated sums, 2^-44 of a force per step. Twelve steps of
    dt = 0.01 with unit masses leave 1e-12 of displacements near 0.01."""
    k, e, m = two_phase_materials()
    img = np.random.default_rng(shape[2]).integers(0, 3, size=shape).astype(np.uint8)
    outs = []
    for calls in ((12,), (1,) * 12):
        g = L.Specimen.from_image(img, k, e, m, precision="f32", dt=0.01)
        g.apply_strain(0.03)
        if rate:
            g.set_strain_rate(rate)
        for n in calls:
            g.step(n)
        outs.append((*g.state(), g.broken()[0]))
        g.close()
    assert np.array_equal(outs[0][2], outs[1][2])
    assert np.abs(outs[0][0] - outs[1][0]).max() <= 1e-10 and np.abs(outs[0][1] - outs[1][1]).max() <= 1e-10


@pytest.mark.parametrize("precision,count", [("df64", 11), ("f32", 11), ("f32", 6), ("df64", 6)])
def test_batch_strips_of_one_wave_agree_bitwise(L, precision, count):
    """Eleven specimens near 400 x 330 take strips of more than 16 rows, so that
    all run at once, six (F32) strips of 8: the states are those of the tiles."""
    from paper_2201_04565_gb300 import batch as B
    k, e, _ = two_phase_materials()
    imgs = [inclusion_image(400 + 7 * q, 330 - 3 * q, 3.0, 9.0, 0.3, q) for q in range(count)]
    imgs[1][100:140, 50:90] = 0
    outs = []
    for sched in (None, (-16, 0, 1), (8, 0, 1)):
        b = B.Batch(imgs, k, e, precision=precision)
        if sched:
            b.set_schedule(*sched)
        for i in range(1, 4):
            b.apply_strain(0.01 * i)
            b.step(6)
        outs.append([(*b.state(q), b.broken(q)[0]) for q in range(count)])
        b.close()
    for o in outs[1:]:
        for p, q in zip(outs[0], o):
            assert all(np.array_equal(a, c) for a, c in zip(p, q))


@pytest.mark.parametrize("eps", [-0.02, -0.15, -0.4])
def test_df64_foam_with_large_forces_agrees_with_the_sample_step(L, eps):
    """Double-float foams below, around and far above the split sums' exact
    range (compressed springs have no largest force): steps without a sample
    against steps of one, which all sample and sum with error terms. Both keep
    a force to about 2^-44; twelve steps of dt = 0.01 leave less than 1e-12."""
    k, e, m = two_phase_materials()
    img = np.random.default_rng(7).integers(0, 3, size=(12, 19, 35)).astype(np.uint8)
    outs = []
    for calls in ((12,), (1,) * 12):
        g = L.Specimen.from_image(img, k, e, m, precision="df64", dt=0.01)
        g.apply_strain(eps)
        for n in calls:
            g.step(n)
        outs.append((*g.state(), g.broken()[0]))
        g.close()
    assert np.array_equal(outs[0][2], outs[1][2])
    assert np.abs(outs[0][0] - outs[1][0]).max() <= 1e-11 and np.abs(outs[0][1] - outs[1][1]).max() <= 1e-10
