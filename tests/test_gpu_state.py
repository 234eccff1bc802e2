"""State readback: particles packed on the device against the grid positions
known on the host, over the block and staging limits of the packing kernel."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lsm():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2201_04565_gb300 import build
    build.build()
    from paper_2201_04565_gb300 import lsm
    return lsm


def _image(shape, holes):
    img = np.ones(shape, np.uint8)
    rng = np.random.default_rng(shape[-1])
    if holes == "one":
        img.reshape(-1)[img.size // 2] = 0
    elif holes == "ends":  # whole blocks without a particle at both ends and inside
        f = img.reshape(-1)
        f[:1500] = 0
        f[-1100:] = 0
        f[f.size // 2:f.size // 2 + 2100] = 0
    elif holes == "noise":
        img[rng.random(shape) < 0.4] = 0
    return img


@pytest.mark.parametrize("shape,holes,precision,lattice", [
    ((32, 32), "one", "exact64", 0), ((33, 31), "none", "f32", 0), ((96, 64), "ends", "df64", 0),
    ((41, 103), "noise", "exact64", 0), ((40, 57), "none", "df64", 1), ((64, 300), "noise", "f32", 1),
    ((11, 40, 37), "noise", "df64", 0), ((8, 16, 16), "none", "f32", 0), ((2300, 2600), "noise", "f32", 0),
    ((2300, 2600), "one", "f32", 0)])
def test_state_round_trip(lsm, shape, holes, precision, lattice):
    """What set_state puts on the grid comes back bit for bit, position and
    velocity alone and together; the last two images hold less and more
    particles than the staging (4,194,304)."""
    img = _image(shape, holes)
    g = lsm.Specimen.from_image(img, np.full((1, 1), 10.0), np.full((1, 1), 0.1), precision=precision,
                                lattice=lattice, dt=0.01, damping=0.1)
    x, v = g.state()
    assert not v.any() and np.unique(x.T, axis=0).shape[0] == x.shape[1]  # distinct lattice positions
    if not lattice:
        pos = np.nonzero(img.reshape(-1))[0]
        assert np.array_equal(x[0], (pos % shape[-1]).astype(float))
    rng = np.random.default_rng(5)
    x2, v2 = x + np.round(rng.uniform(-0.01, 0.01, x.shape) * 2 ** 20) / 2 ** 20, rng.uniform(-1e-3, 1e-3, x.shape)
    g.set_state(x2, v2)
    a, b = g.state()
    assert np.array_equal(a, x2) and np.array_equal(b, v2)
    out = np.empty_like(x)
    lsm._check(lsm.load_library().lsm_get_state(g.h, None, lsm._ptr(out)), g.h)
    assert np.array_equal(out, v2)
    g.close()
