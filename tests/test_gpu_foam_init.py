"""The initial acceleration of a 3D state with springs beyond their critical length:
the force that set_state's velocities start from has no break test, on the voxel
kernel as on the spring lists."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,bound", [("df64", 1e-11), ("f32", 1e-5)])
@pytest.mark.parametrize("stretch,ec", [(1.2, 0.05), (1.0, -0.02), (1.05, 0.05)])
def test_first_velocities_agree_with_the_exact_mode(precision, bound, stretch, ec):
    """One step of dt from rest: v = dt / 2 (a before + a after the breaks). Against
    the exact mode, relative to the largest; f32 forces are single precision."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2201_04565_gb300 import lsm
    img = np.random.default_rng(2).integers(0, 3, size=(11, 18, 23)).astype(np.uint8)
    k = np.array([[1.0, 0.3], [0.3, 0.2]])
    outs = []
    for p in ("exact64", precision):
        g = lsm.Specimen.from_image(img, k, np.full((2, 2), ec), precision=p, dt=0.01)
        X = g.state()[0]
        x = np.round((stretch * X + np.random.default_rng(3).uniform(-0.02, 0.02, X.shape)) * 2.0 ** 30) / 2.0 ** 30
        g.set_state(x, np.zeros_like(x))
        g.step(1)
        outs.append((*g.state(), g.broken()[0]))
        g.close()
    assert np.array_equal(outs[0][2], outs[1][2]) and outs[0][2].any()
    top = np.abs(outs[0][1]).max()
    assert top > 1e-5
    assert np.abs(outs[1][1] - outs[0][1]).max() <= bound * top
