"""3D time steps give the same bits however they are grouped into calls: the last
step of a call takes one spring at a time and samples, the others two."""
import numpy as np
import pytest

from gen.images import two_phase_materials

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2201_04565_gb300 import lsm
    lsm.load_library()
    return lsm


@pytest.mark.parametrize("precision", ["df64", "f32"])
@pytest.mark.parametrize("shape,eps,rate,kw", [((9, 17, 33), 0.03, 0.0, {}), ((8, 8, 16), 0.06, 0.0, dict(a=1.3)),
                                               ((20, 24, 21), 0.02, 0.3, dict(k2_ratio=0.5)),
                                               ((12, 19, 35), -0.02, 0.0, dict(grip_mode=1)), ((12, 19, 35), -0.15, 0.0, {}),
                                               ((12, 19, 35), -0.4, 0.0, dict(a=0.01)), ((1, 2, 40), 0.02, -0.2, {})])
def test_calls_of_any_length_give_the_same_bits(L, precision, shape, eps, rate, kw):
    k, e, m = two_phase_materials()
    img = np.random.default_rng(shape[2]).integers(0, 3, size=shape).astype(np.uint8)
    outs = []
    for calls in ((12,), (1,) * 12, (5, 7)):
        g = L.Specimen.from_image(img, k, e, m, precision=precision, dt=0.01, **kw)
        g.apply_strain(eps)
        if rate:
            g.set_strain_rate(rate)
        for n in calls:
            g.step(n)
        outs.append((*g.state(), *g.broken(), g.break_steps()))
        g.close()
    for o in outs[1:]:
        assert all(np.array_equal(a, b) for a, b in zip(outs[0], o))
