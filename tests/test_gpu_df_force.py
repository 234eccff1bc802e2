"""The force of the double-float mode on a soft phase beside a much stiffer one, or
with a large critical strain, against extended precision."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

DT = 2.0 ** -25  # so short that positions near 8 do not move: v / (n dt) is the force of the set state


@pytest.fixture(scope="module")
def L():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2201_04565_gb300 import lsm
    lsm.load_library()
    return lsm


def _tables(contrast, ec_soft):
    c = 1.0 / contrast
    k = np.array([[1.0, 2.0 * c / (1.0 + c)], [2.0 * c / (1.0 + c), c]])
    return k, np.array([[0.05, 0.05], [0.05, ec_soft]])


def _image(shape):
    img = np.full(shape, 2, np.uint8)
    img[..., : shape[-1] // 3] = 1
    return img


def _positions(X, strain, rng):
    """A smooth strain and some noise on multiples of 2^-34, which every fixed-point
    scale of these specimens holds exactly."""
    d = strain * rng.uniform(-1, 1, (X.shape[0], X.shape[0])) @ X / 8 + 0.3 * strain * rng.uniform(-1, 1, X.shape)
    return np.round((X + 8.0 + d) * 2.0 ** 34) / 2.0 ** 34


def _error(topo, x, v, steps, k_soft, n):
    """Force error in units of k_soft at the particles all of whose springs are soft."""
    si, sj = topo["si"], topo["sj"]
    xl = x.astype(np.longdouble)
    d = xl[:, sj] - xl[:, si]
    r = np.sqrt((d * d).sum(0))
    f = topo["k"].astype(np.longdouble) * (1 - topo["r0"].astype(np.longdouble) / r) * d
    F = np.zeros((x.shape[0], n), np.longdouble)
    stiff = np.zeros(n, bool)
    for c in range(x.shape[0]):
        np.add.at(F[c], si, f[c])
        np.add.at(F[c], sj, -f[c])
    for end in (si, sj):
        stiff[end[topo["k"] != k_soft]] = True
    soft = ~stiff & (np.bincount(si, minlength=n) + np.bincount(sj, minlength=n) > 2)
    soft &= (v != 0).all(0)  # not a grip
    assert soft.sum() > 100
    e = ((v.astype(np.longdouble) / (steps * np.longdouble(DT)) - F) / k_soft).astype(float)[:, soft]
    return np.sqrt((e * e).mean()), np.abs(e).max()


# Eight springs (18 in 3D): the root mean square of the sum's error is 2.8e-14 k r0
# (3.7e-14) with the force's low parts at full length and 1 - r0/r to its first
# correction, the largest of some 1e5 sums 2.2e-13
RMS, MAX = 5e-14, 4e-13


@pytest.mark.parametrize("contrast,ec,strain", [(10.0, 0.3, 1e-2), (1e3, 0.3, 1e-2), (1e6, 0.3, 1e-3), (2.0, 10.0, 1e-2),
                                                (1.0, 1000.0, 1e-2)])
@pytest.mark.parametrize("shape,kw", [((48, 60), dict(path=0)), ((48, 60), dict(path=2)), ((48, 60), dict(path=3)),
                                      ((300, 310), dict(path=0)), ((48, 60), dict(lattice=1)), ((14, 18, 30), {})])
@pytest.mark.parametrize("steps", [1, 2])
def test_soft_phase_keeps_its_accuracy(L, shape, kw, contrast, ec, strain, steps):
    """Multi-step and one-step tiles, strips, the packing and 3D voxels, with (the
    last step of a call) and without a sample."""
    k, e = _tables(contrast, ec)
    g = L.Specimen.from_image(_image(shape), k, e, precision="df64", dt=DT, damping=0.0, **kw)
    X = g.state()[0]
    x = _positions(X, strain, np.random.default_rng(len(shape)))
    g.set_state(x, np.zeros_like(x))
    g.step(steps)
    x1, v = g.state()
    rms, most = _error(g.topology(), x, v, steps, k[1, 1], g.n)
    free = v[0] != 0
    g.close()
    assert np.array_equal(x1[:, free], x[:, free])
    assert rms <= RMS and most <= MAX


@pytest.mark.parametrize("sched", [(8, 0, 1), (16, 0, 1), (32, 0, 1), (-16, 0, 1)])
@pytest.mark.parametrize("steps", [1, 2])
def test_soft_phase_of_a_batch(L, sched, steps):
    from paper_2201_04565_gb300 import batch as B
    k, e = _tables(1e4, 0.3)
    shapes = [(48, 60), (70, 33)]
    b = B.Batch([_image(s) for s in shapes], k, e, precision="df64", dt=DT, damping=0.0)
    b.set_schedule(*sched)
    xs, topo = [], []
    for q, s in enumerate(shapes):
        x = _positions(b.state(q)[0], 1e-2, np.random.default_rng(q))
        b.set_state(q, x, np.zeros_like(x))
        g = L.Specimen.from_image(_image(s), k, e, precision="exact64")
        topo.append(g.topology())
        g.close()
        xs.append(x)
    b.step(steps)
    for q in range(len(shapes)):
        rms, most = _error(topo[q], xs[q], b.state(q)[1], steps, k[1, 1], xs[q].shape[1])
        assert rms <= RMS and most <= MAX
    b.close()


@pytest.mark.parametrize("kw,stretch", [(dict(path=0), 2.03), (dict(path=3), 2.03), (dict(lattice=1), 3.5), ("batch", 2.03)])
def test_forces_of_springs_beyond_their_critical_length(L, kw, stretch):
    """A soft sheet folded over and stretched beyond its critical strain by set_state:
    the springs hold until the next step tests them, so the initial acceleration has
    six springs of a particle on the fold pulling one way, more together than any
    intact ones. All break in the step: v is dt / 2 times the force before it."""
    k, e = _tables(10.0, 0.3)
    img = np.full((30, 41), 2, np.uint8)
    img[0, 0] = 1
    g = L.Specimen.from_image(img, k, e, precision="exact64", **({} if kw == "batch" else dict(lattice=kw.get("lattice", 0))))
    topo, X = g.topology(), g.state()[0]
    g.close()
    fold = 20.25 if "lattice" in kw else 20.0  # no two sites of a row onto one point
    x = stretch * np.stack([np.abs(X[0] - fold), X[1]])
    x += np.random.default_rng(3).uniform(-5e-3, 5e-3, x.shape)
    x = np.round((x + 8.0) * 2.0 ** 34) / 2.0 ** 34
    if kw == "batch":
        from paper_2201_04565_gb300 import batch as B
        s = B.Batch([img], k, e, precision="df64", dt=DT, damping=0.0)
        s.set_state(0, x, np.zeros_like(x))
        s.step(1)
        v, broken = s.state(0)[1], s.broken(0)[0]
    else:
        s = L.Specimen.from_image(img, k, e, precision="df64", dt=DT, damping=0.0, **kw)
        s.set_state(x, np.zeros_like(x))
        s.step(1)
        v, broken = s.state()[1], s.broken()[0]
    s.close()
    assert broken.all()
    rms, most = _error(topo, x, 2.0 * v, 1, k[1, 1], x.shape[1])
    assert rms <= 10 * RMS and most <= 10 * MAX  # the forces are ten times those of small strains
