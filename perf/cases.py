"""Performance cases: the work a user of the library gives it, through its public calls.

listed() gives the cases, draw(rng) more of the same ranges, prepare(case, seed)
a program's inputs and handles, run(state) one pass, work(case) the bytes and
operations of a pass that no implementation can do without, and exact(case,
seed) the outputs of the first pass in plain 64-bit torch, without the library.

Every stepping pass is what the examples and the benchmark do: load increments
of a number of time steps each, then the read of the results (latest sample,
broken springs, positions and velocities). Passes on the same state load
upwards and unload again in turn, so that any number of them stays in the
range of strains that the first one covers.
"""
import math

import numpy as np
import torch

from paper_2201_04565_gb300 import batch as lsm_batch
from paper_2201_04565_gb300 import lsm, nn

# The stiff matrix and soft inclusions of every two-phase workload: spring
# constants (interface: the two half springs in series) and critical strains.
K_TWO = np.array([[1.0, 2.0 * 0.1 / 1.1], [2.0 * 0.1 / 1.1, 0.1]])
E_TWO = np.array([[0.05, 0.175], [0.175, 0.3]])
K_ONE, E_ONE = np.array([[1.0]]), np.array([[0.04]])
# The paper's spring table (stiff-stiff, stiff-soft, soft-soft; r0 = 10).
K_PAPER = np.array([[2.00e-3, 1.25e-4], [1.25e-4, 2.00e-5]])
RC_PAPER = np.array([[10.1, 10.4], [10.4, 11.0]])

# (Cin, Cout) of the network's fourteen 3 x 3 convolutions.
CONVS = [(32, 32), (32, 32), (32, 64), (64, 64), (64, 128), (128, 128), (128, 256),
         (256, 256), (384, 128), (128, 128), (192, 64), (64, 64), (96, 32), (32, 32)]
LEVEL = [0, 0, 1, 1, 2, 2, 3, 3, 2, 2, 1, 1, 0, 0]


def listed():
    return [
        # one load increment of the 64 x 64 specimen at the binding's default
        # precision: the smallest call, bound by launches and latency
        dict(name="increment_64", kind="image", nx=64, ny=64, nz=1, precision="exact64", lattice=0, rate=False,
             increments=1, steps=20, eps0=0.03, eps1=0.0311, fields=False),
        # a whole tension curve of a small specimen in the benchmark's
        # precision: 2,000 short time steps, one after another
        dict(name="curve_100_df64", kind="image", nx=100, ny=90, nz=1, precision="df64", lattice=0, rate=False,
             increments=100, steps=20, eps0=0.0, eps1=0.0437, fields=False),
        # a ragged composite at the default precision, with the per-particle
        # stress and strain maps that post-processing asks for
        dict(name="composite_1000_exact64", kind="image", nx=1000, ny=700, nz=1, precision="exact64", lattice=0,
             rate=False, increments=15, steps=20, eps0=0.0, eps1=0.0431, fields=True),
        # the benchmark's composite towards its first fracture
        dict(name="composite_2048_df64", kind="image", nx=2048, ny=2048, nz=1, precision="df64", lattice=0,
             rate=False, increments=40, steps=20, eps0=0.0, eps1=0.0437, fields=False),
        # the single-precision force variant on an odd-sized image
        dict(name="composite_1537_f32", kind="image", nx=1537, ny=1111, nz=1, precision="f32", lattice=0, rate=False,
             increments=40, steps=20, eps0=0.0, eps1=0.0423, fields=False),
        # the paper's own lattice and loading: triangular packing, a strained
        # specimen whose grips move on at a constant strain rate
        dict(name="triangular_1200_df64", kind="image", nx=1200, ny=900, nz=1, precision="df64", lattice=1,
             rate=True, increments=20, steps=20, eps0=0.03, eps1=0.03011, fields=False),
        # 3D voxel foam under compression, the largest volume in use
        dict(name="foam_256_df64", kind="image", nx=256, ny=256, nz=256, precision="df64", lattice=0, rate=False,
             increments=15, steps=20, eps0=0.0, eps1=-0.0313, fields=False),
        # a small foam at the default precision (general spring lists)
        dict(name="foam_90_exact64", kind="image", nx=90, ny=81, nz=77, precision="exact64", lattice=0, rate=False,
             increments=10, steps=20, eps0=0.0, eps1=-0.0213, fields=False),
        # an explicit particle and spring list of the paper's size, as read
        # from a LAMMPS data file
        dict(name="network_47k", kind="network", nx=217, ny=216, precision="exact64", increments=20, steps=20,
             eps1=0.0083),
        # uneven specimens (sides 32 to 512) stepped together
        dict(name="batch_20", kind="batch", count=20, side0=32, side1=512, precision="df64", increments=20, steps=20,
             eps1=0.0437),
        # quasi-static increments of equal specimens to a force residual and
        # their displacement fields, as the warm start's training data are made
        dict(name="relax_12x128", kind="relax", count=12, side=128, precision="df64", check=50, tol=2e-5,
             increments=2, deps=1e-3),
        # the warm-start network: a prediction and the gradients of a
        # training step
        dict(name="unet_256_b8", kind="unet", side=256, batch=8),
    ]


def _log(rng, a, b):
    return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))


def _rate_end(rng, eps0, increments, nx):
    """A strain reached at a rate whose grips move far slower than sound (1 per unit time)."""
    return round(eps0 + rng.uniform(0.001, 0.02) * increments * 0.2 / (0.5 * nx), 9)


def draw(rng):
    kind = rng.choice(["image2", "image2", "image2", "tri", "foam", "foam", "network", "batch", "relax", "unet"])
    if kind == "image2":
        nx, ny = _log(rng, 48, 2048), _log(rng, 48, 2048)
        precision = rng.choice(["exact64", "fast64", "f32", "df64"])
        inc = max(1, min(60, int(6e7 / (nx * ny)) if precision in ("f32", "df64") else int(9e6 / (nx * ny))))
        inc, rate, fields = rng.randint(1, inc), rng.random() < 0.25, rng.random() < 0.25
        eps0 = 0.03 if rate else 0.0
        eps1 = _rate_end(rng, eps0, inc, nx) if rate else round(rng.uniform(0.0033, 0.0453), 6)
        return dict(kind="image", nx=nx, ny=ny, nz=1, precision=precision, lattice=0, rate=rate, increments=inc,
                    steps=20, eps0=eps0, eps1=eps1, fields=fields)
    if kind == "tri":
        nx, ny = _log(rng, 48, 1200), _log(rng, 48, 1200)
        inc = rng.randint(1, max(1, min(40, int(2e7 / (nx * ny)))))
        return dict(kind="image", nx=nx, ny=ny, nz=1, precision=rng.choice(["df64", "f32"]), lattice=1, rate=True,
                    increments=inc, steps=20, eps0=0.03, eps1=_rate_end(rng, 0.03, inc, nx), fields=False)
    if kind == "foam":
        precision = rng.choice(["df64", "f32", "exact64", "fast64"])
        top = 200 if precision in ("df64", "f32") else 96
        nx, ny, nz = (_log(rng, 24, top) for _ in range(3))
        return dict(kind="image", nx=nx, ny=ny, nz=nz, precision=precision, lattice=0, rate=False,
                    increments=rng.randint(1, 10), steps=20, eps0=0.0, eps1=-round(rng.uniform(0.0033, 0.0313), 6),
                    fields=False)
    if kind == "network":
        return dict(kind="network", nx=_log(rng, 60, 300), ny=_log(rng, 60, 300),
                    precision=rng.choice(["exact64", "fast64"]), increments=rng.randint(2, 20), steps=20,
                    eps1=round(rng.uniform(0.0023, 0.0087), 6))
    if kind == "batch":
        side0 = rng.randint(32, 128)
        return dict(kind="batch", count=rng.randint(3, 20), side0=side0, side1=rng.randint(side0, 512),
                    precision=rng.choice(["df64", "f32", "exact64"]), increments=rng.randint(1, 10), steps=20,
                    eps1=round(rng.uniform(0.0033, 0.0453), 6))
    if kind == "relax":
        return dict(kind="relax", count=rng.randint(2, 12), side=_log(rng, 48, 128), precision="df64", check=50,
                    tol=2e-5, increments=rng.randint(1, 2), deps=round(rng.uniform(5e-4, 1e-3), 6))
    return dict(kind="unet", side=8 * rng.randint(4, 32), batch=rng.randint(1, 8))


# ------------------------------------------------------------------ inputs

def _disks(nx, ny, r0, r1, frac, rng):
    """Stiff matrix (1) with overlapping soft disks (2) up to an area fraction."""
    img = np.ones((ny, nx), np.uint8)
    soft, target = 0, frac * nx * ny
    while soft < target:
        cx, cy, r = rng.uniform(0, nx), rng.uniform(0, ny), rng.uniform(r0, r1)
        x0, x1 = max(0, int(cx - r - 1)), min(nx, int(cx + r + 2))
        y0, y1 = max(0, int(cy - r - 1)), min(ny, int(cy + r + 2))
        px, py = np.arange(x0, x1) + 0.5 - cx, np.arange(y0, y1) + 0.5 - cy
        sub = img[y0:y1, x0:x1]
        new = (py[:, None] ** 2 + px[None, :] ** 2 <= r * r) & (sub == 1)
        sub[new] = 2
        soft += int(np.count_nonzero(new))
    return img


def _composite(nx, ny, rng):
    big = min(nx, ny) >= 512
    return _disks(nx, ny, 10.0 if big else 3.0, 60.0 if big else 8.0, 0.30, rng)


def _foam(nx, ny, nz, seed):
    """Smoothed noise (Gaussian, periodic), its top 35% solid (1), the rest void (0)."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    f = torch.randn((nz, ny, nx), device="cuda", dtype=torch.float64, generator=gen)
    sigma = 4.0 if max(nx, ny, nz) >= 128 else 2.0
    h = torch.fft.rfftn(f)
    for d, n in enumerate((nz, ny, nx)):
        q = torch.fft.rfftfreq(n, device="cuda") if d == 2 else torch.fft.fftfreq(n, device="cuda")
        g = torch.exp(-2.0 * (math.pi * sigma * q.double()) ** 2)
        h = h * g.reshape([-1 if e == d else 1 for e in range(3)])
    f = torch.fft.irfftn(h, s=(nz, ny, nx))
    k = int(0.65 * f.numel())
    cut = f.flatten().sort().values[k]
    return (f > cut).to(torch.uint8).cpu().numpy()


def _image(case, seed):
    if case["nz"] > 1:
        return _foam(case["nx"], case["ny"], case["nz"], seed), K_ONE, E_ONE
    rng = np.random.default_rng([11, seed])
    return _composite(case["nx"], case["ny"], rng), K_TWO, E_TWO


def _network(case, seed):
    """The paper's Poisson composites: a triangular particle lattice of spacing
    10 with soft disks, springs to the six first neighbours, the first and last
    particle of each row held in x."""
    nx, ny, a = case["nx"], case["ny"], 10.0
    h = a * math.sqrt(3.0) * 0.5
    ph = _disks(nx, ny, 3.0, 8.0, 0.30, np.random.default_rng([13, seed]))
    iy, ix = np.mgrid[0:ny, 0:nx]
    X = np.stack([((ix + 0.5 * (iy & 1)) * a).ravel(), (iy * h).ravel()])
    pid = np.arange(nx * ny).reshape(ny, nx)
    ends = [(pid[:, :-1], pid[:, 1:])]
    for par in (0, 1):  # the next row's particles at x - a/2 and x + a/2
        lo, up = pid[par:-1:2], pid[par + 1::2]
        lo = lo[:up.shape[0]]
        ends += [(lo[:, 1:], up[:, :-1]), (lo, up)] if par == 0 else [(lo, up), (lo[:, :-1], up[:, 1:])]
    si = np.concatenate([e[0].ravel() for e in ends])
    sj = np.concatenate([e[1].ravel() for e in ends])
    order = np.lexsort((sj, si))
    si, sj = si[order].astype(np.int32), sj[order].astype(np.int32)
    p = ph.ravel().astype(np.int64) - 1
    fix = np.zeros((2, nx * ny), np.uint8)
    grip = np.zeros(nx * ny, np.uint8)
    for col, code in ((0, 1), (nx - 1, 2)):
        fix[0, pid[:, col]] = 1
        grip[pid[:, col]] = code
    return dict(X=X, si=si, sj=sj, k=K_PAPER[p[si], p[sj]], r0=np.full(si.size, a), rc2=RC_PAPER[p[si], p[sj]] ** 2,
                fix=fix, grip=grip, xc=0.5 * (nx - 0.5) * a, omega=(nx - 1) * a * ny * h, grip_area=ny * h)


def _sides(case):
    """Sides of a batch's square specimens: of the case alone (whatever the seed)."""
    if case["kind"] == "relax":
        return [case["side"]] * case["count"]
    rng = np.random.default_rng([case["count"], case["side0"], case["side1"]])
    return [int(s) for s in rng.integers(case["side0"], case["side1"] + 1, case["count"])]


def _batch_images(case, seed):
    rng = np.random.default_rng([17, seed])
    return [_disks(s, s, 3.0, 8.0, float(rng.uniform(0.10, 0.50)), rng) for s in _sides(case)]


def _unet_inputs(case, seed):
    """Phase map, displacement and strain channels of the range that the
    network's inputs have, targets of a unit-sized field, He-sized weights."""
    s, b = case["side"], case["batch"]
    gen = torch.Generator().manual_seed(seed)
    x = torch.zeros((b, s, s, 32))
    soft = torch.nn.functional.avg_pool2d(torch.randn((b, 1, s, s), generator=gen), 5, 1, 2)[:, 0] > 0.1
    x[..., 0] = soft.float() - 0.5
    for c in (1, 2):
        x[..., c] = 0.3 * torch.nn.functional.avg_pool2d(torch.randn((b, 1, s, s), generator=gen), 7, 1, 3)[:, 0]
    x[..., 3] = 1.0
    x[..., 4] = torch.rand((b, 1, 1), generator=gen)
    pos = (torch.arange(s) - 0.5 * (s - 1)) / (0.5 * s)
    x[..., 5], x[..., 6] = pos[None, None, :], pos[None, :, None]
    target = 0.3 * torch.nn.functional.avg_pool2d(torch.randn((b, 2, s, s), generator=gen), 9, 1, 4)
    parts = []
    for cin, cout in CONVS:
        parts += [torch.randn(cout * 9 * cin, generator=gen) * math.sqrt(2.0 / (9 * cin)),
                  0.01 * torch.randn(cout, generator=gen)]
    parts += [0.1 * torch.randn(64, generator=gen), torch.zeros(2)]
    return (x.to(torch.bfloat16).cuda(), target.permute(0, 2, 3, 1).contiguous().cuda(), torch.cat(parts).numpy())


# ------------------------------------------------------------------ the pass

def prepare(case, seed):
    s = dict(case=case, up=True)
    if case["kind"] == "image":
        img, k, e = _image(case, seed)
        s["g"] = lsm.Specimen.from_image(img, k, e, precision=case["precision"], lattice=case["lattice"],
                                         grip_mode=1 if case["nz"] > 1 else 0, dt=0.01, damping=0.1)
        if case["eps0"]:
            s["g"].apply_strain(case["eps0"])
        s["mask"] = _mask_buffer(s["g"].n * (9 if case["nz"] > 1 else 4 - case["lattice"]))
    elif case["kind"] == "network":
        net = _network(case, seed)
        s["mask"] = _mask_buffer(net["si"].size)
        s["g"] = lsm.Specimen.from_network(net.pop("X"), net.pop("si"), net.pop("sj"), net.pop("k"), net.pop("r0"),
                                           net.pop("rc2"), dt=0.1, damping=0.02, precision=case["precision"], **net)
    elif case["kind"] == "batch":
        s["b"] = lsm_batch.Batch(_batch_images(case, seed), K_TWO, E_TWO, dt=0.01, damping=0.1,
                                 precision=case["precision"])
    elif case["kind"] == "relax":
        s["b"] = lsm_batch.Batch(_batch_images(case, seed), K_TWO, E_TWO, dt=0.5, damping=0.03,
                                 precision=case["precision"])
        s["u"] = torch.empty((case["increments"], case["count"], 2, case["side"], case["side"]), device="cuda")
        torch.cuda.current_stream().synchronize()
    else:
        x, target, params = _unet_inputs(case, seed)
        net = nn.UNet(case["side"], case["side"], case["batch"])
        net.set_params(params)
        s.update(net=net, x=x, target=target, pred=torch.empty_like(target))
    return s


def _levels(case, up):
    """The strains of a pass's increments: up from eps0 to eps1, or back."""
    n, e0, e1 = case["increments"], case.get("eps0", 0.0), case["eps1"]
    q = range(1, n + 1) if up else range(n - 1, -1, -1)
    return [e0 + (e1 - e0) * i / n for i in q]


def _mask_buffer(springs):
    """Page-locked room for the broken flags, reused by every read (an image's
    network has at most a fixed number of springs per particle)."""
    return torch.zeros(springs, dtype=torch.uint8).pin_memory().numpy()


def _read(g, buffer):
    _, first = g.broken(buffer)
    x, v = g.state()
    return dict(sample=g.last_sample(), broken=buffer, first_break=first, x=x, v=v)


def run(s):
    case, kind = s["case"], s["case"]["kind"]
    up = s["up"]
    s["up"] = not up
    if kind == "unet":
        s["net"].forward(s["x"], s["pred"], case["batch"])
        loss, grad = s["net"].gradients(s["x"], s["target"], case["batch"])
        return dict(pred=s["pred"], loss=loss, grad=grad)
    if kind == "relax":
        b, u, out = s["b"], s["u"], {}
        for i in range(case["increments"]):
            b.apply_strain(case["deps"] * ((i + 1) if up else (case["increments"] - 1 - i)))
            _, taken, conv = b.relax(case["tol"], 20000, case["check"])
            nn.check(nn.lib().lsm_batch_fields(b.h, nn.ptr(u[i]), None, case["side"], case["side"]), b.h, batch=True)
            out["taken%d" % i], out["converged%d" % i] = taken, conv
        b.synchronize()
        out["u"] = u
        return out
    if kind == "batch":
        b = s["b"]
        for eps in _levels(case, up):
            b.apply_strain(eps)
            b.step(case["steps"])
        return dict(states=[b.state(q) for q in range(b.count)], broken=[b.broken(q)[0] for q in range(b.count)])
    g = s["g"]
    if case.get("rate"):
        r = (case["eps1"] - case["eps0"]) / (case["increments"] * case["steps"] * 0.01)
        g.set_strain_rate(r if up else -r)
        for _ in range(case["increments"]):
            g.step(case["steps"])
    else:
        for eps in _levels(case, up):
            g.apply_strain(eps)
            g.step(case["steps"])
    out = _read(g, s["mask"])
    if case.get("fields"):
        out["stress"], out["strain"] = g.fields()
    return out


# ------------------------------------------------------------------ bytes and operations

def work(case):
    """The state of every particle (position and half-step velocity, read and
    written, with two bytes of phase and broken flags on image lattices, or
    the spring records of a network: endpoints, type, state), once per time
    step where it is larger than the 129 MB L2 and once per pass where it can
    stay there; operations of Eqs. 2-5 per spring and particle and time step;
    the results that a pass returns, once. Relaxations count one check
    interval (how many they need is found by running them)."""
    kind = case["kind"]
    if kind == "unet":
        b, s = case["batch"], case["side"]
        conv = [2.0 * b * (s >> l) ** 2 * cin * cout * 9 for (cin, cout), l in zip(CONVS, LEVEL)]
        params = sum(cin * cout * 9 + cout for cin, cout in CONVS) + 66
        return dict(bytes=b * s * s * (64.0 + 16.0) + 8.0 * params, flops=5.0 * sum(conv) - conv[0])
    d, m_per = (3, 9.0) if case.get("nz", 1) > 1 else (2, 4.0)
    if kind in ("batch", "relax"):
        mean = (lambda a, b: (b ** 3 - a ** 3) / (3.0 * (b - a)) if b > a else a * a)
        n = case["count"] * (mean(case["side0"], case["side1"]) if kind == "batch" else case["side"] ** 2)
        steps = case["increments"] * (case["steps"] if kind == "batch" else case["check"])
    else:
        n = float(case["nx"]) * case["ny"] * case.get("nz", 1) * (0.35 if d == 3 else 1.0)
        steps = case["increments"] * case["steps"]
        if case.get("lattice"):
            n, m_per = n * 2.0 / math.sqrt(3.0), 3.0
    m = n * m_per * (0.9 if d == 3 else 1.0)
    if kind == "network":
        m_per, m = 3.0, 3.0 * n
    per_step = n * (32.0 * d + 2.0) if kind != "network" else n * 32.0 * d + 11.0 * m
    flops = steps * (m * (3.0 * d + 2 * d + 5) + n * 8.0 * d)
    out = n * 16.0 * d + m + (n * 8.0 * 6 if case.get("fields") else 0.0)
    return dict(bytes=(steps if n * 16.0 * d > 129e6 else 1) * per_step + out, flops=flops)


# ------------------------------------------------------------------ the same in plain 64 bits

def _pairs(img, tri):
    """Springs of an image: (positions [d, n], phase - 1 [n], si, sj, rest
    lengths), canonical order, all on the GPU."""
    if tri:
        ny, nx = img.shape
        rows, c = 0, math.sqrt(3.0) * 0.5
        while 3 * rows * rows <= 4 * (ny - 1) ** 2:
            rows += 1
        grid = np.zeros((rows, nx), np.uint8)
        for iy in range(rows):
            prow = (math.isqrt(3 * iy * iy) + 1) // 2
            grid[iy, :nx - (iy & 1)] = img[prow, (iy & 1):]
        ph = torch.from_numpy(grid).cuda()
        iy, ix = torch.meshgrid(torch.arange(rows, device="cuda"), torch.arange(nx, device="cuda"), indexing="ij")
        X = torch.stack([ix + 0.5 * (iy % 2), iy.double() * c]).double()
    else:
        ph = torch.from_numpy(img).cuda()
        axes = torch.meshgrid(*[torch.arange(q, device="cuda", dtype=torch.float64) for q in img.shape], indexing="ij")
        X = torch.stack(list(axes)[::-1])
    here = ph > 0
    pid = torch.where(here, torch.cumsum(here.flatten().long(), 0).reshape(ph.shape) - 1, -1)
    found = []

    def join(lo, hi, r0):
        i, j = pid[lo].flatten(), pid[hi].flatten()
        ok = (i >= 0) & (j >= 0)
        found.append((i[ok], j[ok], r0))

    cut = lambda o, n: (slice(max(0, -o), n - max(0, o)), slice(max(0, o), n - max(0, -o)))  # noqa: E731
    if tri:
        join((slice(None), slice(0, -1)), (slice(None), slice(1, None)), 1.0)
        for par in (0, 1):
            lo, hi = slice(par, rows - 1, 2), slice(par + 1, rows, 2)
            for o in ((-1, 0) if par == 0 else (0, 1)):
                a, b = cut(o, nx)
                join((lo, a), (hi, b), 1.0)
    else:
        d = img.ndim
        for off in np.ndindex(*(3,) * d):
            o = [q - 1 for q in off]  # z, y, x
            l2 = sum(q * q for q in o)
            if l2 in (1, 2) and next(q for q in o if q) > 0:
                sl = [cut(q, n) for q, n in zip(o, img.shape)]
                join(tuple(a for a, _ in sl), tuple(b for _, b in sl), math.sqrt(2.0) if l2 == 2 else 1.0)
    si, sj = torch.cat([f[0] for f in found]), torch.cat([f[1] for f in found])
    r0 = torch.cat([torch.full((f[0].numel(),), f[2], dtype=torch.float64, device="cuda") for f in found])
    order = torch.argsort(si * int(here.sum()) + sj)
    return X[:, here], ph[here].long() - 1, si[order], sj[order], r0[order]


class _Plain:
    """Eqs. 2-5 and 7 on a spring list, in torch float64."""

    def __init__(self, X, si, sj, k, r0, rc2, fix, right, xc, omega, area, dt, damping):
        self.X, self.x, self.v, self.a = X, X.clone(), torch.zeros_like(X), torch.zeros_like(X)
        self.si, self.sj, self.k, self.r0, self.rc2 = si, sj, k, r0, rc2
        self.intact = torch.ones_like(k)
        self.fix, self.right, self.xc, self.omega, self.area = fix, right, xc, omega, area
        self.free = (~fix).double()
        self.dt, self.damping, self.eps = dt, damping, 0.0

    @classmethod
    def image(cls, img, ktab, etab, tri, clamp, dt, damping):
        X, ph, si, sj, r0 = _pairs(img, tri)
        kt, et = torch.from_numpy(ktab).cuda(), torch.from_numpy(etab).cuda()
        rc = r0 * (1.0 + et[ph[si], ph[sj]])
        nx = img.shape[-1]
        if tri:
            odd = torch.round(X[1] / (math.sqrt(3.0) * 0.5)).long() % 2
            col, last = torch.round(X[0] - 0.5 * odd).long(), nx - 1 - odd
            rows = int(torch.round(X[1].max() / (math.sqrt(3.0) * 0.5))) + 1
            area = rows * math.sqrt(3.0) * 0.5
        else:
            col, last = X[0].long(), nx - 1
            area = float(np.prod(img.shape[:-1]))
        grip = (col == 0) | (col == last)
        fix = torch.zeros_like(X, dtype=torch.bool)
        fix[0] = grip
        if clamp:
            fix[:] = grip
        return cls(X, si, sj, kt[ph[si], ph[sj]], r0, rc * rc, fix, col == last, 0.5 * (nx - 1), (nx - 1) * area,
                   area, dt, damping)

    def strain(self, eps):
        self.x[0] = self.xc + (self.x[0] - self.xc) * ((1.0 + eps) / (1.0 + self.eps))
        self.grips(eps)
        self.eps = eps

    def grips(self, eps):
        f = self.fix[0]
        self.x[0] = torch.where(f, self.X[0] + eps * (self.X[0] - self.xc), self.x[0])
        self.v[0] *= self.free[0]
        self.a[0] *= self.free[0]

    def step(self, n, rate=None):
        dt, si, sj = self.dt, self.si, self.sj
        for q in range(n):
            vh = (self.v + 0.5 * dt * self.a) * self.free
            self.x = self.x + dt * vh
            if rate is not None:  # (strain before the call, strain per step)
                self.eps = rate[0] + (q + 1) * rate[1]
                self.grips(self.eps)
            d = self.x[:, sj] - self.x[:, si]
            r2 = (d * d).sum(0)
            self.intact = self.intact * (r2 <= self.rc2)
            r = torch.sqrt(r2)
            f = (self.k * (r - self.r0) / r * self.intact) * d
            F = torch.zeros_like(self.x)
            F.index_add_(1, si, f)
            F.index_add_(1, sj, -f)
            self.a = (F - self.damping * vh) * self.free
            self.v = vh + 0.5 * dt * self.a
        self.F, self.d, self.r, self.f = F, d, r, f

    def residual(self):
        return float(torch.maximum(self.F.abs(), self.v.abs()).mul(self.free).max())

    def sample(self):
        stretch = self.r - self.r0
        mv = (self.v[0] * self.v[0]).sum()
        return dict(eps=self.eps, sigma_vir=float(((self.d[0] * self.f[0]).sum() - mv) / self.omega),
                    sigma_grip=float(-self.F[0][self.right].sum() / self.area),
                    pe=float((0.5 * self.k * stretch * stretch * self.intact).sum()),
                    ke=float(0.5 * (self.v * self.v).sum()), residual=self.residual(), n_broken=None, step=None)

    def fields(self):
        """Virial stress and Lagrangian strain per particle of a void-free
        square lattice of unit spacing."""
        n = self.x.shape[1]
        st = torch.zeros((3, n), dtype=torch.float64, device="cuda")
        for q, (a, b) in enumerate(((0, 0), (1, 1), (0, 1))):
            w = 0.5 * self.d[a] * self.f[b]
            st[q].index_add_(0, self.si, w)
            st[q].index_add_(0, self.sj, w)
            st[q] -= self.v[a] * self.v[b]
        near = self.r0 < 1.2
        si, sj = self.si[near], self.sj[near]
        d0, d1 = self.X[:, sj] - self.X[:, si], self.x[:, sj] - self.x[:, si]
        A = torch.zeros((2, 2, n), dtype=torch.float64, device="cuda")
        B = torch.zeros_like(A)
        for a in range(2):
            for b in range(2):
                for M, w in ((A, d0[a] * d0[b]), (B, d1[a] * d0[b])):
                    M[a, b].index_add_(0, si, w)
                    M[a, b].index_add_(0, sj, w)
        J = torch.linalg.solve(A.permute(2, 0, 1), B.permute(2, 1, 0)).transpose(1, 2)
        E = 0.5 * (J.transpose(1, 2) @ J - torch.eye(2, dtype=torch.float64, device="cuda"))
        return st, torch.stack([E[:, 0, 0], E[:, 1, 1], E[:, 0, 1]])


def exact(case, seed):
    kind = case["kind"]
    if kind == "unet":
        return _exact_unet(case, seed)
    if kind in ("batch", "relax"):
        states, broken, us = [], [], []
        for img in _batch_images(case, seed):
            if kind == "batch":
                o = _Plain.image(img, K_TWO, E_TWO, False, False, 0.01, 0.1)
                for eps in _levels(case, True):
                    o.strain(eps)
                    o.step(case["steps"])
            else:
                o = _Plain.image(img, K_TWO, E_TWO, False, False, 0.5, 0.03)
                for i in range(case["increments"]):
                    o.strain(case["deps"] * (i + 1))
                    for _ in range(20000 // case["check"]):
                        o.step(case["check"])
                        if o.residual() <= case["tol"]:
                            break
                    us.append((o.x - o.X).reshape(2, case["side"], case["side"]))
            states.append((o.x, o.v))
            broken.append(None)
        if kind == "batch":
            return dict(states=states, broken=broken)
        n = case["increments"]
        out = dict(u=torch.stack([torch.stack(us[i::n]) for i in range(n)]))
        for i in range(n):
            out["taken%d" % i] = out["converged%d" % i] = None
        return out
    if kind == "network":
        net = _network(case, seed)
        t = {q: torch.from_numpy(net[q]).cuda() for q in ("X", "si", "sj", "k", "r0", "rc2", "fix", "grip")}
        o = _Plain(t["X"], t["si"].long(), t["sj"].long(), t["k"], t["r0"], t["rc2"], t["fix"] > 0, t["grip"] == 2,
                   net["xc"], net["omega"], net["grip_area"], 0.1, 0.02)
    else:
        img, k, e = _image(case, seed)
        o = _Plain.image(img, k, e, case["lattice"] == 1, case["nz"] > 1, 0.01, 0.1)
        if case["eps0"]:
            o.strain(case["eps0"])
    if case.get("rate"):
        per = (case["eps1"] - case["eps0"]) / (case["increments"] * case["steps"])
        for i in range(case["increments"]):
            o.step(case["steps"], (case["eps0"] + i * case["steps"] * per, per))
    else:
        for eps in _levels(case, True):
            o.strain(eps)
            o.step(case["steps"])
    out = dict(sample=o.sample(), broken=None, first_break=None, x=o.x, v=o.v)
    if case.get("fields"):
        out["stress"], out["strain"] = o.fields()
    return out


def _exact_unet(case, seed):
    x, target, params = _unet_inputs(case, seed)
    F = torch.nn.functional
    p = torch.from_numpy(params).double().cuda().requires_grad_(True)
    at = 0

    def conv(h):
        nonlocal at, q
        cin, cout = CONVS[q]
        q += 1
        w = p[at:at + cout * 9 * cin].reshape(cout, 3, 3, cin)
        b = p[at + cout * 9 * cin:at + cout * 9 * cin + cout]
        at += cout * 9 * cin + cout
        hp = F.pad(h, (0, 0, 1, 1, 1, 1))  # NHWC, one product per tap
        H, W = h.shape[1], h.shape[2]
        y = b
        for ky in range(3):
            for kx in range(3):
                y = y + hp[:, ky:ky + H, kx:kx + W] @ w[:, ky, kx].T
        return torch.relu(y)

    pool = lambda h: F.max_pool2d(h.permute(0, 3, 1, 2), 2).permute(0, 2, 3, 1)  # noqa: E731
    up = lambda h: h.repeat_interleave(2, 1).repeat_interleave(2, 2)  # noqa: E731
    q = 0
    e1 = conv(conv(x.double()))
    e2 = conv(conv(pool(e1)))
    e3 = conv(conv(pool(e2)))
    h = conv(conv(pool(e3)))
    for skip in (e3, e2, e1):
        h = conv(conv(torch.cat([up(h), skip], 3)))
    pred = h @ p[at:at + 64].reshape(2, 32).T + p[at + 64:at + 66]
    loss = ((pred - target.double()) ** 2).mean()
    loss.backward()
    return dict(pred=pred.detach(), loss=float(loss.detach()), grad=p.grad)
