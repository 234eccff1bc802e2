"""The schedule a new batch starts with against the ones that can be set: none of
them is clearly faster."""
import time

import numpy as np
import pytest

from gen.images import two_phase_materials

pytestmark = pytest.mark.gpu


def _per_step(b):
    b.step(20)
    b.synchronize()
    best = 1.0
    for _ in range(5):
        t = time.perf_counter()
        for _ in range(4):
            b.step(20)
        b.synchronize()
        best = min(best, time.perf_counter() - t)
    return best


# F32: on both sides of the tile height's line, many narrow specimens (three strips
# for two tiles) and few wide ones; strips of 16 rows for one to three times the warps
@pytest.mark.parametrize("precision,count,side,bound", [("f32", 6, 200, 1.1), ("f32", 5, 200, 1.1), ("f32", 200, 64, 1.1),
                                                        ("f32", 24, 150, 1.1), ("df64", 60, 256, 1.05),
                                                        ("df64", 24, 256, 1.05), ("f32", 60, 256, 1.05)])
def test_default_schedule_is_among_the_fastest(precision, count, side, bound):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2201_04565_gb300 import batch as B
    k, e, _ = two_phase_materials()
    rng = np.random.default_rng(1)
    imgs = [1 + (rng.random((side // 8 + 1, side // 8 + 1)) < 0.3).repeat(8, 0).repeat(8, 1)[:side, :side].astype(np.uint8)
            for _ in range(count)]
    b = B.Batch(imgs, k, e, precision=precision)
    b.apply_strain(0.01)
    default = _per_step(b)
    others = []
    for ty in (8, 16, -8, -16):
        b.set_schedule(ty, 0, 1)
        others.append(_per_step(b))
    b.close()
    assert default < bound * min(others)
