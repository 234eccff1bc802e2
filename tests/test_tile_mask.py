"""The broken flags' last word: the multi-step kernel sets a cell's flags by a 32-bit
atomic, which on grids of any size stays within the allocation."""
import os
import re
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2201_04565_gb300", "csrc")
CUDA = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")

HARNESS = r"""
#include "lsm_internal.h"
#include <cstdio>
int main()
{
    long bad = 0;
    for (int64_t np = 1; np < 5000; np++)
        for (int64_t g = np > 8 ? np - 8 : 0; g < np; g++)
            bad += (size_t)((g & ~(int64_t)3) + 4) > lsm::tile_mask_bytes(np);  // the word of cell g
    std::printf("%ld\n", bad);
    return bad != 0;
}
"""


def test_word_of_every_cell_is_allocated(tmp_path):
    src = open(os.path.join(CSRC, "kernels.cu")).read()
    assert re.findall(r"dalloc\(&c\.tmask, (.*)\)\);", src) == ["tile_mask_bytes(np)"]
    gxx = shutil.which("g++")
    if gxx is None or not os.path.exists(os.path.join(CUDA, "cuda_runtime.h")):
        pytest.skip("no g++ or no CUDA headers")
    (tmp_path / "t.cpp").write_text(HARNESS)
    subprocess.check_call([gxx, "-std=c++17", "-I", CSRC, "-I", CUDA, "-c", "-o", str(tmp_path / "t.o"),
                           str(tmp_path / "t.cpp")])
    subprocess.check_call([gxx, "-o", str(tmp_path / "t"), str(tmp_path / "t.o"), "-Wl,--unresolved-symbols=ignore-all"])
    assert subprocess.run([str(tmp_path / "t")], capture_output=True, text=True).stdout.strip() == "0"


@pytest.mark.gpu
@pytest.mark.parametrize("precision", ["df64", "exact64"])
@pytest.mark.parametrize("nx,ny", [(31, 9), (18, 3), (5, 1), (33, 31)])
def test_breaks_in_the_last_cells(precision, nx, ny):
    """Every spring of grids with 1, 2 and 3 cells in the last word breaks."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2201_04565_gb300 import lsm
    assert nx * ny % 4
    outs = []
    for path in (0, 2):
        g = lsm.Specimen.from_image(np.ones((ny, nx), np.uint8), np.ones((1, 1)), np.full((1, 1), 0.05),
                                    precision=precision, path=path)
        x = g.state()[0]
        g.set_state(1.5 * x, np.zeros_like(x))
        g.step(4)
        outs.append((*g.state(), *g.broken(), g.break_steps()))
        g.close()
    assert outs[0][2].all()
    assert all(np.array_equal(a, b) for a, b in zip(*outs))
