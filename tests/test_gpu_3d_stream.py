"""The streamed 3D passes at every pair of sizes against the plain ones."""
import numpy as np
import pytest

from paper_2201_08500_gb300 import bpm
from test_gpu_3d import case3d

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx", [256, 512, 1024])
@pytest.mark.parametrize("ny", [256, 512, 1024])
def test_streamed_passes_give_the_plain_passes_bits(nx, ny):
    """First, inner and last row passes and the column pass, over groups with one
    or two items and a ragged end; run whole (the default form) and in parts."""
    w = case3d(nx, ny, 7, 3 if nx * ny > 1 << 18 else 5, seed=nx + ny)
    w.tan_psi = 0.07
    out = []
    for form, steps in ((0, (7,)), (None, (7,)), (2, (1, 4, 2))):
        p = bpm.plan_from_workload(w)
        if form is not None:
            p.set_launch(form=form, row_threads=256 if form == 0 or nx == 1024 else 128)
        for n in steps:
            p.run(n)
        p.sync()
        out.append((p.e0(), p.eh(), *p.reflectivity()[:2]))
        p.close()
    for got in out[1:]:
        for a, b in zip(out[0], got):
            assert np.array_equal(a, b)
