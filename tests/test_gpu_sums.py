"""R and T of fields set at the exit: FP64 sums of the exact squares of FP32 values."""
import numpy as np
import pytest

from paper_2201_08500_gb300 import bpm
from test_gpu_3d import case3d
from test_gpu_parity import deformed_small

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["ordinary", "denormal", "huge", "mixed"])
@pytest.mark.parametrize("dims,nx,ny,n_ch", [(2, 256, 1, 3), (2, 4096, 1, 2), (2, 8192, 1, 1),
                                             (3, 256, 256, 3), (3, 256, 1024, 1)])
def test_sums_of_any_field_values(dims, nx, ny, n_ch, kind):
    r = np.random.default_rng(nx * ny)
    w = case3d(nx, ny, 4, n_ch, 1) if dims == 3 else deformed_small(nx, nz=4, n_ch=n_ch)
    f = r.standard_normal((2, n_ch, nx * ny, 2))
    scale = {"ordinary": 1.0, "denormal": 1e-41, "huge": 1e37}.get(kind)
    f *= 10.0 ** r.uniform(-44, 18, f.shape) if scale is None else scale
    f[r.random(f.shape) < 0.1] = 0.0
    f = f.astype(np.float32)
    p = bpm.plan_from_workload(w)
    p.run(0)
    p.sync()
    inc = (np.abs(p.e0().reshape(n_ch, -1).astype(np.complex128)) ** 2).sum(1)
    p.set_fields(*np.ascontiguousarray(f).view(np.complex64).reshape(2, n_ch, -1), 4)
    p.run(0)
    p.sync()
    R, T, _ = p.reflectivity()
    p.close()
    want = (f.astype(np.float64) ** 2).sum((2, 3))  # exact squares
    # sums of n positive FP64 terms, and the norm's FP32 rounding of each value
    tol = 2 * nx * ny * 2.0 ** -53 + 2.0 ** -22
    for got, s in ((T, want[0]), (R, want[1])):
        assert np.all(np.abs(got * inc / s - 1.0) <= tol)
