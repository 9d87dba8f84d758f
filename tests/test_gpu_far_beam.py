"""The incident norm of beams whose centre is far off the grid: |S g|^2 of every cell in
FP64, also where |g|^2 alone is below its range."""
import numpy as np
import pytest

from paper_2201_08500_gb300 import bpm, workloads
from test_gpu_parity import deformed_small

pytestmark = pytest.mark.gpu


# waists from the centre to the grid's edge, and the amplitude's decimal exponent
@pytest.mark.parametrize("waists,mag", [(0.0, 0), (10.0, 20), (14.0, 0), (14.3, -40), (18.0, 0),
                                        (19.5, 12), (20.5, 25), (24.0, 120), (24.0, 200)])
@pytest.mark.parametrize("dims,nx,ny,side,zx", [(2, 256, 1, -1, 0.0), (2, 4096, 1, 1, 0.0),
                                                (2, 1024, 1, -1, 6e-4), (3, 256, 512, 1, 4e-4)])
def test_norm_of_a_beam_off_the_grid(dims, nx, ny, side, zx, waists, mag):
    n_ch = 3
    w = workloads.large_3d(n_ch=n_ch, nx=nx, ny=ny, nz=4, with_u=False) if dims == 3 else \
        deformed_small(nx, nz=4, n_ch=n_ch, seed=2)
    w.w0, w.zx, w.zR = 4 * w.dx, zx, 1e-3
    edge = 0.0 if side < 0 else (nx - 1) * w.dx
    w.x0 = edge + side * waists * w.w0
    w.S = 10.0 ** mag * np.array([1.0, 0.3j, -0.7 + 0.2j])
    p = bpm.plan_from_workload(w)
    p.run(0)
    p.sync()
    R = p.reflectivity()[0]
    assert np.all(R == 0.0)  # nothing in Eh, and a norm above zero
    # the norm through the T of one cell of 2^-40
    f = np.zeros((n_ch, ny * nx), np.complex64)
    f[:, 17] = 2.0 ** -40
    p.set_fields(f, 0 * f, 4)
    p.run(0)
    p.sync()
    T = p.reflectivity()[1]
    p.close()
    den = 1.0 + 1j * zx / w.zR
    x = np.arange(nx) * w.dx
    y = (np.arange(ny) - ny // 2) * w.dy if dims == 3 else np.zeros(1)
    rr = ((x - w.x0)[None, :] ** 2 + y[:, None] ** 2) / w.w0 ** 2
    power = -2.0 * rr * (1.0 / den).real
    top = power.max()
    # log of sum |S pref g|^2 (pref = den^-1 in 3D, den^-1/2 in 2D)
    log_inc = 2 * np.log(np.abs(w.S)) - (2 if dims == 3 else 1) * np.log(np.abs(den)) + top + \
        np.log(np.sum(np.exp(power - top)))
    log_inc = np.log(np.exp(log_inc))  # as the FP64 number that it is, denormal below e^-708
    got = -80 * np.log(2.0) - np.log(T)
    # the exponents reach 1400: a few roundings of them and of the logarithms
    assert np.max(np.abs(got - log_inc)) <= 16 * 1400 * 2.0 ** -53
