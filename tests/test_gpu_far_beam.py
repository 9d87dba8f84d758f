"""The incident norm of beams whose centre is far off the grid: |S g|^2 of every cell in
FP64, also where |g|^2 alone is below its range."""
import numpy as np
import pytest

from paper_2201_08500_gb300 import bpm, workloads
from test_gpu_parity import deformed_small

pytestmark = pytest.mark.gpu


def check(w):
    n_ch, nx, ny, zx = w.n_ch, w.nx, w.ny, w.zx
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
    y = (np.arange(ny) - ny // 2) * w.dy if w.dims == 3 else np.zeros(1)

    def log_norm(x):
        rr = (x[None, :] ** 2 + y[:, None] ** 2) / w.w0 ** 2
        power = (-2.0 * rr * (1.0 / den).real).astype(np.float64)
        top = power.max()
        # log of sum |S pref g|^2 (pref = den^-1 in 3D, den^-1/2 in 2D)
        s = 2 * np.log(np.abs(w.S)) - (2 if w.dims == 3 else 1) * np.log(np.abs(den)) + top + \
            np.log(np.sum(np.exp(power - top)))
        return np.log(np.exp(s))  # as the FP64 number that it is, denormal below e^-708

    # j dx - x0 cancels next to the centre: with j dx rounded, or fused into the difference
    j = np.arange(nx)
    want = [log_norm(j * w.dx - w.x0), log_norm(j.astype(np.longdouble) * w.dx - w.x0)]
    got = -80 * np.log(2.0) - np.log(T)
    # the exponents reach 1400: a few roundings of them and of the logarithms
    assert min(np.max(np.abs(got - x)) for x in want) <= 16 * 1400 * 2.0 ** -53


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
    check(w)


@pytest.mark.parametrize("mag", [12, 25, 200])
@pytest.mark.parametrize("dims,nx,ny", [(2, 512, 1), (2, 8192, 1), (3, 256, 256)])
def test_norm_of_a_beam_between_two_cells(dims, nx, ny, mag):
    """A waist of 1/39 of the grid's step, halfway between cells: 19.5 waists to either."""
    w = workloads.large_3d(n_ch=2, nx=nx, ny=ny, nz=4, with_u=False) if dims == 3 else \
        deformed_small(nx, nz=4, n_ch=2, seed=2)
    w.w0, w.x0 = w.dx / 39, (nx - 6.5) * w.dx
    w.S = 10.0 ** mag * np.array([1.0, 0.6 - 0.3j])
    check(w)
