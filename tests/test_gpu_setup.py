"""Setup kernels (propagator tables, coefficients) over every bin and channel grouping."""
import numpy as np
import pytest

from paper_2201_08500_gb300 import bpm, workloads
from test_gpu_parity import deformed_small

pytestmark = pytest.mark.gpu

T4 = 1.0 / (2.0 - 2.0 ** (1.0 / 3.0))


@pytest.mark.parametrize("nx,order", [(256, 1), (512, 2), (1024, 4), (2048, 1), (4096, 4),
                                      (8192, 1)])
def test_every_bin_of_the_propagators(nx, order):
    """White noise through one step without crystal: all bins carry the same
    weight, the Nyquist bin (whose mirror is off the grid) among them."""
    w = deformed_small(nx, nz=1, n_ch=2, seed=nx)
    w.thickness, w.u, w.split_order = 0.0, None, order
    rng = np.random.default_rng(nx)
    e = (rng.standard_normal((2, 2, nx)) + 1j * rng.standard_normal((2, 2, nx))).astype(np.complex64)
    p = bpm.plan_from_workload(w)
    p.set_fields(e[0], e[1], 0)
    p.run()
    p.sync()
    got = np.stack([p.e0(), p.eh()])
    p.close()
    k = (w.omega / workloads.C_LIGHT)[:, None]
    h = 4.0 * np.pi * np.sin(w.theta_B) / w.lambda_B
    q = 2.0 * np.pi * np.fft.fftfreq(nx, w.dx)[None, :]
    spec = np.fft.fft(e.astype(np.complex128), axis=-1)
    for env, sign in enumerate((1.0, -1.0)):
        Q2 = (q + sign * 0.5 * h) ** 2
        # the fractions t, 1 - 2t, t of the fourth order add up to one step
        ph = -w.dz * Q2 / (np.sqrt(k * k - Q2) + k)
        want = spec[env] * np.exp(1j * ph)
        have = np.fft.fft(got[env].astype(np.complex128), axis=-1)
        # FP32 transforms (a few 1e-7 rms a propagation), per bin against the rms bin
        rms = np.sqrt(np.mean(np.abs(want) ** 2))
        assert np.max(np.abs(have - want)) <= 1e-5 * rms
        nyq = np.max(np.abs(have - want)[:, nx // 2])
        assert nyq <= 5e-6 * rms


@pytest.mark.parametrize("nx,n_ch", [(4096, 309), (1024, 611), (256, 67)])
def test_channel_groups_of_the_setup(nx, n_ch):
    """Setup blocks take up to eight channels (309 and 611 leave a remainder):
    each channel's fields are bitwise those of a plan of its own."""
    w = deformed_small(nx, nz=3, n_ch=n_ch, seed=5)
    p = bpm.plan_from_workload(w)
    p.run()
    p.sync()
    e0, eh, R = p.e0(), p.eh(), p.reflectivity()[0]
    p.close()
    for ch in (0, 7, 8, n_ch // 2, n_ch - 2, n_ch - 1):
        q = bpm.plan_from_workload(w.subset([ch]))
        q.run()
        q.sync()
        assert np.array_equal(q.e0()[0], e0[ch]) and np.array_equal(q.eh()[0], eh[ch])
        assert q.reflectivity()[0][0] == R[ch]
        q.close()


@pytest.mark.parametrize("dims,nx,ny,n_ch,zx", [(2, 256, 1, 1, 0.0), (2, 512, 1, 9, 3e-4),
                                                (2, 4096, 1, 309, 0.0), (2, 8192, 1, 3, -2e-4),
                                                (3, 256, 512, 2, 0.0), (3, 1024, 256, 3, 4e-4)])
def test_incident_field_and_norm(dims, nx, ny, n_ch, zx):
    """Every cell of the incident field against the formula in FP64, from cells
    that round to zero to amplitudes far from one, and the norm through T."""
    w = workloads.large_3d(n_ch=n_ch, nx=nx, ny=ny, nz=1, with_u=False) if dims == 3 else \
        deformed_small(nx, nz=1, n_ch=n_ch, seed=2)
    w.zx, w.zR = zx, 1e-3
    w.w0 = (6 if n_ch > 8 else nx // 20) * w.dx
    rng = np.random.default_rng(nx)
    w.S = rng.standard_normal(n_ch) * 10.0 ** rng.integers(-24, 4, n_ch) * np.exp(
        1j * rng.uniform(0, 6, n_ch))
    p = bpm.plan_from_workload(w)
    p.run(0)
    p.sync()
    got, R, T = p.e0().reshape(n_ch, ny, nx), *p.reflectivity()[:2]
    assert not p.eh().any()
    p.close()
    x = np.arange(nx) * w.dx
    y = (np.arange(ny) - ny // 2) * w.dy if dims == 3 else np.zeros(1)
    den = 1.0 + 1j * zx / w.zR
    r2 = ((x - w.x0)[None, :] ** 2 + y[:, None] ** 2) / w.w0 ** 2
    g = np.exp(-r2 / den) / (den if dims == 3 else np.sqrt(den))
    h = 4.0 * np.pi * np.sin(w.theta_B) / w.lambda_B
    dq = w.omega / workloads.C_LIGHT * np.sin(w.theta_i) - 0.5 * h
    want = w.S[:, None, None] * g * np.exp(1j * dq[:, None, None] * x)
    # dq is a difference of numbers 1e5 times larger: its FP64 rounding (8e-6 per
    # metre) moves the phase by at most 1e-7 over the grid; FP32 rounds to 6e-8
    # (1e-45 where it is denormal)
    assert np.max(np.abs(got - want) - 3e-7 * np.abs(want)) <= 2e-45
    assert np.all(R == 0.0) and np.max(np.abs(T - 1.0)) < 2e-7
