"""The frequency-to-time transform at every kind of channel count against numpy's FP64 FFT."""
import numpy as np
import pytest

from paper_2201_08500_gb300 import bpm, workloads

pytestmark = pytest.mark.gpu


# one channel; each radix and mixtures of them; columns a block from 64 to one;
# primes and composites of large primes (chirp form, its lengths 32 ... 4096);
# the longest of either form, and the direct sum beyond
@pytest.mark.parametrize("n", [1, 2, 3, 5, 7, 8, 11, 16, 24, 49, 60, 97, 128, 201, 611, 1000, 1024,
                               1031, 2047, 2048, 2053, 3750, 4096])
def test_time_response_equals_the_fft_of_the_fields(n):
    w = workloads.tiny(n_ch=n)
    rng = np.random.default_rng(n)
    e = (rng.standard_normal((2, n, w.nx)) + 1j * rng.standard_normal((2, n, w.nx))).astype(
        np.complex64)
    p = bpm.plan_from_workload(w)
    p.set_fields(e[0], e[1], w.nz)
    p.run(0)
    p.sync()
    got = p.eh_time()
    p.close()
    dw = w.omega[1] - w.omega[0] if n > 1 else 1.0
    j = np.arange(n)
    turn = np.exp(2j * np.pi * ((j * (n // 2)) % n) / n)
    want = dw * turn[:, None] * np.fft.fft(e[1].astype(np.complex128), axis=0)
    # FP64 rounding of a transform of up to 4096 points, twice in the chirp form:
    # a few 1e-16 per octave (the direct sum: sqrt(n) terms), against the rms
    assert np.max(np.abs(got - want)) <= 2e-13 * np.sqrt(np.mean(np.abs(want) ** 2))
