"""The per-step kernels of linear waves above 16384 cells, where the small grids' cluster kernel
ends: the four-cell and one-cell FP32 kernels and the two-cell and one-cell FP64 kernels, at sizes
whose last pair or quadruple falls inside a warp, with arrays on and off 16-byte boundaries."""
import math

import numpy as np
import pytest

from oracle import wave_oracle as W
from test_gpu_wave import _fp32_steps

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
C = 3.43


def _run(f0, g0, dtype, dt, steps, offset):
    """hydro_wave_run on arrays that start `offset` values past a 16-byte boundary."""
    from paper_1204_4779_gb300 import hydro
    n = len(f0)
    f, g = (torch.zeros(n + offset, dtype=dtype, device="cuda")[offset:] for _ in range(2))
    f.copy_(torch.from_numpy(f0))
    g.copy_(torch.from_numpy(g0))
    assert f.data_ptr() % 16 == offset * f.element_size()
    E = np.array(hydro.wave_run(f, g, C, 2 * math.pi, dt, steps))
    return f.cpu().numpy(), g.cpu().numpy(), E


# n a multiple of four on a boundary: the four-cell kernel, else the one-cell kernel
@pytest.mark.parametrize("n", [16385, 16386, 16388, 16391, 16516, 17408, 17412, 40000])
@pytest.mark.parametrize("offset", [0, 1, 2])
def test_fp32_states_and_energies(n, offset):
    f0, g0 = W.initial(n)
    dx = 2 * math.pi / n
    dt = dx / C
    f, g, E = _run(f0, g0, torch.float32, dt, 40, offset)
    fe, ge, Ee = _fp32_steps(f0, g0, dt, C * C * dt / (dx * dx), C * C, dx, 40)
    assert np.array_equal(f, fe) and np.array_equal(g, ge)
    # the same FP32 states: the energies differ by the FP64 rounding of the sums alone
    assert np.max(np.abs(E - Ee)) <= 1e-13 * Ee.mean()


# even n on a boundary: the two-cell kernel (512 cells a CTA), else the one-cell kernel
@pytest.mark.parametrize("n", [16385, 16386, 16388, 16446, 16450, 16896, 16898, 40000])
@pytest.mark.parametrize("offset", [0, 1])
def test_fp64_states_and_energies(n, offset):
    f0, g0 = W.initial(n)
    dt = 2 * math.pi / n / C
    fo, go, Eo = W.run(f0, g0, C, 2 * math.pi, dt, 40)
    f, g, E = _run(f0, g0, torch.float64, dt, 40, offset)
    assert np.array_equal(f, fo) and np.array_equal(g, go)
    # each term is the square of a difference that cancels by up to n / (2 pi)
    assert np.max(np.abs(E - Eo)) <= 2.0 ** -53 * n * Eo.mean()
