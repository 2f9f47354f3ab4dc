"""Accuracy of the linear wave's energies on small grids, whose CTAs each leave a sum per step."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
C = 3.43


@pytest.mark.parametrize("n", [1024, 3072, 3001, 9000])
def test_energies_against_more_than_64_bits(n):
    """The states are the update formulas' own IEEE operations; the energy of each, K1 sum D^2 +
    K2 sum G^2, in long double from them.  A tree of sums of depth about 12 over positive terms
    rounds by some 0.8-0.9e-16 rms (2^-53 / sqrt(3) per level, most of it in the last few, where the
    sums are a sizeable part of the total); 16 sums added in a row at the end, by 1.1e-16."""
    from paper_1204_4779_gb300 import hydro
    L = np.longdouble
    if np.finfo(L).nmant < 60:
        pytest.skip("long double is no wider than double here")
    x = np.arange(n) * (2 * math.pi / n)
    dx = 2 * math.pi / n
    dt = dx / C
    k = C * C * dt / (dx * dx)
    k1, k2 = C * C * dx / (8.0 * dx * dx), dx / 8.0
    rel = []
    for phase in (0.3, 1.7, 4.0):
        f, g = np.sin(x + phase), np.cos(3 * x + 2 * phase)
        E = hydro.wave_run(torch.from_numpy(f.copy()).cuda(), torch.from_numpy(g.copy()).cuda(), C,
                           2 * math.pi, dt, 200)
        for e in E:
            f = f + dt * g
            fp, fm = np.roll(f, -1), np.roll(f, 1)
            g1 = g + k * (fp + fm - 2.0 * f)
            exact = L(k1) * ((L(1) * fp - fm) ** 2).sum() + L(k2) * ((L(1) * g + g1) ** 2).sum()
            rel.append(float((L(e) - exact) / exact))
            g = g1
    assert np.sqrt(np.mean(np.square(rel))) <= 1.0e-16
