"""Small linear-wave grids, whose steps run in one launch of a thread-block cluster: sizes around the
clusters' and warps' edges and the largest the cluster takes, against the FP64 oracle's states and
energies, FP32 states against the same run cut into single-step calls, and a run of more steps than
one launch takes."""
import math

import numpy as np
import pytest

from oracle import wave_oracle as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
C = 3.43


@pytest.mark.parametrize("n", [3, 31, 32, 33, 127, 128, 129, 1025, 4096, 4097, 16383, 16384, 16385])
def test_fp64_matches_oracle_at_the_edges(n):
    from paper_1204_4779_gb300 import hydro
    f0, g0 = W.initial(n)
    dt = 2 * math.pi / n / C
    fo, go, Eo = W.run(f0, g0, C, 2 * math.pi, dt, 21)
    f, g = torch.from_numpy(f0.copy()).cuda(), torch.from_numpy(g0.copy()).cuda()
    E = np.array(hydro.wave_run(f, g, C, 2 * math.pi, dt, 21))
    # the update's operations are the oracle's, in its order: the states are the same
    assert np.array_equal(f.cpu().numpy(), fo) and np.array_equal(g.cpu().numpy(), go)
    # the energy sums n squares of differences that cancel by up to n / (2 pi) (test_gpu_wave.py)
    assert np.max(np.abs(E - Eo)) <= max(1e-13, 2.0 ** -53 * n) * Eo.mean()


@pytest.mark.parametrize("n", [17, 640, 5000])
def test_fp32_run_equals_its_single_steps(n):
    from paper_1204_4779_gb300 import hydro
    f0, g0 = W.initial(n)
    dt = 2 * math.pi / n / C
    f, g = (torch.from_numpy(a).float().cuda() for a in (f0, g0))
    a, b = f.clone(), g.clone()
    E = hydro.wave_run(f, g, C, 2 * math.pi, dt, 40)
    single = [hydro.wave_run(a, b, C, 2 * math.pi, dt, 1)[0] for _ in range(40)]
    assert torch.equal(f, a) and torch.equal(g, b) and E == single


def test_more_steps_than_a_launch():
    from paper_1204_4779_gb300 import hydro
    n, steps = 96, 5000
    f0, g0 = W.initial(n)
    dt = 2 * math.pi / n / C
    fo, go, Eo = W.run(f0, g0, C, 2 * math.pi, dt, steps)
    f, g = torch.from_numpy(f0.copy()).cuda(), torch.from_numpy(g0.copy()).cuda()
    E = np.array(hydro.wave_run(f, g, C, 2 * math.pi, dt, steps))
    assert len(E) == steps
    assert np.array_equal(f.cpu().numpy(), fo) and np.array_equal(g.cpu().numpy(), go)
    assert np.max(np.abs(E - Eo)) <= 1e-13 * Eo.mean()
