"""The FP64 kernels' own quotients, roots and comparisons (exact64.cuh): a step equals the oracle's
plain IEEE operations bit for bit -- on ordinary states, on supersonic ones, and on states whose
values leave the range those quotients are exact in (tiny and huge densities, pressures and
momenta, where the plain operations take over), in every dimension."""
import numpy as np
import pytest

import oracle
from _helpers import shape_of
from paper_1204_4779_gb300 import hydro, inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SHAPES = [(97,), (41, 23), (19, 14, 11)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("vmax", [0.0, 1e-150, 0.3, 5.0])
@pytest.mark.parametrize("scale", [1.0, 1e-135, 1e135])
def test_step_equals_oracle_bitwise(shape, vmax, scale):
    """scale multiplies density and pressure (velocities and the time step stay): 1e+-135 lies
    outside the exact range of 2^+-400, so the plain operations run."""
    V = inputs.smooth(shape, seed=11, vmax=vmax)
    V[0] *= scale
    V[-1] *= scale
    bc = tuple(a % 2 for a in range(len(shape)))
    U0 = oracle.prim_to_cons(V, 1.4)
    O, _, n, _ = oracle.run(U0, 1.4, 0.4, 5, bc=bc, threads=oracle.max_threads())
    U = torch.from_numpy(U0.copy()).cuda()
    S = hydro.Solver(shape_of(V), 1.4, bc=list(bc), dtype=torch.float64, cfl=0.4)
    _, m = S.step(U, 5)
    assert m == n == 5
    assert np.array_equal(U.cpu().numpy(), O)
