"""The FP32 strip kernels of 2D grids (row tiles): widths around the edges of a strip (60 stored
columns of 64) and of its lane pairs, even (64-bit accesses) and odd (32-bit) rows, chunks of one
row to all rows, every boundary pair, subsonic and supersonic flow in both directions and the
scheme options, each against the FP64 oracle; and planes that start on odd words."""
import numpy as np
import pytest

from _helpers import gpu_state, oracle_run
from paper_1204_4779_gb300 import hydro, inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
F32 = torch.float32

# Eight steps of two stages, each a chain of some twenty rounded FP32 operations on values of the
# field's size: at most 8 * 2 * 20 * 2^-24 = 1.9e-5 of the field's largest value.
TOL = 2e-5
STEPS = 8


def _fields(nx, ny, vmax, seed):
    return inputs.smooth((nx, ny), seed=seed, vmax=vmax)


def _check(V, bc, march, scheme=None):
    shape = (V.shape[2], V.shape[1])
    U = gpu_state(V, 1.4, F32)
    S = hydro.Solver(shape, 1.4, bc=list(bc), dtype=F32, cfl=0.4,
                     variant=dict(march=march) if march else None)
    order, riemann = scheme or (2, 0)
    S.set_scheme(order, riemann)
    S.step(U, STEPS)
    O, _, n, _ = oracle_run(V, 1.4, bc, 0.4, STEPS, order=order, riemann=riemann)
    assert n == STEPS
    G = U.double().cpu().numpy()
    for k in range(4):
        assert np.max(np.abs(G[k] - O[k])) <= TOL * np.max(np.abs(O[k])), (k, shape, bc, march)


@pytest.mark.parametrize("nx", [1, 2, 3, 4, 58, 59, 60, 61, 62, 63, 64, 119, 120, 121, 122, 241, 242])
@pytest.mark.parametrize("bc", [(0, 0), (1, 1), (0, 1), (1, 0)])
def test_strip_widths(nx, bc):
    ny = 1 + (7 * nx) % 23
    _check(_fields(nx, ny, 0.2, nx), bc, 1 + nx % 5)


@pytest.mark.parametrize("march", [0, 1, 2, 3, 7, 64])
@pytest.mark.parametrize("nx", [66, 67])
def test_chunks_of_rows(nx, march):
    _check(_fields(nx, 41, 0.2, march), (0, 1), march)


@pytest.mark.parametrize("shape", [(124, 37), (125, 38)])
@pytest.mark.parametrize("scheme", [(2, 0), (1, 0), (2, 1), (1, 1)])
def test_supersonic_flow_and_scheme_options(shape, scheme):
    """Velocities up to 4 against sound speeds of about 1: faces of all four kinds."""
    _check(_fields(*shape, 4.0, 5), (0, 0), 5, scheme)


@pytest.mark.parametrize("nx", [64, 65])
def test_planes_on_odd_words(nx):
    """Planes 4 bytes past an 8-byte boundary run the 32-bit accesses: the same state, bit for
    bit, as aligned planes."""
    ny = 19
    U = gpu_state(_fields(nx, ny, 0.5, 9), 1.4, F32)
    S = hydro.Solver((nx, ny), 1.4, dtype=F32, cfl=0.4)
    flat = torch.zeros(4 * nx * ny + 1, dtype=F32, device="cuda")
    W = flat[1:].view(4, ny, nx)
    W.copy_(U)
    assert W.data_ptr() % 8 == 4
    S.step(U, STEPS)
    S.step(W, STEPS)
    assert torch.equal(U, W)
