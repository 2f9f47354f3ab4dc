"""The FP32 strip kernels of 2D grids (row tiles) and 3D grids (the default tile): widths around
the edges of a strip (60 stored columns of 64; in 3D also 28 of 32) and of its lane pairs, heights
around a CTA's rows (7 and 14), even (64-bit accesses) and odd (32-bit) rows, chunks of one row or
plane to all of them, every boundary pair, subsonic and supersonic flow in both directions and the
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
    shape = tuple(reversed(V.shape[1:]))
    U = gpu_state(V, 1.4, F32)
    S = hydro.Solver(shape, 1.4, bc=list(bc), dtype=F32, cfl=0.4,
                     variant=dict(march=march) if march else None)
    order, riemann = scheme or (2, 0)
    S.set_scheme(order, riemann)
    S.step(U, STEPS)
    O, _, n, _ = oracle_run(V, 1.4, bc, 0.4, STEPS, order=order, riemann=riemann)
    assert n == STEPS
    G = U.double().cpu().numpy()
    for k in range(len(V)):
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


# ---- 3D ----------------------------------------------------------------------------------------

@pytest.mark.parametrize("nx", [1, 2, 3, 27, 28, 29, 30, 56, 57, 59, 60, 61, 62, 84, 85, 119, 120, 121, 122])
@pytest.mark.parametrize("bc", [(0, 0, 0), (1, 1, 1), (0, 1, 0), (1, 0, 1)])
def test_3d_strip_widths(nx, bc):
    ny, nz = 1 + (5 * nx) % 17, 1 + (3 * nx) % 7
    _check(inputs.smooth((nx, ny, nz), seed=nx, vmax=0.2), bc, nx % 4)


@pytest.mark.parametrize("ny", [1, 2, 6, 7, 8, 13, 14, 15, 21, 28, 29])
@pytest.mark.parametrize("nx", [26, 60])
def test_3d_rows_of_a_cta(nx, ny):
    """nx = 26 takes the 16-lane rows (14 a CTA) from 8 rows on, nx = 60 the 32-lane ones."""
    _check(inputs.smooth((nx, ny, 6), seed=ny, vmax=0.2), (0, ny % 2, 1), 4)


@pytest.mark.parametrize("march", [0, 1, 2, 5, 64])
@pytest.mark.parametrize("nx", [31, 64])
def test_3d_chunks_of_planes(nx, march):
    _check(inputs.smooth((nx, 17, 23), seed=march, vmax=0.2), (1, 0, 0), march)


@pytest.mark.parametrize("shape", [(62, 16, 9), (27, 15, 8)])
@pytest.mark.parametrize("scheme", [(2, 0), (1, 0), (2, 1), (1, 1)])
def test_3d_supersonic_flow_and_scheme_options(shape, scheme):
    _check(inputs.smooth(shape, seed=3, vmax=4.0), (0, 0, 0), 3, scheme)


@pytest.mark.parametrize("nx", [62, 63, 26])
def test_3d_planes_on_odd_words(nx):
    ny, nz = 15, 6
    U = gpu_state(inputs.smooth((nx, ny, nz), seed=4, vmax=0.5), 1.4, F32)
    S = hydro.Solver((nx, ny, nz), 1.4, dtype=F32, cfl=0.4)
    flat = torch.zeros(5 * nx * ny * nz + 1, dtype=F32, device="cuda")
    W = flat[1:].view(5, nz, ny, nx)
    W.copy_(U)
    assert W.data_ptr() % 8 == 4
    S.step(U, STEPS)
    S.step(W, STEPS)
    assert torch.equal(U, W)
