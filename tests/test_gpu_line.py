"""Small 1D grids, whose steps run in one launch of a thread-block cluster, against the grid kernels
(profiling launches those one by one): the same states, times, step counts and status, bit for
bit, at sizes around the clusters' and warps' edges, in both precisions, with both boundaries, the
scheme options, time clipping, runs continued across calls and failing states."""
import numpy as np
import pytest

from _helpers import gpu_state
from paper_1204_4779_gb300 import hydro, inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
F32, F64 = torch.float32, torch.float64


def _run(V, bc, dtype, calls, scheme=(2, 0), t_end=0.0, cfl=0.4, profiling=False):
    U = gpu_state(V, 1.4, dtype)
    S = hydro.Solver((V.shape[1],), 1.4, bc=[bc], dtype=dtype, cfl=cfl)
    S.set_scheme(*scheme)
    S.set_profiling(profiling)
    t, done, status = 0.0, [], 0
    for n in calls:
        try:
            t, k = S.step(U, n, t_end=t_end, t=t)
            done.append(k)
        except hydro.HydroError as e:
            status = e.status
            break
    return U.cpu().numpy(), t, done, status


def _same(V, bc, dtype, calls, **kw):
    a = _run(V, bc, dtype, calls, **kw)
    b = _run(V, bc, dtype, calls, profiling=True, **kw)
    assert np.array_equal(a[0], b[0], equal_nan=True) and a[1:] == b[1:], (V.shape, bc, dtype)
    return a


@pytest.mark.parametrize("dtype", [F32, F64])
@pytest.mark.parametrize("n", [31, 32, 33, 63, 64, 65, 95, 127, 128, 129, 500, 1023, 1024, 1025, 2047, 2048, 2049])
def test_line_equals_grid_kernels(n, dtype):
    _same(inputs.smooth((n,), seed=n, vmax=0.3), n % 2, dtype, (7, 3))


@pytest.mark.parametrize("dtype", [F32, F64])
@pytest.mark.parametrize("bc", [0, 1])
@pytest.mark.parametrize("scheme", [(2, 0), (1, 0), (2, 1), (1, 1)])
def test_line_scheme_options_and_shocks(scheme, bc, dtype):
    _, t, done, _ = _same(inputs.sod_1d(300), bc, dtype, (1000,), scheme=scheme, t_end=0.1)
    assert t == 0.1 and done[0] < 1000


@pytest.mark.parametrize("dtype", [F32, F64])
def test_line_supersonic(dtype):
    _same(inputs.smooth((777,), seed=3, vmax=4.0), 0, dtype, (40,))


@pytest.mark.parametrize("dtype", [F32, F64])
def test_line_reports_a_failing_state(dtype):
    """A Courant number of 20 makes the scheme unstable: some step leaves a non-positive state."""
    _, _, _, status = _same(inputs.sod_1d(200), 1, dtype, (400,), cfl=20.0)
    assert status == hydro.HYDRO_ENONFINITE


# ---- totals, conversions and the CFL pass with wide accesses (FP32) ------------------------------

@pytest.mark.parametrize("n", [1, 3, 4, 5, 1023, 4095, 4096, 4097, 10007, 300001])
def test_audit_passes_on_any_length_and_alignment(n):
    """Planes on 16-byte boundaries take four cells an access, others one; both against FP64."""
    V = inputs.smooth((n,), seed=n, vmax=0.3)
    U = gpu_state(V, 1.4, F32)
    S = hydro.Solver((n,), 1.4, dtype=F32, cfl=0.4)
    flat = torch.zeros(3 * n + 1, dtype=F32, device="cuda")
    W = flat[1:].view(3, n)
    W.copy_(U)
    ref = U.double().sum(1).cpu().numpy() / n
    for X in (U, W):
        t = S.totals(X)
        got = np.array([t[0], t[1], t[4]])
        # the sums carry 48 bits
        assert np.all(np.abs(got - ref) <= 1e-13 * U.double().abs().sum(1).cpu().numpy() / n)
    assert S.cfl_dt(U) == S.cfl_dt(W)
    assert torch.equal(hydro.cons_to_prim(U, 1.4), hydro.cons_to_prim(W, 1.4))
    assert torch.equal(hydro.prim_to_cons(U, 1.4), hydro.prim_to_cons(W, 1.4))
