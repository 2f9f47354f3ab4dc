"""Small 1D grids whose run takes more steps than one launch of the line kernel does (2048): the
state, time and step count of the grid kernels, bit for bit, with and without an end time, which is
reached in the second or third launch."""
import pytest

from paper_1204_4779_gb300 import inputs
from test_gpu_line import _run, _same

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
F32, F64 = torch.float32, torch.float64


@pytest.mark.parametrize("dtype", [F32, F64])
@pytest.mark.parametrize("bc", [0, 1])
def test_runs_of_several_launches(dtype, bc):
    V = inputs.smooth((64,), seed=4, vmax=0.3)
    _, t, done, _ = _same(V, bc, dtype, (5000,))
    assert done == [5000]
    for steps in (2048, 3000, 4097):
        end = _run(V, bc, dtype, (steps,))[1] * (1.0 + 1e-9)
        # a generous bound: the call stops launching once the device has reached the end
        _, t, done, _ = _same(V, bc, dtype, (12000,), t_end=end)
        assert t == end and steps <= done[0] <= steps + 1
