"""The FP64 strips of 2D grids (28 of 32 columns a warp) against the FP64 row tiles, bit for bit:
widths around one and two strips, heights of one to three rows and so tall that a warp marches
through several, with a short last chunk, every boundary pair, supersonic flow and the scheme
options."""
import pytest

from paper_1204_4779_gb300 import hydro, inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
F64 = torch.float64


def _same(shape, bc, vmax, scheme=(2, 0), steps=4):
    V = torch.from_numpy(inputs.smooth(shape, seed=shape[0] + shape[1], vmax=vmax)).cuda()
    U = hydro.prim_to_cons(V, 1.4).contiguous()
    A = hydro.Solver(shape, 1.4, bc=list(bc), dtype=F64, cfl=0.4)
    B = hydro.Solver(shape, 1.4, bc=list(bc), dtype=F64, cfl=0.4, variant=dict(tile=(128, 1), march=5))
    assert (A.launch()["kernel"], B.launch()["kernel"]) == ("strip", "tile")
    W = U.clone()
    A.set_scheme(*scheme)
    B.set_scheme(*scheme)
    assert A.step(U, steps) == B.step(W, steps)
    assert torch.equal(U, W), (shape, bc, scheme)
    return A.launch()["march"]


@pytest.mark.parametrize("nx", [1, 2, 3, 27, 28, 29, 30, 31, 32, 55, 56, 57, 58, 84, 85])
@pytest.mark.parametrize("bc", [(0, 0), (1, 1), (0, 1), (1, 0)])
def test_widths_and_marches(nx, bc):
    for ny in (1, 2, 3, 23):
        _same((nx, ny), bc, 0.3)
    march = _same((nx, 3001 + nx), bc, 0.3)
    if torch.cuda.get_device_properties(0).multi_processor_count <= 152:
        assert march > 1


@pytest.mark.parametrize("scheme", [(2, 0), (1, 0), (2, 1), (1, 1)])
@pytest.mark.parametrize("bc", [(0, 1), (1, 0)])
def test_supersonic_flow_and_scheme_options(scheme, bc):
    _same((61, 4003), bc, 4.0, scheme)
    _same((61, 17), bc, 4.0, scheme)
