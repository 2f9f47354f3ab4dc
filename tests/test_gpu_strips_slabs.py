"""The 3D FP32 strips in the chunks that their march makes: one chunk of all planes, evened chunks,
a last chunk of one plane; and stepping from and to host memory, whose last step launches them slab
by slab, where the slabs interleave and where they do not.  Each case first checks that the launch
has the form it is here for (the marches are those of a 152-SM GPU)."""
import pytest

from _helpers import gpu_state
from paper_1204_4779_gb300 import hydro, inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
F32 = torch.float32


def _solver(shape, bc, march):
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the expected marches are those of a 152-SM GPU")
    return hydro.Solver(shape, 1.4, bc=list(bc), dtype=F32, variant=dict(march=march) if march else None)


# shape, named march, planes a CTA marches through
@pytest.mark.parametrize("shape,march,planes", [
    ((300, 300, 5), 0, 5), ((300, 301, 9), 0, 9), ((420, 420, 23), 0, 23),      # all planes in one chunk
    ((420, 420, 23), 12, 12),                                                   # 12 and 11
    ((40, 36, 7), 3, 2), ((40, 36, 10), 5, 3), ((40, 36, 100), 40, 17)])        # 2 2 2 1; 3 3 3 1; 17 ... 15
@pytest.mark.parametrize("bc", [(0, 0, 0), (0, 1, 1)])
def test_chunks_equal_the_tiles(shape, march, planes, bc):
    A = _solver(shape, bc, march)
    assert A.launch() == dict(kernel="strip", march=planes, split=2)
    B = hydro.Solver(shape, 1.4, bc=list(bc), dtype=F32, variant=dict(staging=2, march=6))
    assert B.launch()["kernel"] == "tile"
    U = gpu_state(inputs.smooth(shape, seed=2, vmax=0.3), 1.4, F32)
    W = U.clone()
    assert A.step(U, 4) == B.step(W, 4)
    assert torch.equal(U, W)


@pytest.mark.parametrize("n_steps,t_end", [(1, 0.0), (3, 0.0), (5, 0.002)])
@pytest.mark.parametrize("shape,bc,march,planes,form", [
    ((40, 36, 100), (0, 0, 0), 40, 17, "interleaved"),    # six slabs, the last of 15 planes
    ((40, 36, 100), (0, 1, 1), 0, 2, "interleaved"),      # 50 chunks in eight slabs
    ((40, 36, 9), (0, 0, 0), 32, 5, "interleaved"),       # two slabs
    ((40, 36, 7), (0, 0, 0), 3, 2, "whole"),              # a last slab of one plane: stage 1 whole first
    ((40, 36, 10), (1, 0, 0), 5, 3, "whole"),
    ((24, 20, 57), (0, 0, 0), 0, 1, "whole")])            # chunks of one plane
def test_host_stepping_slab_by_slab(shape, bc, march, planes, form, n_steps, t_end):
    S = _solver(shape, bc, march)
    assert S.launch() == dict(kernel="strip", march=planes, split=2)
    chunks = -(-shape[2] // planes)
    last = shape[2] - chunks * (min(chunks, 8) - 1) // min(chunks, 8) * planes
    assert (planes >= 2 and last >= 2) == (form == "interleaved")
    U = gpu_state(inputs.blast_3d(shape=shape, radius_cells=4.0), 1.4, F32)
    Ud = U.clone()
    td, nd = S.step(Ud, n_steps, t_end=t_end)
    host = U.cpu().pin_memory()
    out = torch.full_like(host, float("nan")).pin_memory()
    dev = torch.empty_like(U)
    th, nh = S.step_host(dev, host, out, n_steps, t_end=t_end)
    assert (th, nh) == (td, nd)
    assert torch.equal(out, Ud.cpu()) and torch.equal(dev, Ud)
