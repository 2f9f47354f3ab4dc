"""What a context launches (hydro_get_launch), and that the variant it reports selects the same
launches when it is passed back, whichever kernels chose their march for themselves."""
import pytest

from paper_1204_4779_gb300 import hydro, inputs, tuner

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
F32, F64 = torch.float32, torch.float64

GRIDS = [((1024,), F64), ((2500,), F32), ((300, 77), F64), ((1024, 1024), F64), ((3001, 2003), F32),
         ((512, 512), F32), ((40, 36, 5), F32), ((128, 128, 128), F32), ((256, 256, 256), F32),
         ((97, 83, 75), F64), ((40, 36, 100), F64)]


@pytest.mark.parametrize("shape,dtype", GRIDS)
@pytest.mark.parametrize("bc", ["periodic", "outflow"])
def test_a_reported_variant_runs_the_same_launches(shape, dtype, bc):
    variants = [None]
    if len(shape) == 3:
        variants += [dict(march=20), dict(march=64), dict(split=1)]
        if dtype == F32:
            variants += [dict(staging=2), dict(staging=3), dict(tile=(32, 8)), dict(manifest=2)]
    elif len(shape) == 2:
        variants += [dict(split=1), dict(split=2)]
        variants += [dict(march=16), dict(march=64), dict(tile=(64, 1))] if dtype == F32 else \
            [dict(tile=(128, 1)), dict(tile=(128, 1), march=7)]
    for var in variants:
        A = hydro.Solver(shape, 1.4, bc=bc, dtype=dtype, variant=var)
        B = hydro.Solver(shape, 1.4, bc=bc, dtype=dtype, variant=A.variant())
        assert A.variant() == B.variant() and A.launch() == B.launch(), (var, A.launch(), B.launch())
        A.close()
        B.close()


@pytest.mark.parametrize("shape,dtype,variant,want", [
    ((1024,), F64, None, ("line", 0, 2)), ((1024,), F32, None, ("line", 0, 2)),
    ((2049,), F64, None, ("tile", 1, 1)),
    ((512, 512), F32, None, ("strip", 2, 2)), ((1024, 1024), F32, None, ("strip", 8, 2)),
    ((2048, 2048), F32, None, ("strip", 32, 2)), ((3001, 2003), F32, None, ("strip", 48, 2)),
    ((4096, 4096), F32, None, ("strip", 24, 2)),
    ((1024, 1024), F32, dict(march=12, split=1), ("strip", 12, 1)),
    ((1024, 1024), F64, None, ("strip", 21, 2)), ((300, 77), F64, dict(tile=(128, 1)), ("tile", 16, 2)),
    ((128, 128, 128), F32, None, ("strip", 22, 2)), ((256, 256, 256), F32, None, ("strip", 26, 2)),
    ((512, 512, 512), F32, None, ("strip", 128, 2)), ((512, 512, 512), F32, dict(march=40), ("strip", 40, 2)),
    ((128, 128, 128), F32, dict(march=40, staging=3), ("tile", 40, 2)),
    ((97, 83, 75), F64, None, ("tile", 25, 2)), ((97, 83, 75), F64, dict(march=32, split=1), ("tile", 32, 1))])
def test_launches_that_run(shape, dtype, variant, want):
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the expected marches are those of a 152-SM GPU")
    S = hydro.Solver(shape, 1.4, dtype=dtype, variant=variant)
    got = S.launch()
    S.close()
    assert (got["kernel"], got["march"], got["split"]) == want


def _state(shape):
    V = torch.from_numpy(inputs.smooth(shape, seed=5, vmax=0.3)).cuda()
    return hydro.prim_to_cons(V, 1.4).to(F32).contiguous()


@pytest.mark.parametrize("shape,kernel", [
    ((29, 200, 200), "tile"), ((32, 150, 150), "tile"), ((4, 384, 384), "tile"), ((61, 300, 100), "tile"),
    ((64, 16, 384), "tile"), ((28, 200, 200), "strip"), ((60, 150, 150), "strip"), ((29, 64, 48), "strip"),
    ((33, 200, 200), "strip"), ((2, 3, 5), "strip"), ((128, 128, 128), "strip")])
def test_narrow_grids_run_the_faster_kernel_with_the_same_result(shape, kernel):
    """One chunk of all planes leaves too few tiles for the rule, so that form runs the strips: the
    states agree bit for bit."""
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the rule's lines are those of a 152-SM GPU")
    A = hydro.Solver(shape, 1.4, bc=["periodic", "outflow", "periodic"], dtype=F32)
    B = hydro.Solver(shape, 1.4, bc=["periodic", "outflow", "periodic"], dtype=F32,
                     variant=dict(march=max(shape[2], 9)))
    assert A.launch()["kernel"] == kernel and B.launch()["kernel"] == "strip"
    U = _state(shape)
    W = U.clone()
    assert A.step(U, 5) == B.step(W, 5)
    assert torch.equal(U, W)


def test_host_stepping_on_a_narrow_grid():
    """The last step's tiles run slab by slab there, as the strips do."""
    shape = (29, 150, 151)
    S = hydro.Solver(shape, 1.4, dtype=F32)
    U = _state(shape)
    host = U.cpu().pin_memory()
    out = torch.empty_like(host).pin_memory()
    done = S.step(U, 3)
    assert S.step_host(torch.empty_like(U), host, out, 3) == done
    assert torch.equal(out, U.cpu())


@pytest.mark.parametrize("shape", [(512, 512), (1024, 1024), (2048, 2048), (4096, 4096), (300, 77),
                                   (64, 64, 64), (128, 128, 128), (160, 160, 160), (40, 36, 30)])
def test_the_tuner_can_name_the_default(shape):
    """Some variant of the tuner's space runs the launches of a solver created without one, so the
    best one found is no slower than that."""
    S = hydro.Solver(shape, 1.4, dtype=F32)
    want, default = S.launch(), S.variant()
    S.close()
    space = tuner.Space(len(shape))
    named = [v for v in map(space.variant, space.all_genomes())
             if all(default[k] == x for k, x in v.items())]
    assert len(named) == 1
    S = hydro.Solver(shape, 1.4, dtype=F32, variant=named[0])
    got = S.launch()
    S.close()
    assert got == want


def test_null_arguments():
    import ctypes
    lib = hydro.load_library()
    v = ctypes.c_int32()
    assert lib.hydro_get_launch(None, ctypes.byref(v), ctypes.byref(v), ctypes.byref(v)) == hydro.HYDRO_EINVAL
