"""Which calls take several steps per launch, and that those that do give the bits of
single steps: every case here asserts that its calls reach the kernel."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

TAUS = {2: [0.7, 1.0, 0.7], 3: [0.7, 1.0, 0.7, 1.0, 0.7]}


@pytest.fixture(scope="module")
def lbm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1808_04406_gb300 import build as libbuild
    libbuild.build()
    from paper_1808_04406_gb300 import lbm as L
    L.load()
    return L


def _sim(lbm, lattice, dims, storage="f32"):
    if lattice.startswith("E"):
        return lbm.HermiteSimulation(lattice, dims, TAUS[2], storage=storage)
    return lbm.Simulation(lattice, dims, TAUS[len(dims)], storage=storage)


def _fields(dims):
    g = torch.Generator(device="cuda").manual_seed(7)
    N, D = int(np.prod(dims)), len(dims)
    return (1.0 + 0.02 * (torch.rand(N, generator=g, device="cuda", dtype=torch.float64) - 0.5),
            0.05 * (torch.rand(D, N, generator=g, device="cuda", dtype=torch.float64) - 0.5))


def _run(lbm, monkeypatch, lattice, dims, calls, mode, several):
    sim = _sim(lbm, lattice, dims)
    sim.init_fields(*_fields(dims))
    for n in calls:
        monkeypatch.setenv("LBM_MULTI_STEP", mode)
        assert (sim.steps_per_launch(n) > 1) == (several and n > 1)
        sim.step(n)
    assert sim.status() == lbm.LBM_OK and sim.step_count == sum(calls)
    return sim.raw_populations().clone().view(torch.int32)


@pytest.mark.parametrize("lattice,dims,storage,several", [
    ("D2Q9", (2048, 2000), "f32", True), ("D2Q9", (1024, 1024), "f32", False), ("D2Q9", (2047, 2000), "f32", False),
    ("D2Q9", (2048, 2000), "f64", False), ("D2Q9", (4096, 2000), "bf16", False), ("D2Q9", (65536, 64), "f32", False),
    ("D3Q27", (128, 128, 90), "f32", True), ("D3Q27", (64, 64, 64), "f32", False), ("D3Q27", (129, 128, 90), "f32", False),
    ("D3Q27", (128, 128, 90), "f64", False), ("D3Q27", (128, 128, 180), "f16", False), ("D3Q27", (1024, 600, 3), "f32", False),
    ("D2Q37", (1024, 1000), "f32", False), ("E9-A", (700, 700), "f32", False)])
def test_which_grids_take_several_steps(lbm, monkeypatch, lattice, dims, storage, several):
    """FP32 storage, even nx, more populations than L2 and steps that fit into it."""
    monkeypatch.delenv("LBM_MULTI_STEP", raising=False)
    sim = _sim(lbm, lattice, dims, storage)
    assert (sim.steps_per_launch(20) > 1) == several
    assert sim.steps_per_launch(1) == 1
    if several:
        assert sim.steps_per_launch(2) == 2
        assert sim.steps_per_launch(1000) <= 32
        monkeypatch.setenv("LBM_MULTI_STEP", "0")
        assert sim.steps_per_launch(20) == 1
    if several and lattice == "D3Q27":
        monkeypatch.delenv("LBM_MULTI_STEP")
        sim.set_active_planes(1, dims[2] - 2)
        assert sim.steps_per_launch(20) == 1
        sim.set_active_planes(0, dims[2])
        assert sim.steps_per_launch(20) > 1
        sim.set_closure(torch.zeros(5894, device="cuda"), torch.cat([torch.zeros(20), torch.ones(20)]).cuda())
        assert sim.steps_per_launch(20) == 1


def test_bad_arguments(lbm):
    sim = _sim(lbm, "D2Q9", (8, 8))
    for n in (0, -1):
        with pytest.raises(lbm.LBMError) as e:
            sim.steps_per_launch(n)
        assert e.value.code == lbm.LBM_EINVAL
    assert lbm.load().lbm_steps_per_launch(None, 2) == lbm.LBM_EINVAL


# one and several tiles per plane, partial ones, planes of less than a warp, as many steps as planes; 2D runs of whole
# units and with short last ones, rows shorter and longer than a unit; odd first parities
SMALL = [((34, 17, 9), [6, 5]), ((2, 2, 5), [4, 3]), ((130, 98, 5), [1, 5]), ((64, 64, 64), [20]), ((66, 50, 40), [3, 11]),
         ((20, 18, 16), [7, 16]), ((256, 3, 7), [1, 7, 2]), ((4, 6, 3), [3]), ((2, 700), [9]), ((130, 67), [1, 9]),
         ((514, 33), [9, 4]), ((1026, 131), [12]), ((64, 4000), [1, 40]), ((366, 290), [16]), ((6, 1999), [64])]


@pytest.mark.parametrize("dims,calls", SMALL, ids=lambda v: str(v).replace(" ", ""))
def test_small_grids_give_the_bits_of_single_steps(lbm, monkeypatch, dims, calls):
    lattice = "D2Q9" if len(dims) == 2 else "D3Q27"
    a = _run(lbm, monkeypatch, lattice, dims, calls, "0", False)
    for _ in range(3):
        assert torch.equal(a, _run(lbm, monkeypatch, lattice, dims, calls, "always", True))


# calls longer than the planner's own limits; two blocks of nodes per tile, short last units, odd first parities
LARGE = [((2048, 2000), [100]), ((2050, 1990), [1, 71]), ((1366, 2901), [75]), ((64, 65535), [40]), ((4096, 1801), [1, 170]),
         ((130, 98, 101), [1, 40]), ((66, 50, 400), [45]), ((302, 202, 31), [7, 6]), ((1024, 64, 24), [1, 30]),
         ((128, 128, 128), [1, 20])]


@pytest.mark.parametrize("dims,calls", LARGE, ids=lambda v: str(v).replace(" ", ""))
def test_large_grids_give_the_bits_of_single_steps(lbm, monkeypatch, dims, calls):
    lattice = "D2Q9" if len(dims) == 2 else "D3Q27"
    a = _run(lbm, monkeypatch, lattice, dims, calls, "0", False)
    assert torch.equal(a, _run(lbm, monkeypatch, lattice, dims, calls, "1", True))
