"""Odd nx: a grid's size decides between one node and two nodes of a column per
thread; the populations do not depend on it, bit for bit."""
import numpy as np
import pytest

from paper_1808_04406_gb300 import inputs, slab

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def lbm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1808_04406_gb300 import build as libbuild
    libbuild.build()
    from paper_1808_04406_gb300 import lbm as L
    L.load()
    return L


def _bits(a):
    return a.reshape(a.shape[0], -1).view({2: torch.int16, 4: torch.int32, 8: torch.int64}[a.element_size()])


@pytest.mark.parametrize("storage", ["f64", "f32", "f16", "bf16"])
@pytest.mark.parametrize("lattice,dims,copies", [("D2Q9", (613, 8), 32), ("D2Q9", (1023, 6), 50), ("D3Q27", (97, 64, 4), 8),
                                                 ("D3Q27", (99, 63, 3), 11), ("D3Q27", (31, 31, 5), 40)])
def test_copies_of_a_small_grid_evolve_as_it_does(lbm, lattice, dims, copies, storage):
    """A grid of copies along its last axis takes another kernel than one copy (from 608
    blocks of column pairs on) and holds one copy's populations in each, both parities."""
    D = len(dims)
    rho, u = inputs.random_noise(dims, seed=19, du=0.08, drho=0.02)
    taus = [0.6, 0.9, 0.7, 1.1, 0.8][:3 if D == 2 else 5]
    one = lbm.Simulation(lattice, dims, taus, storage=storage)
    many = lbm.Simulation(lattice, dims[:-1] + (dims[-1] * copies,), taus, storage=storage)
    if storage != "f64" and (D, storage) != (2, "f32"):
        assert (one.sweep_kernel(), many.sweep_kernel()) == ("tp_sweep_kernel", "tp_column_kernel")
    one.init_fields(rho, u)
    many.init_fields(np.tile(rho, copies), np.tile(u, (1, copies)))
    for n in (1, 1, 9):
        one.step(n)
        many.step(n)
        assert torch.equal(_bits(one.raw_populations()).tile(1, copies), _bits(many.raw_populations()))
    assert one.status() == many.status() == lbm.LBM_OK


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("dims,world", [((97, 64, 31), 2), ((97, 64, 31), 3), ((99, 63, 26), 2)])
def test_slabs_below_the_switch_equal_the_whole_grid_above_it(lbm, dims, world, storage):
    """A grid of 608 blocks of column pairs or more, cut into slabs that have fewer and
    so take one node per thread: the owned populations are the whole grid's."""
    taus = [0.53, 1.0, 0.53, 1.0, 0.53]
    rho, u = inputs.random_noise(dims, seed=23, du=0.05, drho=0.02)
    whole = lbm.Simulation("D3Q27", dims, taus, storage=storage)
    whole.init_fields(rho, u)
    runs = [slab.SlabRun.create(dims, taus, storage, r, world) for r in range(world)]
    assert whole.sweep_kernel() == "tp_column_kernel" and all(r.sim.sweep_kernel() == "tp_sweep_kernel" for r in runs)
    for run in runs:
        run.sim.init_fields(*run.local_fields(rho, u))
    group = slab.LocalGroup(runs)
    for n in (2, 5):
        whole.step(n)
        group.step(n)
        group.refresh_ghosts()  # odd parity: boundary nodes read populations from the ghost planes
        f = whole.populations().reshape(27, dims[2], -1)
        for run in runs:
            own = run.owned(run.sim.populations(), 27).reshape(27, run.nzl, -1)
            np.testing.assert_array_equal(own, f[:, run.z0:run.z0 + run.nzl])
    assert whole.status() == lbm.LBM_OK
