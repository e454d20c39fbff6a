"""The bounded waits of the launch of several steps: one that runs out on purpose is
reported and leaves the context usable, and a timeout reported earlier does not end a
later launch's waits."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

TAUS = {2: [0.7, 1.0, 0.7], 3: [0.7, 1.0, 0.7, 1.0, 0.7]}
GRIDS = [("D2Q9", (514, 130)), ("D3Q27", (66, 50, 40)), ("D3Q27", (128, 128, 90))]


@pytest.fixture(scope="module")
def lbm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1808_04406_gb300 import build as libbuild
    libbuild.build()
    from paper_1808_04406_gb300 import lbm as L
    L.load()
    return L


def _sim(lbm, lattice, dims):
    g = torch.Generator(device="cuda").manual_seed(3)
    N, D = int(np.prod(dims)), len(dims)
    sim = lbm.Simulation(lattice, dims, TAUS[D], storage="f32")
    fields = (1.0 + 0.02 * (torch.rand(N, generator=g, device="cuda", dtype=torch.float64) - 0.5),
              0.05 * (torch.rand(D, N, generator=g, device="cuda", dtype=torch.float64) - 0.5))
    sim.init_fields(*fields)
    return sim, fields


@pytest.mark.parametrize("polls", [1, 3000])
@pytest.mark.parametrize("lattice,dims", GRIDS)
def test_a_wait_that_runs_out_is_reported(lbm, monkeypatch, lattice, dims, polls):
    monkeypatch.setenv("LBM_MULTI_STEP", "always")
    sim, fields = _sim(lbm, lattice, dims)
    assert sim.steps_per_launch(6) > 1
    sim.step(6)
    assert sim.status() == lbm.LBM_OK
    want = sim.raw_populations().clone()
    lbm.lbm_selftest_steps_timeout(sim.handle, 6, polls)
    assert sim.status() == lbm.LBM_ETIMEOUT and sim.step_count == 6
    assert b"gave up" in lbm.load().lbm_last_error()
    sim.init_fields(*fields)
    sim.step(6)
    assert sim.status() == lbm.LBM_OK
    assert torch.equal(want.view(torch.int32), sim.raw_populations().view(torch.int32))


@pytest.mark.parametrize("lattice,dims", GRIDS)
def test_an_earlier_timeout_does_not_end_later_launches(lbm, monkeypatch, lattice, dims):
    out = []
    for mode in ("0", "always"):
        monkeypatch.setenv("LBM_MULTI_STEP", mode)
        sim, _ = _sim(lbm, lattice, dims)
        lbm.lbm_selftest_wait_timeout(sim.handle, 1)  # leaves the timeout bit in the status word
        sim.step(24)
        assert sim.status() == lbm.LBM_ETIMEOUT
        out.append(sim.raw_populations().clone().view(torch.int32))
    assert torch.equal(*out)


def test_bad_arguments(lbm, monkeypatch):
    monkeypatch.delenv("LBM_MULTI_STEP", raising=False)
    sim, _ = _sim(lbm, "D2Q9", (8, 8))
    for n, polls in ((6, 0), (6, (1 << 20) + 1), (1, 10), (6, 10), (-1, 10)):  # one step per launch on 8 x 8
        with pytest.raises(lbm.LBMError) as e:
            lbm.lbm_selftest_steps_timeout(sim.handle, n, polls)
        assert e.value.code == lbm.LBM_EINVAL
    assert sim.status() == lbm.LBM_OK
    assert lbm.load().lbm_selftest_steps_timeout(None, 6, 10) == lbm.LBM_EINVAL
