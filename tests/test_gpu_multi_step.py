"""Several steps per launch: the same bits as one launch per step.

The multi-step kernel runs a sweep's node arithmetic in another order of nodes, so
its populations equal those of single-step launches exactly, for every storage
type, row length, unit and tile remainder, parity and number of steps."""
import numpy as np
import pytest

from paper_1808_04406_gb300 import inputs

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


def _populations(lbm, monkeypatch, lattice, dims, storage, calls, multi):
    monkeypatch.setenv("LBM_MULTI_STEP", "1" if multi else "0")
    D = len(dims)
    g = torch.Generator(device="cuda").manual_seed(7)
    N = int(np.prod(dims))
    rho = 1.0 + 0.02 * (torch.rand(N, generator=g, device="cuda", dtype=torch.float64) - 0.5)
    u = 0.05 * (torch.rand(D, N, generator=g, device="cuda", dtype=torch.float64) - 0.5)
    taus = [0.7, 1.0, 0.7] if D == 2 else [0.7, 1.0, 0.7, 1.0, 0.7]
    if lattice.startswith("E"):
        sim = lbm.HermiteSimulation(lattice, dims, taus, storage=storage, flags=lbm.LBM_THERMAL)
    else:
        sim = lbm.Simulation(lattice, dims, taus, storage=storage, flags=lbm.LBM_THERMAL if lattice == "D2Q37" else 0)
    sim.init_fields(rho, u)
    for n in calls:
        sim.step(n)
    assert sim.status() == lbm.LBM_OK and sim.step_count == sum(calls)
    return sim.raw_populations().clone().view(torch.int16 if storage in ("f16", "bf16") else
                                              torch.int32 if storage == "f32" else torch.int64)


# FP32 grids larger than L2 take several steps per launch: planes of whole and of partial blocks, odd first
# parities, numbers of steps that the passes divide and do not, 2D runs with and without a short last unit; smaller
# grids, other storage types and odd nx take one
CASES = [
    ("D2Q9", (3, 3), "f64", [2, 3]), ("D2Q9", (128, 128), "f64", [7, 2]), ("D2Q9", (130, 67), "f32", [5, 4]),
    ("D2Q9", (131, 67), "f32", [5, 4]), ("D2Q9", (2, 700), "f32", [4]), ("D2Q9", (1, 389), "f64", [3]),
    ("D2Q9", (514, 33), "bf16", [6, 5]), ("D2Q9", (1026, 31), "f16", [9]), ("D2Q9", (255, 130), "f16", [9]),
    ("D3Q27", (3, 3, 3), "f32", [2, 5]), ("D3Q27", (2, 2, 5), "f32", [4, 3]), ("D3Q27", (34, 17, 9), "f32", [5, 6]),
    ("D3Q27", (33, 17, 9), "f32", [5, 6]), ("D3Q27", (34, 17, 9), "f16", [7]), ("D3Q27", (33, 17, 9), "bf16", [4]),
    ("D3Q27", (20, 18, 16), "f64", [5]), ("D3Q27", (64, 64, 64), "f32", [20]), ("D3Q27", (1, 1, 4), "f64", [3]),
    ("D3Q27", (128, 128, 90), "f32", [1, 20]), ("D3Q27", (130, 101, 150), "f16", [13]),
    ("D3Q27", (161, 95, 77), "f32", [3, 10]), ("D3Q27", (96, 64, 100), "f64", [9]), ("D2Q9", (2050, 1300), "f64", [1, 40]),
    ("D2Q9", (2048, 2000), "f32", [37]), ("D2Q9", (1366, 2901), "f32", [1, 9]), ("D2Q9", (4096, 1801), "f32", [8]),
    ("D3Q27", (130, 98, 101), "f32", [2, 3, 4]), ("D3Q27", (302, 202, 31), "f32", [7]), ("D3Q27", (66, 50, 400), "f32", [11]),
    ("D3Q27", (1024, 600, 3), "f32", [4]), ("D2Q9", (65536, 64), "f32", [6]),
    # velocities that reach three rows: units of 3 and 4 rows, short and long rows, too few rows (single steps)
    ("D2Q37", (128, 128), "f32", [1, 20]), ("D2Q37", (31, 29), "f32", [9]), ("D2Q37", (512, 100), "f32", [9, 8]),
    ("D2Q37", (40, 31), "f64", [9, 10]), ("D2Q37", (5, 41), "f64", [12]), ("D2Q37", (6, 8), "f64", [12]),
    ("D2Q37", (1024, 250), "f16", [1, 10]), ("D2Q37", (130, 64), "bf16", [9]),
    ("E9-A", (80, 80), "f64", [41, 2]), ("E9-C", (33, 20), "f64", [5, 6]), ("E7-A", (47, 31), "f64", [7]),
    ("E7-D", (20, 23), "f32", [7, 4]), ("E9-B", (40, 43), "f32", [6]),
]


@pytest.mark.parametrize("lattice,dims,storage,calls", CASES, ids=lambda v: str(v).replace(" ", ""))
def test_multi_step_launches_match_single_steps_bit_for_bit(lbm, monkeypatch, lattice, dims, storage, calls):
    a = _populations(lbm, monkeypatch, lattice, dims, storage, calls, False)
    b = _populations(lbm, monkeypatch, lattice, dims, storage, calls, True)
    assert torch.equal(a, b)
