"""A call of several steps per launch in a CUDA graph: every replay advances the
populations as the call itself does."""
import numpy as np
import pytest

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


@pytest.mark.parametrize("dims", [(2048, 2000), (128, 128, 90), (64, 64, 64)])
def test_replays_of_a_captured_call_are_calls(lbm, dims):
    D, N = len(dims), int(np.prod(dims))
    g = torch.Generator(device="cuda").manual_seed(5)
    rho = 1.0 + 0.02 * (torch.rand(N, generator=g, device="cuda", dtype=torch.float64) - 0.5)
    u = 0.05 * (torch.rand(D, N, generator=g, device="cuda", dtype=torch.float64) - 0.5)
    torch.cuda.synchronize()
    stream = torch.cuda.Stream()
    out = []
    for captured in (False, True):
        sim = lbm.Simulation("D2Q9" if D == 2 else "D3Q27", dims, [0.7, 1.0, 0.7, 1.0, 0.7][:2 * D - 1], storage="f32",
                             stream=stream)
        sim.init_fields(rho, u)
        stream.synchronize()
        if captured:
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=stream):
                sim.step(6)  # even: every replay starts from the same parity
            for _ in range(3):
                graph.replay()
        else:
            for _ in range(3):
                sim.step(6)
        torch.cuda.synchronize()
        assert sim.status() == lbm.LBM_OK
        out.append(sim.raw_populations().clone().view(torch.int32))
    assert torch.equal(*out)
