"""Several steps on a stream that may use some of the SMs only (a green context): the
launch of several steps counts on all of them, so such a stream takes single sweeps."""
import ctypes

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


@pytest.fixture(scope="module")
def small_stream():
    """A stream of a green context with 16 SMs or a few more."""
    torch.zeros(1, device="cuda")  # the primary context
    cu = ctypes.CDLL("libcuda.so.1")
    dev, n, desc, ctx, stream = (t() for t in (ctypes.c_int, ctypes.c_uint, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p))
    whole, part = ctypes.create_string_buffer(1024), ctypes.create_string_buffer(1024)
    n.value = 1
    sm_resource, default_stream, non_blocking = 1, 1, 1
    for name, *args in (
            ("cuDeviceGet", ctypes.byref(dev), 0), ("cuDeviceGetDevResource", dev, whole, sm_resource),
            ("cuDevSmResourceSplitByCount", part, ctypes.byref(n), whole, None, 0, 16),
            ("cuDevResourceGenerateDesc", ctypes.byref(desc), part, 1),
            ("cuGreenCtxCreate", ctypes.byref(ctx), desc, dev, default_stream),
            ("cuGreenCtxStreamCreate", ctypes.byref(stream), ctx, non_blocking, 0)):
        rc = getattr(cu, name)(*args)
        if rc:
            pytest.skip("%s: error %d" % (name, rc))
    yield torch.cuda.ExternalStream(stream.value)
    torch.cuda.synchronize()
    cu.cuStreamDestroy_v2(stream)
    cu.cuGreenCtxDestroy(ctx)


@pytest.mark.parametrize("lattice,dims", [("D2Q9", (2048, 2000)), ("D3Q27", (128, 128, 90))])
def test_a_stream_with_few_sms_takes_the_same_steps(lbm, small_stream, lattice, dims):
    D, N = len(dims), 1
    for d in dims:
        N *= d
    g = torch.Generator(device="cuda").manual_seed(11)
    rho = 1.0 + 0.02 * (torch.rand(N, generator=g, device="cuda", dtype=torch.float64) - 0.5)
    u = 0.05 * (torch.rand(D, N, generator=g, device="cuda", dtype=torch.float64) - 0.5)
    out = []
    for stream in (None, small_stream):
        torch.cuda.synchronize()
        sim = lbm.Simulation(lattice, dims, [0.7, 1.0, 0.7, 1.0, 0.7][:3 if D == 2 else 5], storage="f32", stream=stream)
        assert (sim.steps_per_launch(7) > 1) == (stream is None)
        sim.init_fields(rho, u)
        sim.step(7)
        assert sim.status() == lbm.LBM_OK and sim.step_count == 7
        out.append(sim.raw_populations().clone().view(torch.int32))
    assert torch.equal(*out)
