"""The 37-velocity sweeps that compute in plain FP32 (16-bit storage, FP32 with
LBM_FAST_TRANSFORMS) keep their bits.

Their collision is the one on Hermite tables, whose transforms drift half as fast
as plain FP32 sums of raw moments; the values below are digests of what it gave
when it was the only one (populations of both parities, and the totals)."""
import hashlib

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


def _noise(n, salt):
    """Multiples of 2^-12 in [-1/2, 1/2): the same numbers on every machine."""
    k = (np.arange(n, dtype=np.uint64) * np.uint64(2654435761) + np.uint64(salt * 40503)) & np.uint64(0xffffffff)
    return ((k ^ (k >> np.uint64(15))) >> np.uint64(4) & np.uint64(4095)).astype(np.float64) / 4096 - 0.5


def digests(lbm, dims, storage, flag):
    flags = sum(getattr(lbm, "LBM_" + name) for name in flag.split("+") if name)
    n = int(np.prod(dims))
    sim = lbm.Simulation("D2Q37", dims, [0.5625, 0.6875, 0.5625], storage=storage, flags=flags, theta_ref=1.25)
    theta = 1.25 + _noise(n, 4) / 32 if "THERMAL" in flag else np.ones(n)
    sim.init_fields(1 + _noise(n, 1) / 32, np.stack([_noise(n, 2), _noise(n, 3)]) / 16, theta)
    sim.step(3)
    totals = [sim.step_totals(), sim.step_totals()]
    sim.step(1)
    assert sim.status() == lbm.LBM_OK
    raw = sim.raw_populations().cpu().view(torch.int32 if storage == "f32" else torch.int16).numpy()
    return tuple(hashlib.sha256(np.ascontiguousarray(a).tobytes()).hexdigest()[:12]
                 for a in (raw, np.array(totals, dtype=np.float64)))


# even nx: two nodes per thread; odd nx: one
CASES = [(dims, storage, flag) for dims in ((40, 12), (41, 11), (301, 220)) for storage, flag in (
    ("f16", "THERMAL"), ("f16", ""), ("f16", "THERMAL+K72"), ("f16", "THERMAL+RAW_MRT"),
    ("f16", "THERMAL+STOCHASTIC_ROUND"), ("bf16", "THERMAL"), ("bf16", "THERMAL+STOCHASTIC_ROUND"),
    ("f32", "THERMAL+FAST_TRANSFORMS"), ("f32", "FAST_TRANSFORMS"))]
WANT = {
    ((40, 12), 'f16', 'THERMAL'): ('fb7a5beb13e0', '8948685c3566'),
    ((40, 12), 'f16', ''): ('ad34e0b20af2', '4259bf3506d8'),
    ((40, 12), 'f16', 'THERMAL+K72'): ('fb7a5beb13e0', '8948685c3566'),
    ((40, 12), 'f16', 'THERMAL+RAW_MRT'): ('8fa8e8be6bac', 'ebda9752eeaf'),
    ((40, 12), 'f16', 'THERMAL+STOCHASTIC_ROUND'): ('fbf7d8bb7187', '6a965130bd75'),
    ((40, 12), 'bf16', 'THERMAL'): ('ef5cb5eb7068', '31a506e52656'),
    ((40, 12), 'bf16', 'THERMAL+STOCHASTIC_ROUND'): ('9ccb6cf247a3', '72e55402b6d5'),
    ((40, 12), 'f32', 'THERMAL+FAST_TRANSFORMS'): ('89f50e6a2e56', 'fd64182420d8'),
    ((40, 12), 'f32', 'FAST_TRANSFORMS'): ('3d0562c52c4c', 'fecd5f55087c'),
    ((41, 11), 'f16', 'THERMAL'): ('9ac4af3afbb2', '67f414fd911f'),
    ((41, 11), 'f16', ''): ('1442e7ce1a82', 'd479b23b00e8'),
    ((41, 11), 'f16', 'THERMAL+K72'): ('9ac4af3afbb2', '67f414fd911f'),
    ((41, 11), 'f16', 'THERMAL+RAW_MRT'): ('916a5733faf3', '4fd7d368c588'),
    ((41, 11), 'f16', 'THERMAL+STOCHASTIC_ROUND'): ('de3101c9a5d9', '2a59a4f4ca28'),
    ((41, 11), 'bf16', 'THERMAL'): ('989ccea4a795', '6fadd6010fe0'),
    ((41, 11), 'bf16', 'THERMAL+STOCHASTIC_ROUND'): ('15dc3f7efb16', '81033103c93e'),
    ((41, 11), 'f32', 'THERMAL+FAST_TRANSFORMS'): ('a47da358ea23', 'bb0d8fde44b8'),
    ((41, 11), 'f32', 'FAST_TRANSFORMS'): ('759d95405af7', '48b930aa24a4'),
    ((301, 220), 'f16', 'THERMAL'): ('798af7f2a38d', '2ca370376879'),
    ((301, 220), 'f16', ''): ('1bd0bee749d9', '9d5a46fa8fd5'),
    ((301, 220), 'f16', 'THERMAL+K72'): ('798af7f2a38d', '2ca370376879'),
    ((301, 220), 'f16', 'THERMAL+RAW_MRT'): ('b9428963fee3', '1a44d5920dda'),
    ((301, 220), 'f16', 'THERMAL+STOCHASTIC_ROUND'): ('0cb91ab7941c', 'dca2cf8bc765'),
    ((301, 220), 'bf16', 'THERMAL'): ('1a58373983d4', 'a687f6d3472b'),
    ((301, 220), 'bf16', 'THERMAL+STOCHASTIC_ROUND'): ('f0b89fa7366a', '98f7a8204640'),
    ((301, 220), 'f32', 'THERMAL+FAST_TRANSFORMS'): ('4ed9739df2b6', 'e38d6946455b'),
    ((301, 220), 'f32', 'FAST_TRANSFORMS'): ('342d4fbb6033', '0ed3add794ea'),
}


@pytest.mark.parametrize("dims,storage,flag", CASES, ids=lambda v: str(v).replace(" ", ""))
def test_plain_fp32_sweeps_keep_their_bits(lbm, dims, storage, flag):
    assert digests(lbm, dims, storage, flag) == WANT[(dims, storage, flag)]
