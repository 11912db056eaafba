"""FP64 -> FP32 -> FP64 in integer arithmetic (the FP32 copy of x and the
widened sums): with an identity matrix in FP32 values and FP32 sums y is
float64(float32(x)) exactly, for halfway cases and their neighbours around
every kept bit, FP32's largest and smallest numbers, subnormals of both types,
infinities and random bit patterns; NaN stays NaN."""
import numpy as np
import pytest
import torch

import paper_1511_02494_gb300 as sp
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1511_02494_gb300.build import build
    build()
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"


def _values():
    g = np.random.default_rng(4)
    bits = [g.integers(0, 1 << 64, 60_000, dtype=np.uint64)]
    # float exponents and beyond, with mantissas at and beside a half of the last kept bit
    e = np.repeat(np.arange(860, 1160, dtype=np.uint64), 12)
    keep = g.integers(0, 1 << 23, e.size, dtype=np.uint64)
    drop = np.tile(np.array([0, 1, (1 << 28) - 1, 1 << 28, (1 << 28) + 1, (1 << 29) - 1], np.uint64), e.size // 6)
    bits.append((e << np.uint64(52)) | (keep << np.uint64(29)) | drop)
    bits.append((e << np.uint64(52)) | (np.uint64((1 << 23) - 1) << np.uint64(29)) | drop)   # carry into the exponent
    v = np.concatenate(bits).view(np.float64)
    f = np.finfo(np.float32)
    edge = np.array([0.0, 5e-324, 2.2e-308, float(f.max), float(f.max) * (1 + 2.0 ** -25), 3.5e38, 1e300, np.inf,
                     float(f.tiny), float(f.tiny) * (1 - 2.0 ** -26), 1.4e-45, 7e-46, 7.1e-46, np.nan, 1.0, 2.0 ** -126])
    v = np.concatenate([v, edge])
    return np.concatenate([v, -v])


@pytest.mark.parametrize("variant", ["sliced", "compressed"])
def test_rounding_is_exact(variant):
    x = _values()
    n = x.size
    A = synth.HostCSR(n, n, torch.arange(n + 1, dtype=torch.int32), torch.arange(n, dtype=torch.int32),
                      torch.ones(n, dtype=torch.float64))
    P = sp.spmv_prepare(sp.DeviceCSR.from_host(A), sp.make_choice(variant, value_type=sp.VAL_F32))
    y = torch.empty(n, dtype=torch.float64, device="cuda")
    sp.spmv(P, torch.from_numpy(x).cuda(), y)
    torch.cuda.synchronize()
    with np.errstate(over="ignore", invalid="ignore", under="ignore"):
        # the sum starts from +0, so a negative zero comes back positive
        want = x.astype(np.float32).astype(np.float64) + 0.0
    got = y.cpu().numpy()
    nan = np.isnan(want)
    assert np.array_equal(np.isnan(got), nan)
    assert np.array_equal(got[~nan], want[~nan])
