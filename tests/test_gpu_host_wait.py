"""spmv_host's wait for x runs out (a part of x that nobody copies, a limit of
a millisecond): the call says so and y is right all the same, and so is the
next call's; and which calls take the kernel that waits: page-locked x apart
from y, half a million columns and more, rows in order and near the diagonal,
FP64 values with plain columns, no long rows."""
import pytest
import torch

import paper_1511_02494_gb300 as sp
import synth

pytestmark = pytest.mark.gpu
HALF_M = 1 << 19
LIMIT = 1_000_000


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1511_02494_gb300.build import build
    build()
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"


def _band(n, width=3, first=0):
    """Columns row + first .. row + first + width - 1, those inside."""
    c = torch.arange(n)[:, None] + first + torch.arange(width)
    keep = (c >= 0) & (c < n)
    rp = torch.cat([torch.zeros(1, dtype=torch.int64), keep.sum(1).cumsum(0)]).to(torch.int32)
    ci = c[keep].to(torch.int32)
    v = torch.rand(ci.numel(), generator=torch.Generator().manual_seed(7), dtype=torch.float64)
    return sp.DeviceCSR(n, n, rp.cuda(), ci.cuda(), v.cuda())


def _host(n, seed=1):
    return synth.uniform_vector(n, seed).pin_memory(), torch.full((n,), float("nan"), dtype=torch.float64).pin_memory()


def _product(P, x):
    y = torch.empty(P.A.n_rows, dtype=torch.float64, device="cuda")
    sp.spmv(P, x.cuda(), y)
    return y.cpu()


def _prepare(A, **kw):
    return sp.spmv_prepare(A, sp.make_choice("sliced", **{"block_nnz": 1, "threads_per_row": 1, **kw}))


@pytest.mark.parametrize("pinned_y", [True, False])
@pytest.mark.parametrize("index_bytes", [1, 4])
@pytest.mark.parametrize("n", [HALF_M, 64 * 32768 + 1])
def test_a_wait_that_gives_up_leaves_the_right_y(n, index_bytes, pinned_y):
    P = _prepare(_band(n), index_bytes=index_bytes)
    for seed in (1, 2):                                  # the staging vector holds the other x by then
        x, y = _host(n, seed)
        if not pinned_y:
            y = torch.full((n,), float("nan"), dtype=torch.float64)
        want = _product(P, x)
        assert sp.spmv_host_wait_check(P, x, y, LIMIT, arrive=False)
        assert torch.equal(y, want)
        y.fill_(float("nan"))
        assert not sp.spmv_host_wait_check(P, x, y, 2_000_000_000, arrive=True)
        assert torch.equal(y, want)
        y.fill_(float("nan"))
        sp.spmv_host(P, x, y)
        assert torch.equal(y, want)


def _long_row():
    A = _band(HALF_M)
    rp = A.rowptr.clone()
    rp[1:] += 2000 - 3
    ci = torch.cat([torch.arange(2000, dtype=torch.int32, device="cuda"), A.colind[3:]])
    return sp.DeviceCSR(HALF_M, HALF_M, rp, ci, torch.ones(ci.numel(), dtype=torch.float64, device="cuda"))


TAKES_THE_COPY = {
    "fewer columns": lambda: _prepare(_band(HALF_M - 1)),
    "rows far ahead": lambda: _prepare(_band(HALF_M, first=HALF_M // 4 + 64)),
    "sorted": lambda: _prepare(_band(HALF_M), block_nnz=64),
    "long rows": lambda: _prepare(_long_row()),
    "deltas": lambda: _prepare(_band(HALF_M), index_coding=1),
    "FP32 values": lambda: _prepare(_band(HALF_M), value_type=sp.VAL_F32),
    "four slices a warp": lambda: _prepare(_band(HALF_M), threads_per_row=4),
    "subwarp": lambda: sp.spmv_prepare(_band(HALF_M), sp.make_choice("subwarp")),
}


@pytest.mark.parametrize("form", TAKES_THE_COPY)
def test_forms_that_copy_x_first(form):
    P = TAKES_THE_COPY[form]()
    x, y = _host(P.A.n_rows)
    with pytest.raises(sp.SpmvError, match="does not wait"):
        sp.spmv_host_wait_check(P, x, y, LIMIT, arrive=False)
    assert torch.equal(y, _product(P, x))


@pytest.mark.parametrize("memory", ["pageable x", "x is y", "x overlaps y"])
def test_vectors_that_are_copied_first(memory):
    P = _prepare(_band(HALF_M))
    x, y = _host(HALF_M)
    if memory == "pageable x":
        x = x.clone()
    elif memory == "x is y":
        y = x
    else:
        buf = torch.empty(HALF_M + 1000, dtype=torch.float64).pin_memory()
        buf[:HALF_M] = x
        x, y = buf[:HALF_M], buf[1000:]
    want = _product(P, x.clone())
    with pytest.raises(sp.SpmvError, match="does not wait"):
        sp.spmv_host_wait_check(P, x, y, LIMIT, arrive=False)
    assert torch.equal(y, want)


@pytest.mark.parametrize("limit", [0, -1, 2_000_000_001])
def test_limits_out_of_range(limit):
    P = _prepare(_band(HALF_M))
    x, y = _host(HALF_M)
    with pytest.raises(sp.SpmvError, match="limit_ns"):
        sp.spmv_host_wait_check(P, x, y, limit, arrive=True)


@pytest.mark.parametrize("pieces", [1, 2])
def test_registered_vectors(pieces):
    """Memory of the caller's own that it registered, as a whole or in two parts
    end to end, is used in place."""
    P = _prepare(_band(HALF_M))
    raw = torch.zeros(8 * HALF_M + 4096, dtype=torch.uint8)
    at = -raw.data_ptr() % 4096
    x = raw[at:at + 8 * HALF_M].view(torch.float64)
    x.copy_(synth.uniform_vector(HALF_M, 5))
    y = torch.empty(HALF_M, dtype=torch.float64).pin_memory()
    want = _product(P, x)
    rt, size = torch.cuda.cudart(), 8 * HALF_M // pieces
    starts = [x.data_ptr() + i * size for i in range(pieces)]
    for p in starts:
        assert int(rt.cudaHostRegister(p, size, 0)) == 0
    try:
        assert not sp.spmv_host_wait_check(P, x, y, 2_000_000_000, arrive=True)
        assert torch.equal(y, want)
    finally:
        for p in starts:
            rt.cudaHostUnregister(p)
