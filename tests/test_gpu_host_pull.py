"""spmv_host where the SLICED kernel pulls x from page-locked memory while it
multiplies (half a million columns and more, rows near the diagonal): column
counts around a lane's, a warp's and a stage's share of x (2, 64 and 32768
columns) and around 64 stages, stored columns of every width, x off a 16-byte
boundary, fewer and more columns than rows, a new x in every call; and where
the copy goes first: fewer columns, x and y in one buffer.  The same row
chains as the device product: the same bits."""
import pytest
import torch

import paper_1511_02494_gb300 as sp
import synth

pytestmark = pytest.mark.gpu
HALF_M = 1 << 19


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1511_02494_gb300.build import build
    build()
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"


def _banded(rows, cols, reach, seed):
    """Up to three columns a row, within reach of the diagonal that joins the
    corners; the last row holds the last column."""
    g = torch.Generator().manual_seed(seed)
    lo = ((torch.arange(rows, dtype=torch.int64) * cols) // rows).clamp(max=cols - 1 - 2 * reach)
    ci = lo[:, None] + torch.stack([torch.zeros(rows, dtype=torch.int64), 1 + torch.randint(0, reach, (rows,), generator=g),
                                    1 + reach + torch.randint(0, reach, (rows,), generator=g)], 1)
    ci[-1, -1] = cols - 1
    keep = torch.rand((rows, 3), generator=g) < 0.9
    keep[-1, -1] = True
    rp = torch.cat([torch.zeros(1, dtype=torch.int64), keep.sum(1).cumsum(0)]).to(torch.int32)
    ci = ci[keep].to(torch.int32)
    v = torch.rand(ci.numel(), generator=g, dtype=torch.float64)
    return sp.DeviceCSR(rows, cols, rp.cuda(), ci.cuda(), v.cuda())


def _device_product(P, x):
    y = torch.empty(P.A.n_rows, dtype=torch.float64, device="cuda")
    sp.spmv(P, x.cuda(), y)
    return y.cpu()


def _same(A, shift=0, **kw):
    P = sp.spmv_prepare(A, sp.make_choice("sliced", block_nnz=1, threads_per_row=1, **kw))
    buf = torch.empty(A.n_cols + shift, dtype=torch.float64).pin_memory()
    yh = torch.empty(A.n_rows, dtype=torch.float64).pin_memory()
    for seed in range(3):
        buf[shift:] = synth.uniform_vector(A.n_cols, seed)
        yh.fill_(float("nan"))
        sp.spmv_host(P, buf[shift:], yh)
        assert torch.equal(yh, _device_product(P, buf[shift:]))
    sp.spmv_prepared_status(P)


@pytest.mark.parametrize("more", [-1, 0, 1, 2, 63, 64, 65, 32767, 32768, 32769])
def test_columns_around_the_shares(more):
    _same(_banded(10_007, HALF_M + more, 20, more + 1))


@pytest.mark.parametrize("more", [-1, 0, 1, 32769])
def test_columns_around_64_stages(more):
    _same(_banded(1_000_003, 64 * 32768 + more, 100, more + 1))


@pytest.mark.parametrize("index_bytes", [1, 2, 4])
def test_stored_columns(index_bytes):
    _same(_banded(700_001, 700_001, 20, 3), index_bytes=index_bytes)


def test_more_rows_than_columns_and_x_off_a_16_byte_boundary():
    _same(_banded(1_200_000, 600_001, 30, 4), shift=1)


def test_pageable_y():
    A = _banded(600_000, 600_000, 30, 5)
    P = sp.spmv_prepare(A, sp.make_choice("sliced", block_nnz=1, threads_per_row=1))
    x, y = synth.uniform_vector(A.n_cols, 1).pin_memory(), torch.empty(A.n_rows, dtype=torch.float64)
    sp.spmv_host(P, x, y)
    assert torch.equal(y, _device_product(P, x))


@pytest.mark.parametrize("ahead", [0, 1, 300_000])
def test_x_and_y_in_one_buffer(ahead):
    A = _banded(600_000, 600_000, 30, 6)
    P = sp.spmv_prepare(A, sp.make_choice("sliced", block_nnz=1, threads_per_row=1))
    buf = torch.empty(A.n_cols + ahead, dtype=torch.float64).pin_memory()
    x, y = buf[:A.n_cols], buf[ahead:]
    x.copy_(synth.uniform_vector(A.n_cols, 2))
    want = _device_product(P, x.clone())
    sp.spmv_host(P, x, y)
    assert torch.equal(y, want)
