"""SLICED prepare at the edges of its kernels, bit-exact against the oracle:
sort windows whose lengths need one to four 5-bit digits, windows of every
size with a partial last one, more than 1024 slice tiles with long rows in
several of them, slice lengths around the fill's chunks of 8 and the
four-element groups of the low-precision form."""
import numpy as np
import pytest
import torch

import oracle
import paper_1511_02494_gb300 as sp
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1511_02494_gb300.build import build
    build()
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"


def _matrix(lengths, seed):
    """Rows of the given lengths: runs of consecutive columns at random places."""
    lengths = np.asarray(lengths, np.int64)
    g = np.random.default_rng(seed)
    n_cols = int(lengths.max()) + 70_000
    rp = np.concatenate([[0], np.cumsum(lengths)])
    start = g.integers(0, n_cols - lengths + 1)
    rows = np.repeat(np.arange(lengths.size), lengths)
    ci = start[rows] + np.arange(rp[-1]) - rp[:-1][rows]
    return synth.HostCSR(lengths.size, n_cols, torch.from_numpy(rp.astype(np.int32)),
                         torch.from_numpy(ci.astype(np.int32)), torch.from_numpy(g.uniform(-1, 1, int(rp[-1]))))


def _export(P, which, n, dtype):
    out = torch.empty(n, dtype=dtype)
    sp.spmv_prepared_export(P, which, out)
    return out.numpy()


def _check(A, sigma, cap, vt=sp.VAL_F64):
    vec = 1 if vt == sp.VAL_F64 else 4
    dA = sp.DeviceCSR.from_host(A)
    P = sp.spmv_prepare(dA, sp.make_choice("sliced", block_nnz=sigma, items_per_warp=cap, value_type=vt))
    perm, rowlen, slen, sptr, n_long = oracle.sliced_layout(A, sigma, cap, vec=vec)
    S, tot = (A.n_rows + 31) // 32, int(sptr[-1])
    assert P.info().n_long_rows == n_long
    assert np.array_equal(_export(P, sp.EXPORT_SLICE_ROWLEN, 32 * S, torch.int32), rowlen)
    assert np.array_equal(_export(P, sp.EXPORT_SLICE_LEN, S, torch.int32), slen)
    assert np.array_equal(_export(P, sp.EXPORT_SLICE_PTR, S + 1, torch.int64), sptr)
    if sigma > 1:
        assert np.array_equal(_export(P, sp.EXPORT_SLICE_PERM, A.n_rows, torch.int32), perm)
    if tot:
        col, val = oracle.sliced_fill(A, perm, rowlen, sptr, vec=vec)
        if vt == sp.VAL_F64:
            if P.info().index_bytes == 4:
                assert np.array_equal(_export(P, sp.EXPORT_SLICE_COL, tot, torch.int32), col)
            assert np.array_equal(_export(P, sp.EXPORT_SLICE_VAL, tot, torch.float64), val)
        else:
            assert np.array_equal(_export(P, sp.EXPORT_SLICE_VAL, tot, torch.float32), val.astype(np.float32))
    if n_long:
        lst, off, be, srow, fix, sfix = oracle.sliced_segments(A, cap, 2048)
        assert np.array_equal(_export(P, sp.EXPORT_SLICE_LONG, len(lst), torch.int32), lst)
        assert np.array_equal(_export(P, sp.EXPORT_SLICE_SEG_OFF, len(lst) + 1, torch.int32), off)
        assert np.array_equal(_export(P, sp.EXPORT_SLICE_SEG_BOUNDS, 2 * len(srow), torch.int64), be.reshape(-1))
        assert np.array_equal(_export(P, sp.EXPORT_SLICE_SEG_ROW, len(srow), torch.int32), srow)
        assert np.array_equal(_export(P, sp.EXPORT_SLICE_FIX, len(fix), torch.int32), fix)
        if vt == sp.VAL_F64:
            assert np.array_equal(_export(P, sp.EXPORT_SLICE_SEG_FIX, len(sfix), torch.int32), sfix)
    # the same product, ticketed rows included, twice
    x = synth.uniform_vector(A.n_cols, 3)
    y_ref, scale = oracle.spmv_ref(A, x)
    for _ in range(2):
        y = torch.full((A.n_rows,), float("nan"), dtype=torch.float64, device="cuda")
        sp.spmv(P, x.cuda(), y)
        torch.cuda.synchronize()
        tol = 1e-12 if vt == sp.VAL_F64 else 1e-6   # FP32 values and sums of at most 2^13 terms
        assert np.all(np.abs(y.cpu().numpy() - y_ref) <= tol * scale)
    P.free()


@pytest.mark.parametrize("sigma", [32, 64, 128, 1024, 4096])
@pytest.mark.parametrize("top,cap", [(1, 1024), (30, 1024), (31, 1024), (40, 32), (1100, 1024), (40_000, 65536)])
def test_sort_digits_and_windows(sigma, top, cap):
    # lengths 0..top, log-uniform above 2000 so that the matrix stays small
    g = np.random.default_rng(sigma + top)
    n = 4096 + 1000 + 17                           # a partial last window and slice
    lengths = g.integers(0, top + 1, n) if top < 2000 else \
        np.floor(np.exp(g.uniform(0, np.log(top), 600))).astype(np.int64)
    lengths[-1] = top
    if top == 1100:
        lengths = lengths // 4
        lengths[::97] = top
    _check(_matrix(lengths, seed=top), sigma, cap)


@pytest.mark.parametrize("vt", [sp.VAL_F64, sp.VAL_F32])
@pytest.mark.parametrize("length", [1, 3, 7, 8, 9, 15, 16, 17, 31, 33])
def test_fill_chunks(length, vt):
    # the slice's longest row is `length`, others shorter, one empty
    lengths = [length - (i % 3) * (i % 2) if i % 11 else 0 for i in range(101)]
    lengths = np.maximum(lengths, 0)
    lengths[5] = length
    _check(_matrix(lengths, seed=length), 1, 1024, vt)
    _check(_matrix(lengths, seed=length), 32, 1024, vt)


@pytest.mark.parametrize("sigma", [1, 4096])
def test_many_tiles(sigma):
    n = 1024 * 32 * 32 + 12_345                    # tiles of more than one unit
    lengths = np.full(n, 2, np.int64)
    lengths[np.arange(0, n, 50_021)] = 40
    lengths[[0, 77_777, n // 2, n - 1]] = [2049, 5000, 2048, 4097]
    _check(_matrix(lengths, seed=sigma), sigma, 32)
