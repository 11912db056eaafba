"""Long rows of one tile are listed together: tiles of nothing but long rows,
one long row at each place of a tile, rows of one and of many pieces side by
side, against the oracle; and a rowptr whose rows overlap, so that the tile
lists more rows and pieces than a valid matrix could: refused, and the next
matrix is right."""
import numpy as np
import pytest
import torch

import oracle
import paper_1511_02494_gb300 as sp
import synth

pytestmark = pytest.mark.gpu
KEYS = ("nnz_min", "nnz_max", "nnz_sum", "nnz_sumsq", "bw_min", "bw_max", "bw_sum", "bw_sumsq", "disp_sum",
        "disp_sumsq", "clust_sum", "ngroups_sum", "misses_sum")


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1511_02494_gb300.build import build
    build()
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"


def _matrix(lengths, n_cols=60_000):
    """Row i: every third column from i % 7 on, so many of them."""
    rows = [(i % 7) + 3 * np.arange(n) for i, n in enumerate(lengths)]
    rp = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int32)
    ci = np.concatenate(rows + [np.zeros(0, np.int64)]).astype(np.int32)
    return synth.HostCSR(len(lengths), n_cols, torch.from_numpy(rp), torch.from_numpy(ci),
                         torch.ones(ci.size, dtype=torch.float64), "listing")


def _check(A):
    dA = sp.DeviceCSR.from_host(A)
    sp.spmv_validate(dA)
    o = oracle.features(A, line_bytes=128, l2_bytes=torch.cuda.get_device_properties(0).L2_cache_size)
    for _ in range(2):
        g = sp.spmv_features(dA, 128).as_dict()
        assert {k: g[k] for k in KEYS} == {k: o[k] for k in KEYS}


@pytest.mark.parametrize("lengths", [
    [1025] * 32, [1025] * 33, [1100] * 200, [19_000] * 3, [2048, 2049, 4096, 4097, 1025] * 13,
    [1025, 17_000] * 16, [0, 1025] * 32, [3] * 40 + [18_000] + [1025] * 31],
    ids=lambda v: f"{len(v)}x{v[0]}")
def test_tiles_of_long_rows(lengths):
    _check(_matrix(lengths))


def test_one_long_row_at_every_place_of_a_tile():
    lengths = []
    for at in range(32):
        lengths += [2] * at + [1025 + 300 * at] + [1] * (31 - at)
    _check(_matrix(lengths))


@pytest.mark.parametrize("n_rows", [64, 1000])
def test_overlapping_rows_are_refused(n_rows):
    nnz = 5000
    rp = torch.tensor([0, nnz] * (n_rows // 2) + [nnz], dtype=torch.int32)   # every other row holds all of it
    ci, v = torch.arange(nnz, dtype=torch.int32), torch.ones(nnz, dtype=torch.float64)
    bad = sp.DeviceCSR(n_rows, nnz, rp.cuda(), ci.cuda(), v.cuda())
    for _ in range(2):
        with pytest.raises(sp.SpmvError, match="rowptr decreasing"):
            sp.spmv_features(bad)
        with pytest.raises(sp.SpmvError, match="rowptr decreasing"):
            sp.spmv_prepare(bad, sp.make_choice("sliced"))
        _check(_matrix([1025] * 40))
