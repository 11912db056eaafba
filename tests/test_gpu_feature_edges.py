"""Feature pass at the edges of its split: rows around a 32-element step, the
1024-element batch and the row length (1024) above which a row is cut into
2048-element pieces, tiles whose rows start anywhere in a batch, and tiles
where long and short rows alternate.  Integer aggregates: bit-exact with the
oracle."""
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


def _matrix(lengths, n_cols, seed):
    g = np.random.default_rng(seed)
    rows = []
    for n in lengths:
        if n and g.random() < 0.3:                 # a run of consecutive columns
            a = g.integers(0, n_cols - n + 1)
            rows.append(np.arange(a, a + n))
        else:
            rows.append(np.sort(g.choice(n_cols, n, replace=False)))
    rp = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int32)
    ci = np.concatenate(rows + [np.zeros(0, np.int64)]).astype(np.int32)
    return synth.HostCSR(len(lengths), n_cols, torch.from_numpy(rp), torch.from_numpy(ci),
                         torch.ones(ci.size, dtype=torch.float64), "edges")


EDGES = [0, 1, 2, 31, 32, 33, 1023, 1024, 1025, 2047, 2048, 2049, 4095, 4096, 4097, 9000]
CASES = {
    "edges": EDGES * 3,
    "one_row_1024": [1024],
    "one_row_1025": [1025],
    "first_row_long": [3000] + [5] * 40,
    "last_row_long": [5] * 63 + [2049],
    "alternating": [1500, 3, 0, 700] * 20,
    "all_long": [1025 + 7 * i for i in range(70)],
    "batch_edges": [1024 - 3, 3, 1024, 1, 1023, 512, 512, 511, 2, 30] * 7,
    "empty_rows_only": [0] * 100,
}


@pytest.mark.parametrize("name", CASES)
def test_features_at_split_edges(name):
    A = _matrix(CASES[name], 20_000, seed=len(name))
    dA = sp.DeviceCSR.from_host(A)
    sp.spmv_validate(dA)
    o = oracle.features(A, line_bytes=128, l2_bytes=torch.cuda.get_device_properties(0).L2_cache_size)
    for _ in range(2):                             # the counters are left as they were found
        g = sp.spmv_features(dA, 128).as_dict()
        for k in ("nnz_min", "nnz_max", "nnz_sum", "nnz_sumsq", "bw_min", "bw_max", "bw_sum", "bw_sumsq",
                  "disp_sum", "disp_sumsq", "clust_sum", "ngroups_sum", "misses_sum"):
            assert g[k] == o[k], k


@pytest.mark.parametrize("row,at", [(0, 1), (2, 1024), (2, 2048), (3, 31), (3, 32), (5, 1023)])
def test_disorder_is_found_in_any_row(row, at):
    """One column equal to its predecessor, at the start of a step, a batch
    or a piece: the matrix is refused, and the next one is accepted."""
    A = _matrix([40, 7, 3000, 64, 0, 1024], 20_000, seed=5)
    ok = sp.DeviceCSR.from_host(A)
    bad = A.colind.clone()
    j = int(A.rowptr[row]) + at
    bad[j] = bad[j - 1]
    with pytest.raises(sp.SpmvError, match="strictly increasing"):
        sp.spmv_validate(sp.DeviceCSR(A.n_rows, A.n_cols, A.rowptr.cuda(), bad.cuda(), A.val.cuda()))
    sp.spmv_validate(ok)
