"""Feature pass on tiles of short rows (at most 8 nonzeros, a lane's own
loads) and on the tiles next to them that one longer row sends through the
streaming: bit-exact with the oracle; and what is refused in such rows."""
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
        a = g.integers(0, n_cols - n + 1)
        # runs of consecutive columns, steps around a line (16 columns), anywhere
        kind = g.integers(0, 3)
        if kind == 0 or n == 0:
            rows.append(np.arange(a, a + n))
        elif kind == 1:
            c = np.cumsum(np.concatenate([[0], g.integers(15, 19, n - 1)]))
            rows.append(g.integers(0, n_cols - c[-1]) + c)
        else:
            rows.append(np.sort(g.choice(n_cols, n, replace=False)))
    rp = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int32)
    ci = np.concatenate(rows + [np.zeros(0, np.int64)]).astype(np.int32)
    return synth.HostCSR(len(lengths), n_cols, torch.from_numpy(rp), torch.from_numpy(ci),
                         torch.ones(ci.size, dtype=torch.float64), "short")


CASES = {
    "one_row": [1],
    "all_8": [8] * 100,
    "upto_8": [0, 1, 2, 3, 4, 5, 6, 7, 8] * 15,
    "one_9_among_them": [3] * 40 + [9] + [8] * 60,
    "tiles_in_turn": ([2] * 32 + [30] * 32) * 3 + [5] * 7,
    "with_a_long_row": [4] * 32 + [1025] + [6] * 50,
    "empty_and_one": [0, 1] * 64,
}


@pytest.mark.parametrize("name", CASES)
def test_features(name):
    A = _matrix(CASES[name], 20_000, seed=len(name))
    dA = sp.DeviceCSR.from_host(A)
    sp.spmv_validate(dA)
    o = oracle.features(A, line_bytes=128, l2_bytes=torch.cuda.get_device_properties(0).L2_cache_size)
    g = sp.spmv_features(dA, 128).as_dict()
    for k in ("nnz_min", "nnz_max", "nnz_sum", "nnz_sumsq", "bw_min", "bw_max", "bw_sum", "bw_sumsq",
              "disp_sum", "disp_sumsq", "clust_sum", "ngroups_sum", "misses_sum"):
        assert g[k] == o[k], k


@pytest.mark.parametrize("length", [2, 7, 8])
def test_what_is_refused(length):
    A = _matrix([length] * 70, 20_000, seed=length)
    for row in (0, 31, 32, 69):
        for value, words in ((-1, "out of"), (20_000, "out of"), (None, "strictly increasing")):
            ci = A.colind.clone()
            j = (row + 1) * length - 1
            ci[j] = ci[j - 1] if value is None else value
            bad = synth.HostCSR(A.n_rows, A.n_cols, A.rowptr, ci, A.val, "bad")
            with pytest.raises(sp.SpmvError, match=words):
                sp.spmv_validate(sp.DeviceCSR.from_host(bad))
    sp.spmv_validate(sp.DeviceCSR.from_host(A))
