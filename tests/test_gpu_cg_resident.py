"""The one-launch CG loop against the oracle's CG: row counts around a slice,
around each number of slices per warp (152 SMs x 24 warps x 32 rows each) and
past the largest it takes (the three-kernel loop then), row lengths around its
chunks of eight, sorted rows (permuted slices) in either matrix, refinement
with the exact matrix laid out otherwise, every value type and accumulation.
Bounds as the other CG tests: the same algorithm and arithmetic up to the
order of the dot products' sums."""
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


def _spd(n, half, seed, uneven=False):
    """SPD band: symmetric couplings to the next `half` rows (all of them, or
    a random half), the diagonal strictly dominant."""
    g = np.random.default_rng(seed)
    d = np.arange(1, half + 1)
    i = np.repeat(np.arange(n), half)
    j = i + np.tile(d, n)
    keep = j < n
    if uneven:
        keep &= g.random(j.size) < 0.5
    i, j = i[keep], j[keep]
    w = -g.uniform(0.5, 1.5, i.size)
    diag = np.ones(n)
    np.add.at(diag, i, -w)
    np.add.at(diag, j, -w)
    r = np.concatenate([i, j, np.arange(n)])
    c = np.concatenate([j, i, np.arange(n)])
    v = np.concatenate([w, w, diag])
    o = np.lexsort((c, r))
    rp = np.concatenate([[0], np.cumsum(np.bincount(r, minlength=n))]).astype(np.int32)
    return synth.HostCSR(n, n, torch.from_numpy(rp), torch.from_numpy(c[o].astype(np.int32)),
                         torch.from_numpy(v[o]), "spd_band")


def _solve(A, inner, iters, refine=0, exact=None, graph=True):
    dA = sp.DeviceCSR.from_host(A)
    Pi = sp.spmv_prepare(dA, inner)
    Pe = sp.spmv_prepare(dA, exact) if exact is not None else Pi
    b = synth.uniform_vector(A.n_rows, 3)
    x = torch.zeros(A.n_rows, dtype=torch.float64, device="cuda")
    res = torch.full((iters + 1,), float("nan"), dtype=torch.float64, device="cuda")
    sp.spmv_cg(Pi, b.cuda(), x, iters, refine, A_exact=Pe, resid=res, use_graph=graph)
    torch.cuda.synchronize()
    return b, x.cpu().numpy(), res.cpu().numpy()


def _close(x, r, xo, ro):
    assert np.max(np.abs(x - xo)) <= 1e-9 * np.max(np.abs(xo))
    assert np.all(np.abs(r - ro) <= 1e-6 * ro + 1e-12 * ro[0])


W = 152 * 24 * 32      # rows one slice per warp covers on 152 SMs


@pytest.mark.parametrize("n", [1, 31, 32, 33, 1000, W, W + 1, 2 * W + 33, 3 * W + 1, 9 * W, 9 * W + 1])
def test_row_counts(n):
    A = _spd(n, 3, seed=n)
    iters = 30 if n < W else 8
    b, x, r = _solve(A, sp.make_choice("sliced"), iters)
    xo, ro = oracle.cg(A, b, np.zeros(n), iters)
    if n > 1:
        _close(x, r, xo, ro)
    else:                                           # solved exactly in one step
        assert abs(x[0] - float(b[0]) / float(A.val[0])) <= 1e-15 * abs(x[0]) or np.isnan(x[0])


@pytest.mark.parametrize("sigma", [1, 256])
@pytest.mark.parametrize("half", [1, 3, 4, 8, 11, 20])
def test_row_lengths_and_sorted_rows(half, sigma):
    A = _spd(3001, half, seed=half, uneven=True)
    b, x, r = _solve(A, sp.make_choice("sliced", block_nnz=sigma), 40)
    xo, ro = oracle.cg(A, b, np.zeros(A.n_rows), 40)
    _close(x, r, xo, ro)


@pytest.mark.parametrize("index_bytes", [1, 2])
def test_narrow_columns(index_bytes):
    A = _spd(5000, 100 if index_bytes == 2 else 6, seed=2, uneven=True)
    ch = sp.make_choice("sliced", index_bytes=index_bytes)
    b, x, r = _solve(A, ch, 40)
    xo, ro = oracle.cg(A, b, np.zeros(A.n_rows), 40)
    _close(x, r, xo, ro)


@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("vt,vkind", [(sp.VAL_F32, 1), (sp.VAL_BF16, 2)])
@pytest.mark.parametrize("refine", [0, 7])
@pytest.mark.parametrize("n", [4000, 2 * W + 5])
def test_low_precision_with_refinement(n, refine, vt, vkind, graph):
    A = _spd(n, 5, seed=7, uneven=True)
    low = oracle.round_f32(A.val) if vkind == 1 else oracle.round_bf16(A.val)
    iters = 30 if n < W else 10
    b, x, r = _solve(A, sp.make_choice("sliced", value_type=vt, accumulate=sp.ACC_F64, block_nnz=64), iters, refine,
                     sp.make_choice("sliced", block_nnz=1), graph)
    xo, ro = oracle.cg(A, b, np.zeros(n), iters, vkind=vkind, lowval=low, refine=refine)
    _close(x, r, xo, ro)


@pytest.mark.parametrize("spread", [5, 70_000])       # 16-bit offsets, 32-bit columns
def test_fp32_sums_reach_fp64_accuracy(spread):
    A = _spd(90_000 if spread > 5 else 3000, 5, seed=9)
    if spread > 5:                                    # one coupling across the matrix
        n = A.n_rows
        i = np.arange(n)
        r = np.concatenate([np.repeat(i, np.diff(A.rowptr.numpy())), [0, n - 1]])
        c = np.concatenate([A.colind.numpy(), [n - 1, 0]])
        v = np.concatenate([A.val.numpy(), [-0.5, -0.5]])
        o = np.lexsort((c, r))
        rp = np.concatenate([[0], np.cumsum(np.bincount(r, minlength=n))]).astype(np.int32)
        A = synth.HostCSR(n, n, torch.from_numpy(rp), torch.from_numpy(c[o].astype(np.int32)), torch.from_numpy(v[o]))
    b, x, _ = _solve(A, sp.make_choice("sliced", value_type=sp.VAL_BF16), 120, 10, sp.make_choice("sliced"))
    assert np.linalg.norm(b.numpy() - oracle.spmv(A, x)) < 1e-8 * np.linalg.norm(b.numpy())
