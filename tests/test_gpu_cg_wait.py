"""The one-launch CG loop's waits run out (one arrival short, two seconds): x and
the residuals after the first are NaN, and the next solve on the same objects is
right.  Which solves run as one launch.  And the
smallest system, one row, solved exactly by its first iteration."""
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


def _prepare(A, **kw):
    return sp.spmv_prepare(sp.DeviceCSR.from_host(A), sp.make_choice("sliced", **kw))


def _vectors(n, iters):
    x = torch.zeros(n, dtype=torch.float64, device="cuda")
    return synth.uniform_vector(n, 3, device="cuda"), x, torch.full((iters + 1,), -1.0, dtype=torch.float64, device="cuda")


@pytest.mark.parametrize("side,kw,refine", [
    (5, {}, 0), (33, {}, 3), (64, {}, 0), (33, dict(index_bytes=2), 0), (33, dict(value_type=sp.VAL_F32), 0),
    (64, dict(value_type=sp.VAL_BF16), 3), (5, dict(value_type=sp.VAL_BF16, accumulate=sp.ACC_F64), 3)])
def test_a_wait_that_gives_up(side, kw, refine):
    A = synth.laplacian_3d_7pt(side)
    P, E = _prepare(A, **kw), _prepare(A)
    iters = 8
    b, x, r = _vectors(A.n_rows, iters)
    sp.spmv_cg_wait_check(P, b, x, iters, False, refine, E, r)
    assert torch.isnan(x).all() and torch.isnan(r[1:]).all()
    start = float(r[0])
    assert abs(start - float(torch.linalg.vector_norm(b))) <= 1e-12 * start
    solved = []
    for check in (True, False):
        b, x, r = _vectors(A.n_rows, iters)
        if check:
            sp.spmv_cg_wait_check(P, b, x, iters, True, refine, E, r)
        else:
            sp.spmv_cg(P, b, x, iters, refine, A_exact=E, resid=r)
        solved.append((x.cpu(), r.cpu()))
        assert float(r[0]) == start and float(r[-1]) < 0.9 * start
    assert torch.equal(solved[0][0], solved[1][0]) and torch.equal(solved[0][1], solved[1][1])


def test_one_row_is_solved_by_the_first_iteration():
    A = synth.HostCSR(1, 1, torch.tensor([0, 1], dtype=torch.int32), torch.tensor([0], dtype=torch.int32),
                      torch.tensor([4.0], dtype=torch.float64), "one")
    P = _prepare(A)
    b = torch.tensor([1.5], dtype=torch.float64)
    for iters in (1, 3):
        x = torch.zeros(1, dtype=torch.float64, device="cuda")
        r = torch.full((iters + 1,), -1.0, dtype=torch.float64, device="cuda")
        sp.spmv_cg_wait_check(P, b.cuda(), x, iters, True, resid=r)
        xo, ro = oracle.cg(A, b, np.zeros(1), iters)
        assert np.array_equal(r.cpu().numpy(), ro, equal_nan=True)
        assert np.array_equal(x.cpu().numpy(), xo, equal_nan=True)
        if iters == 1:                          # every step of it is exact; the ones after divide 0 by 0
            assert float(x[0]) == 0.375 and r.tolist() == [1.5, 0.0]
        else:
            assert r[:2].tolist() == [1.5, 0.0] and torch.isnan(r[2:]).all() and torch.isnan(x).all()


def _uneven(n, longest):
    rp = torch.tensor([0] + [longest] + [1] * (n - 1)).cumsum(0).to(torch.int32)
    ci = torch.cat([torch.arange(longest), torch.arange(1, n)]).to(torch.int32)
    return synth.HostCSR(n, n, rp, ci, torch.ones(ci.numel(), dtype=torch.float64), "uneven")


OTHER_FORMS = {
    "another variant": lambda: (sp.spmv_prepare(sp.DeviceCSR.from_host(synth.laplacian_3d_7pt(8)), sp.make_choice("subwarp")), None, 4, 0),
    "long rows": lambda: (_prepare(_uneven(4000, 2000), block_nnz=1), None, 4, 0),
    "coded columns": lambda: (_prepare(synth.laplacian_3d_7pt(8), index_coding=1), None, 4, 0),
    "refined with another variant": lambda: (_prepare(synth.laplacian_3d_7pt(8)), sp.spmv_prepare(sp.DeviceCSR.from_host(synth.laplacian_3d_7pt(8)), sp.make_choice("subwarp")), 4, 2),
    "refined with FP32 values": lambda: (_prepare(synth.laplacian_3d_7pt(8)), _prepare(synth.laplacian_3d_7pt(8), value_type=sp.VAL_F32), 4, 2),
    "more rows than the shared memory holds": lambda: (_prepare(synth.laplacian_3d_7pt(102)), None, 1, 0),
    "no iterations": lambda: (_prepare(synth.laplacian_3d_7pt(8)), None, 0, 0),
}


@pytest.mark.parametrize("form", OTHER_FORMS)
def test_solves_that_do_not_run_as_one_launch(form):
    P, E, iters, refine = OTHER_FORMS[form]()
    b, x, _ = _vectors(P.A.n_rows, iters)
    with pytest.raises(sp.SpmvError, match="does not run as one launch"):
        sp.spmv_cg_wait_check(P, b, x, iters, False, refine, E)
    assert not x.any()


def _band(n, width):
    """Rows of `width` columns around the diagonal, as many as lie inside."""
    c = torch.arange(n, device="cuda")[:, None] + torch.arange(-(width // 2), width - width // 2, device="cuda")
    keep = (c >= 0) & (c < n)
    rp = torch.cat([torch.zeros(1, dtype=torch.int64, device="cuda"), keep.sum(1).cumsum(0)]).to(torch.int32)
    ci = c[keep].to(torch.int32)
    v = torch.where(ci == torch.repeat_interleave(torch.arange(n, device="cuda"), keep.sum(1)), 2.0 * width, -1.0)
    return sp.DeviceCSR(n, n, rp, ci, v.to(torch.float64))


@pytest.mark.parametrize("kw,bytes_a_slot,head,vector,tenths", [
    ({}, 12, 140, 8, 17), (dict(index_bytes=2), 10, 140, 8, 17), (dict(value_type=sp.VAL_F32), 6, 268, 4, 7),
    (dict(value_type=sp.VAL_BF16), 4, 268, 4, 7), (dict(value_type=sp.VAL_BF16, accumulate=sp.ACC_F64), 4, 268, 8, 7)])
def test_one_launch_by_the_products_bytes_and_the_l2(kw, bytes_a_slot, head, vector, tenths):
    """Rows of 40 (whole groups of four): the row counts, in slices, just
    inside and just past the limit; both solve the system."""
    l2 = torch.cuda.get_device_properties(0).L2_cache_size
    slices = tenths * l2 // 10 // (32 * 40 * bytes_a_slot + head + 32 * vector)
    for n, one in ((32 * (slices - 1), True), (32 * (slices + 2), False)):
        A = _band(n, 40)
        P, E = sp.spmv_prepare(A, sp.make_choice("sliced", block_nnz=1, **kw)), sp.spmv_prepare(A, sp.make_choice("sliced"))
        b, x, r = _vectors(n, 6)
        if one:
            sp.spmv_cg_wait_check(P, b, x, 6, True, 3, E, r)
        else:
            with pytest.raises(sp.SpmvError, match="does not run as one launch"):
                sp.spmv_cg_wait_check(P, b, x, 6, True, 3, E, r)
        x.zero_()
        sp.spmv_cg(P, b, x, 6, 3, A_exact=E, resid=r)
        y = torch.empty_like(b)
        sp.spmv(E, x, y)
        left = float(torch.linalg.vector_norm(b - y))
        # the last iteration refined: the residual is the FP64 one of x
        assert abs(float(r[-1]) - left) <= 1e-9 * float(r[0]) and left < 0.5 * float(r[0])
