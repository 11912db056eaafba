"""spmv_host where the kernel writes y into the caller's page-locked memory
itself, and where it must not: every variant, rows in order and sorted, several
lanes a row, pageable memory, a page-locked vector that starts inside its
block, x and y in one buffer.  The same bits as the device product."""
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


FORMS = [("scalar", {}), ("subwarp", dict(threads_per_row=1)), ("subwarp", dict(threads_per_row=2)),
         ("subwarp", dict(threads_per_row=8)), ("latency", dict(threads_per_row=2)), ("stream", {}), ("merge", {}),
         ("dynamic", {}), ("compressed", dict(threads_per_row=1)), ("compressed", dict(value_type=sp.VAL_BF16)),
         ("sliced", dict(block_nnz=1)), ("sliced", dict(block_nnz=1, items_per_warp=8)), ("sliced", dict(block_nnz=64)),
         ("sliced", dict(block_nnz=1, value_type=sp.VAL_F32))]


@pytest.mark.parametrize("memory", ["pinned", "pinned_inside", "pageable"])
@pytest.mark.parametrize("variant,kw", FORMS, ids=[f"{v}-{'-'.join(map(str, k.values()))}" for v, k in FORMS])
def test_same_bits_as_on_the_device(variant, kw, memory):
    A = synth.random_csr(5003, 5003, 40, seed=3, empty_frac=0.2)
    P = sp.spmv_prepare(sp.DeviceCSR.from_host(A), sp.make_choice(variant, **kw))
    x = synth.uniform_vector(A.n_cols, 1)
    y = torch.full((A.n_rows,), float("nan"), dtype=torch.float64, device="cuda")
    sp.spmv(P, x.cuda(), y)
    torch.cuda.synchronize()
    buf = torch.full((A.n_rows + 6,), float("nan"), dtype=torch.float64)
    if memory != "pageable":
        buf = buf.pin_memory()
    yh = buf[3:3 + A.n_rows] if memory == "pinned_inside" else buf[:A.n_rows]
    for _ in range(2):
        yh.fill_(float("nan"))
        sp.spmv_host(P, x.pin_memory(), yh)
        assert torch.equal(yh, y.cpu())
    rest = torch.cat([buf[:3], buf[3 + A.n_rows:]]) if memory == "pinned_inside" else buf[A.n_rows:]
    assert torch.isnan(rest).all()                  # nothing beside y is written


def test_x_and_y_in_one_buffer():
    A = synth.stencil_27pt(20, seed=1)
    P = sp.spmv_prepare(sp.DeviceCSR.from_host(A), sp.make_choice("sliced"))
    x = synth.uniform_vector(A.n_cols, 2)
    want = torch.empty(A.n_rows, dtype=torch.float64).pin_memory()
    sp.spmv_host(P, x.pin_memory(), want)
    both = x.clone().pin_memory()
    sp.spmv_host(P, both, both)
    assert torch.equal(both, want)
