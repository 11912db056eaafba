"""The feature pass at the largest accepted number of nonzeros, 2^31 - 2, with
short rows at the very end: the matrix's last tile has rows of eight down to
one element and empty rows, whose first element lies within eight of 2^31 - 1.
Every aggregate against its closed form.  The column array has room for more
elements than the matrix, out of range, so an element past the end that is
looked at makes the matrix invalid.  About 9 GB of device memory."""
import pytest
import torch

import paper_1511_02494_gb300 as sp

pytestmark = pytest.mark.gpu
NNZ = 2**31 - 2
COLS = 1 << 21
FULL = 1023                                             # rows 0..1022 hold every column
TAIL = [3] * 20 + [8, 7, 6, 5, 4, 3, 2, 1] + [0] * 4    # rows 1024..1055: one tile
GAP = 40                                                # columns between a tail row's elements
LONG = NNZ - FULL * COLS - sum(TAIL)                    # row 1023
ROOM = 64


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1511_02494_gb300.build import build
    build()
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"


@pytest.fixture(scope="module", params=[0, 3])          # elements past a 16-byte boundary
def at_the_limit(request):
    buf = torch.full((NNZ + ROOM,), COLS + 5, dtype=torch.int32, device="cuda")
    ci = buf[request.param:request.param + NNZ]
    cols = torch.arange(COLS, dtype=torch.int32, device="cuda")
    ci[:FULL * COLS].view(FULL, COLS).copy_(cols)
    ci[FULL * COLS:FULL * COLS + LONG] = cols[:LONG]
    ci[NNZ - sum(TAIL):] = torch.cat([GAP * torch.arange(n, dtype=torch.int32) for n in TAIL]).cuda()
    lens = torch.tensor([COLS] * FULL + [LONG] + TAIL, dtype=torch.int64)
    rp = torch.cat([torch.zeros(1, dtype=torch.int64), lens.cumsum(0)]).to(torch.int32).cuda()
    one = torch.ones(1, dtype=torch.float64, device="cuda")   # the pass reads no values
    yield sp.DeviceCSR(len(lens), COLS, rp, ci, one), lens.tolist()
    del ci, buf
    torch.cuda.empty_cache()


def test_features_with_short_rows_at_the_end(at_the_limit):
    A, lens = at_the_limit
    assert A.nnz == NNZ and int(A.rowptr[-1]) == NNZ
    f = sp.spmv_features(A).as_dict()
    sp.spmv_validate(A)
    bw, groups, disp, clust = [], [], [], []
    for i, n in enumerate(lens):
        tail = i > FULL
        bw.append(0 if n == 0 else GAP * (n - 1) if tail else n - 1)
        groups.append(0 if n == 0 else n if tail else 1)   # and as many line changes: 8 GAP > 128
        disp.append(0 if n == 0 else (n << 32) // (bw[-1] + 1))
        clust.append(0 if n == 0 else (groups[-1] << 32) // n)
    want = dict(nnz=NNZ, nnz_min=0, nnz_max=COLS, nnz_sum=NNZ, nnz_sumsq=sum(n * n for n in lens),
                bw_min=0, bw_max=COLS - 1, bw_sum=sum(bw), bw_sumsq=sum(b * b for b in bw),
                disp_sum=sum(disp), disp_sumsq=sum(d * d for d in disp), clust_sum=sum(clust),
                ngroups_sum=sum(groups), misses_sum=sum(groups))
    assert {k: f[k] for k in want} == want
