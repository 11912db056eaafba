"""Training kernel at the edges of its tiling: widths that are not multiples
of the 4 x 4 gradient tiles, the smallest and the largest network, sample
counts around a slice (8) and past one slice per CTA (2 CTAs per SM), where a
CTA adds further slices to its partial.  Against the FP64 oracle with the
bounds of the other training tests: the network's sums have at most 128 + 128
+ 32 terms and the batch's at most 2,500, all of mixed sign, so FP32 rounding
stays far below 1e-4 of the largest gradient entry."""
import numpy as np
import pytest
import torch

import oracle
import paper_1511_02494_gb300 as sp

pytestmark = pytest.mark.gpu
NAMES = ("W1", "b1", "W2", "b2", "W3", "b3")


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1511_02494_gb300.build import build
    build()
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"


def _params(h1, h2, k, seed):
    g = np.random.default_rng(seed)
    return {"W1": (g.standard_normal((h1, 16)) * 0.3).astype(np.float32),
            "b1": (g.standard_normal(h1) * 0.1).astype(np.float32),
            "W2": (g.standard_normal((h2, h1)) / np.sqrt(h1)).astype(np.float32),
            "b2": (g.standard_normal(h2) * 0.1).astype(np.float32),
            "W3": (g.standard_normal((k, h2)) / np.sqrt(h2)).astype(np.float32),
            "b3": (g.standard_normal(k) * 0.1).astype(np.float32)}


@pytest.mark.parametrize("soft", [False, True])
@pytest.mark.parametrize("n", [1, 7, 8, 9, 2500])
@pytest.mark.parametrize("shape", [(1, 1, 2), (3, 5, 3), (64, 64, 8), (65, 127, 31), (128, 128, 32)])
def test_loss_grad_shapes(shape, n, soft):
    h1, h2, k = shape
    P = _params(h1, h2, k, 7 * n + k)
    g = np.random.default_rng(n)
    z = g.standard_normal((n, 16)).astype(np.float32)
    lab = g.integers(0, k, n).astype(np.int32)
    q = g.random((n, k)).astype(np.float32)
    q /= q.sum(1, keepdims=True)
    # parameters at a 4-byte offset: nothing may rely on wider alignment
    flat = np.concatenate([[0.0]] + [P[m].reshape(-1) for m in NAMES]).astype(np.float32)
    p = torch.from_numpy(flat).cuda()[1:]
    dz = torch.from_numpy(z).cuda()
    t = torch.from_numpy(q if soft else lab).cuda()
    fn = sp.spmv_mlp_loss_grad_soft if soft else sp.spmv_mlp_loss_grad
    grads = []
    for _ in range(2):
        grad = torch.full((p.numel(),), float("nan"), dtype=torch.float32, device="cuda")
        loss = torch.empty(1, dtype=torch.float32, device="cuda")
        fn(p, h1, h2, k, dz, t, grad, loss)
        grads.append(grad)
    torch.cuda.synchronize()
    assert torch.equal(grads[0], grads[1])
    P64 = {m: P[m].astype(np.float64) for m in NAMES}
    ref_loss, G = oracle.mlp_loss_grad_soft_f64(P64, z, q) if soft else oracle.mlp_loss_grad_f64(P64, z, lab)
    ref = np.concatenate([G[m].reshape(-1) for m in NAMES])
    assert abs(loss.item() - ref_loss) <= 1e-5 * max(1.0, abs(ref_loss))
    assert np.max(np.abs(grads[0].cpu().numpy() - ref)) <= 1e-4 * np.max(np.abs(ref))
