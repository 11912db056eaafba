"""Training with as many CTAs per SM as a network's shared memory admits, two to
four: sample counts one past a slice (8) for each of them and well past it, so
that CTAs add a second and third slice to their partials.  Against the FP64
oracle.  An entry is a sum of at most 12,000 terms of mixed sign, in partials of
at most 24 and a tree over at most 608 of them; with its rounding errors as
random as its terms it stays far below 1e-4 of the largest entry, the bound of
the other training tests."""
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


@pytest.mark.parametrize("more", [0, 1, 7135])
@pytest.mark.parametrize("shape,ctas", [((7, 5, 3), 4), ((64, 64, 8), 4), ((128, 64, 8), 3), ((128, 128, 32), 2)])
def test_samples_around_one_slice_per_cta(shape, ctas, more):
    h1, h2, k = shape
    n = 8 * ctas * torch.cuda.get_device_properties(0).multi_processor_count + more
    g = np.random.default_rng(n)
    P = {"W1": g.standard_normal((h1, 16)) * 0.3, "b1": g.standard_normal(h1) * 0.1,
         "W2": g.standard_normal((h2, h1)) / np.sqrt(h1), "b2": g.standard_normal(h2) * 0.1,
         "W3": g.standard_normal((k, h2)) / np.sqrt(h2), "b3": g.standard_normal(k) * 0.1}
    P = {m: P[m].astype(np.float32) for m in NAMES}
    z = g.standard_normal((n, 16)).astype(np.float32)
    lab = g.integers(0, k, n).astype(np.int32)
    p = torch.from_numpy(np.concatenate([P[m].reshape(-1) for m in NAMES])).cuda()
    grads = []
    for _ in range(2):
        grad, loss = torch.full_like(p, float("nan")), torch.empty(1, dtype=torch.float32, device="cuda")
        sp.spmv_mlp_loss_grad(p, h1, h2, k, torch.from_numpy(z).cuda(), torch.from_numpy(lab).cuda(), grad, loss)
        grads.append(grad)
    assert torch.equal(grads[0], grads[1])
    ref_loss, G = oracle.mlp_loss_grad_f64({m: P[m].astype(np.float64) for m in NAMES}, z, lab)
    ref = np.concatenate([G[m].reshape(-1) for m in NAMES])
    assert abs(loss.item() - ref_loss) <= 1e-5 * max(1.0, abs(ref_loss))
    assert np.max(np.abs(grads[0].cpu().numpy() - ref)) <= 1e-4 * np.max(np.abs(ref))
