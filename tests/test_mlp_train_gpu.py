"""The training step's GEMM tiles at the sizes where their edges lie: one row, row counts around a
tile, odd input widths (n^3 + 6 = 33), and enough rows for the large tile."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


# 2560 rows: 160 tiles of 64 x 64 per 256-column product, the large tile; fewer: the split one
@pytest.mark.parametrize("N,batch", [(2, 1), (2, 31), (2, 33), (3, 65), (2, 2560)])
def test_step_matches_fp64(N, batch):
    import torch

    import paper_1403_0968_gb300 as sem
    from paper_1403_0968_gb300 import learn

    n3, h = (N + 1) ** 3, sem.MLP_H1
    g = W.rng(100 * N + batch)
    p = learn.he_init(N, seed=batch)
    X = g.normal(size=(batch, n3 + 6)).astype(np.float32)
    T = g.normal(size=(batch, n3)).astype(np.float32)
    m, v = (g.normal(size=p.shape) * 1e-3).astype(np.float32), g.uniform(1e-6, 1e-5, p.shape).astype(np.float32)
    tr = sem.MlpTrainer(N, torch.from_numpy(p).cuda(), batch, lr=1e-3)
    tr.m.copy_(torch.from_numpy(m))
    tr.v.copy_(torch.from_numpy(v))
    tr.step_count = 9
    grad = torch.empty_like(tr.params)
    loss = tr.step(torch.from_numpy(X).cuda(), torch.from_numpy(T).cuda(), grad_out=grad)
    tr2 = sem.MlpTrainer(N, torch.from_numpy(p).cuda(), batch)
    tr2.step(torch.from_numpy(X).cuda(), torch.from_numpy(T).cuda(), lr=0.0)  # no update, no gradient asked
    np.testing.assert_array_equal(tr2.params.cpu().numpy(), p)

    q = torch.from_numpy(p).double().requires_grad_()
    at, a = 0, torch.from_numpy(X).double()
    for i, (ni, no) in enumerate(((n3 + 6, h), (h, h), (h, n3))):
        a = a @ q[at:at + ni * no].reshape(ni, no) + q[at + ni * no:at + ni * no + no]
        a = torch.relu(a) if i < 2 else a
        at += ni * no + no
    lref = ((a - torch.from_numpy(T).double()) ** 2).mean()
    (gref,) = torch.autograd.grad(lref, q)
    gref, lref = gref.numpy(), float(lref.detach())
    # each FP32 sum of K terms is off by at most K 2^-24 of the sum of |terms|; five products with
    # K <= 2560 follow one another, and sums of random terms stay far below that: 1e-5 of the largest
    assert abs(float(loss.item()) - lref) < 1e-5 * lref
    got = grad.cpu().numpy()
    assert np.max(np.abs(got - gref)) < 1e-5 * np.max(np.abs(gref))
    # Adam from the gradient that was returned: elementwise FP32, a few roundings; the decay rates
    # are the library's FP32 constants
    b1, b2 = np.float32(0.9), np.float32(0.999)
    c1, c2 = float(np.float32(1) - b1), float(np.float32(1) - b2)
    m1, v1 = float(b1) * m + c1 * got.astype(float), float(b2) * v + c2 * got.astype(float) ** 2
    p1 = p - 1e-3 * (m1 / (1 - 0.9 ** 10)) / (np.sqrt(v1 / (1 - 0.999 ** 10)) + 1e-8)
    np.testing.assert_allclose(tr.m.cpu().numpy(), m1, rtol=1e-5, atol=1e-9)
    np.testing.assert_allclose(tr.v.cpu().numpy(), v1, rtol=1e-5)
    np.testing.assert_allclose(tr.params.cpu().numpy(), p1, rtol=1e-5, atol=1e-7)
