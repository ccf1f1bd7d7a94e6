"""The CG vector kernels at the lengths and alignments where they differ: fewer nodes than one vector
of 16 bytes per block, every remainder of the vector length, and a solution vector that starts 8 bytes
off a 16-byte boundary (one node at a time); and tiles of the fused batched step whose elements belong
to several problems."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


# nodes of the box: 8 (one element, N = 1), 27, 45, 75, 539 ...: remainders 0..3 of four FP32 values
@pytest.mark.parametrize("N,box", [(1, (1, 1, 1)), (2, (1, 1, 1)), (2, (2, 1, 1)), (1, (4, 4, 2)), (3, (2, 2, 3)),
                                   (5, (3, 3, 3))])
@pytest.mark.parametrize("mode", ["fp64", "ir"])
@pytest.mark.parametrize("offset", [0, 1])
def test_solve_from_offset_vector(orc, N, box, mode, offset):
    import torch

    import paper_1403_0968_gb300 as sem

    v = W.box_vertices(*box, seed=N)
    E, n3 = box[0] * box[1] * box[2], (N + 1) ** 3
    alpha = W.uniform(E * n3, seed=3, lo=1.0, hi=2.0).reshape(E, n3)
    P = sem.Problem(N, v, box=box, alpha=alpha, bc="none",
                    features=sem.SEM_FEAT_FP64 | sem.SEM_FEAT_FP32 | sem.SEM_FEAT_PCG)
    b = torch.from_numpy(W.uniform(P.nglobal, seed=N + 9)).cuda()
    x = torch.zeros(P.nglobal + 1, dtype=torch.float64, device="cuda")[offset:P.nglobal + offset]
    o = sem.SemPcgOpts()
    o.rtol, o.max_it, o.apply_prec, o.inner_rtol, o.check_every, o.use_graph = 1e-10, 2000, sem.SEM_FP64, 1e-3, 5, 1
    o.mode = {"fp64": sem.SEM_SOLVE_FP64, "ir": sem.SEM_SOLVE_IR}[mode]
    res = sem.sem_pcg(P.handle, b, x, o)
    assert res.true_relres <= 1e-10
    G, wJ = orc.factors(N, v)
    y = orc.apply(N, orc.box_numbering(*box, N), G, x.cpu().numpy(), wJalpha=wJ * alpha)
    assert np.linalg.norm(y - b.cpu().numpy()) < 1.1e-10 * np.linalg.norm(b.cpu().numpy())


def test_fused_batch_tiles_of_many_problems():
    import torch

    import paper_1403_0968_gb300 as sem

    # one to three elements per problem: a tile of order 3 (16 elements) or 5 (7) spans several
    boxes = [(1, 1, 1), (2, 1, 1), (3, 1, 1), (1, 2, 1), (1, 1, 1), (1, 1, 3), (2, 2, 1), (1, 1, 2)]
    probs = [{"N": N, "box": b, "vertices": W.box_vertices(*b, seed=i)}
             for i, (N, b) in enumerate((N, b) for N in (3, 5, 7) for b in boxes)]
    B = sem.Batch(probs)
    assert B.fused_state() == (True, True)
    b = torch.cat([sem.Problem(p["N"], p["vertices"], box=p["box"], features=sem.SEM_FEAT_EMU | sem.SEM_FEAT_PCG)
                   .residual(torch.from_numpy(W.uniform(n, seed=i)).cuda(), torch.zeros(n, dtype=torch.float64, device="cuda"))
                   for i, (p, n) in enumerate(zip(probs, B.sizes))])
    x, out, status = B.pcg(b, rtol=1e-10, inner_rtol=1e-3)
    assert status == "SEM_OK" and max(r["true_relres"] for r in out) <= 1e-10
    x2, out2, _ = B.pcg(b, rtol=1e-10, inner_rtol=1e-3, multi_launch=True)
    assert np.max(np.abs((x - x2).cpu().numpy())) < 1e-8 * float(x2.abs().max())
