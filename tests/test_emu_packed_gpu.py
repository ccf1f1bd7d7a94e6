"""The double-float apply's packed and scalar forms at every order: element counts of one, around a
block (up to 32 elements) and ragged, against the oracle; and the kernel of a CG step (with the fused
reduction) through a short solve's true residual."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", range(1, 16))
@pytest.mark.parametrize("box", [(1, 1, 1), (3, 2, 1), (5, 3, 3)])
def test_apply_matches_oracle(orc, N, box):
    import torch

    import paper_1403_0968_gb300 as sem

    if N > 9 and box == (5, 3, 3):
        box = (3, 1, 1)  # one or two elements per block there
    v = W.box_vertices(*box, perturb=0.15, seed=N)
    modes = W.kappa_modes(4, seed=N)
    P = sem.Problem(N, v, box=box, kappa_modes=modes, bc="none", features=sem.SEM_FEAT_EMU)
    u = W.uniform(P.nglobal, seed=N + 40)
    y = P.apply(torch.from_numpy(u).cuda(), prec="fp64_emu").cpu().numpy()
    G, _ = orc.factors(N, v, modes=modes)
    ref = orc.apply(N, orc.box_numbering(*box, N), G, u)
    assert np.max(np.abs(y - ref)) < 1e-12 * np.max(np.abs(ref))  # the tolerance of every FP64-accurate apply


@pytest.mark.parametrize("N", [2, 3, 5, 7, 8, 9, 11, 12, 14, 15])
def test_cg_step_kernel(orc, N):
    import torch

    import paper_1403_0968_gb300 as sem

    box = (2, 3, 2)
    v = W.box_vertices(*box, seed=N)
    P = sem.Problem(N, v, box=box, bc="box", features=sem.SEM_FEAT_EMU | sem.SEM_FEAT_PCG)
    b = P.rhs(W.sine_forcing(P.node_coords()))
    x, info = P.pcg(b, rtol=1e-10, mode="fp64", apply_prec="fp64_emu")
    G, _ = orc.factors(N, v)
    rel = orc.true_relres(N, orc.box_numbering(*box, N), G, b.cpu().numpy(), x.cpu().numpy(),
                          mask=orc.box_dirichlet(*box, N))
    assert rel < 1e-10
