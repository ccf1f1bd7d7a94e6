"""The FP64 apply with three threads per column: every order it covers and the ones beside its range, one
and a few elements, both sides of its size limits, box and general numbering with a mask, against the oracle; and its
fused reduction through a solve's true residual."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
TOL = 1e-12  # of max |y|: the bound of every FP64-accurate apply


@pytest.mark.parametrize("general", [False, True])
@pytest.mark.parametrize("N,box", [(N, (2, 1, 1)) for N in range(2, 16)] + [(N, (3, 2, 3)) for N in range(3, 12)] +
                         [(3, (8, 8, 9)), (3, (8, 7, 11)), (4, (8, 8, 7)), (4, (8, 8, 8)), (7, (1, 1, 1)), (13, (7, 7, 7))])
def test_apply_matches_oracle(orc, N, box, general):
    import torch

    import paper_1403_0968_gb300 as sem

    v = W.box_vertices(*box, perturb=0.15, seed=N)
    E, n3 = v.shape[0], (N + 1) ** 3
    modes = W.kappa_modes(4, seed=N)
    al = (0.5 + W.uniform(E * n3, seed=33, lo=0, hi=1)).reshape(E, n3)
    glo, mask = orc.box_numbering(*box, N), orc.box_dirichlet(*box, N)
    ng = orc.box_nglobal(*box, N)
    if general:
        perm = W.rng(5).permutation(ng)
        glo = perm[glo]
        m = np.zeros(ng, dtype=np.uint8)
        m[perm] = mask
        P = sem.Problem(N, v, box=box, glo_num=glo, nglobal=ng, kappa_modes=modes, alpha=al, bc="mask", dirichlet=m,
                        features=sem.SEM_FEAT_FP64)
        mask = m
    else:
        P = sem.Problem(N, v, box=box, kappa_modes=modes, alpha=al, bc="box", features=sem.SEM_FEAT_FP64)
    u = W.uniform(ng, seed=N + 40)
    y = P.apply(torch.from_numpy(u).cuda(), prec="fp64").cpu().numpy()
    G, wJ = orc.factors(N, v, modes=modes)
    ref = orc.apply(N, glo, G, u, mask=mask, wJalpha=al * wJ)
    assert np.max(np.abs(y - ref)) < TOL * np.max(np.abs(ref))


@pytest.mark.parametrize("N", [3, 4, 5, 7, 8, 9, 11, 14])
def test_cg_step_kernel(orc, N):
    import paper_1403_0968_gb300 as sem

    box = (2, 3, 2)
    v = W.box_vertices(*box, seed=N)
    P = sem.Problem(N, v, box=box, bc="box", features=sem.SEM_FEAT_FP64 | sem.SEM_FEAT_PCG)
    b = P.rhs(W.sine_forcing(P.node_coords()))
    x, info = P.pcg(b, rtol=1e-10, mode="fp64", apply_prec="fp64")
    G, _ = orc.factors(N, v)
    rel = orc.true_relres(N, orc.box_numbering(*box, N), G, b.cpu().numpy(), x.cpu().numpy(),
                          mask=orc.box_dirichlet(*box, N))
    assert rel < 1e-10
