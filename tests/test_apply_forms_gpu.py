"""The double-float apply and the FP64 apply with three threads per column on both sides of the element counts
where their form changes (limits are elements per SM, 152 SMs), with full and ragged last blocks, in box
numbering and in explicit numbering with a mask and alpha; and their CG step kernels above the limits."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
TOL = 1e-12  # of max |y|: the bound of every FP64-accurate apply

# double-float: N = 5 staged below 4256 elements; 6 scalar to 1976, then blocks of 5; 7 scalar from 457 to 1216; 8 scalar
# to 760 and from 913 to 1216, else blocks of 3; 9 small to 304 and from 609 to 912, scalar between and to 1216, then
# blocks of 3; 11 small to 152, scalar to 304 and from 609 to 912, else blocks of 2
EMU = [(5, (7, 16, 38)), (5, (16, 16, 17)), (5, (5, 23, 37)), (5, (12, 13, 13)), (6, (1, 1, 1)), (6, (8, 13, 19)),
       (6, (12, 13, 13)), (7, (3, 8, 19)), (7, (8, 8, 8)), (7, (8, 8, 19)), (7, (11, 11, 11)), (8, (4, 10, 19)),
       (8, (9, 9, 10)), (8, (10, 10, 10)), (8, (11, 11, 11)), (9, (1, 16, 19)), (9, (7, 7, 7)), (9, (2, 16, 19)),
       (9, (8, 9, 9)), (9, (4, 16, 16)), (9, (4, 16, 19)), (9, (11, 11, 11)), (11, (1, 8, 19)), (11, (4, 6, 7)),
       (11, (7, 7, 9)), (11, (3, 16, 19)), (11, (10, 10, 10)), (11, (9, 11, 11))]
COLS = [(14, (4, 4, 19)), (14, (7, 7, 7)), (13, (5, 7, 9)), (6, (2, 2, 2)), (12, (2, 2, 2))]


def _compare(orc, N, box, general, prec):
    import torch

    import paper_1403_0968_gb300 as sem

    v = W.box_vertices(*box, perturb=0.15, seed=N)
    E, n3 = v.shape[0], (N + 1) ** 3
    modes = W.kappa_modes(4, seed=N)
    glo, mask = orc.box_numbering(*box, N), orc.box_dirichlet(*box, N)
    ng = orc.box_nglobal(*box, N)
    feat = sem.SEM_FEAT_EMU if prec == "fp64_emu" else sem.SEM_FEAT_FP64
    G, wJ = orc.factors(N, v, modes=modes)
    wJa = None
    if general:
        al = (0.5 + W.uniform(E * n3, seed=33, lo=0, hi=1)).reshape(E, n3)
        wJa = al * wJ
        perm = W.rng(5).permutation(ng)
        glo = perm[glo]
        m = np.zeros(ng, dtype=np.uint8)
        m[perm] = mask
        mask = m
        P = sem.Problem(N, v, box=box, glo_num=glo, nglobal=ng, kappa_modes=modes, alpha=al, bc="mask", dirichlet=m,
                        features=feat)
    else:
        P = sem.Problem(N, v, box=box, kappa_modes=modes, bc="box", features=feat)
    u = W.uniform(ng, seed=N + 40)
    y = P.apply(torch.from_numpy(u).cuda(), prec=prec).cpu().numpy()
    ref = orc.apply(N, glo, G, u, mask=mask, wJalpha=wJa)
    assert np.max(np.abs(y - ref)) < TOL * np.max(np.abs(ref))


@pytest.mark.parametrize("general", [False, True])
@pytest.mark.parametrize("N,box", EMU)
def test_double_float_forms(orc, N, box, general):
    _compare(orc, N, box, general, "fp64_emu")


@pytest.mark.parametrize("general", [False, True])
@pytest.mark.parametrize("N,box", COLS)
def test_three_threads_per_column(orc, N, box, general):
    _compare(orc, N, box, general, "fp64")


# above and below the limits of the step kernel, which N = 9 and 11 have apart with explicit numbering: the true
# residual of a solve
@pytest.mark.parametrize("prec,N,box,general",
                         [("fp64_emu", 5, (12, 14, 15), False), ("fp64_emu", 6, (3, 4, 5), False),
                          ("fp64_emu", 6, (11, 12, 13), False), ("fp64_emu", 8, (10, 10, 10), False),
                          ("fp64_emu", 8, (3, 4, 5), False), ("fp64_emu", 9, (5, 7, 9), False),
                          ("fp64_emu", 9, (14, 15, 15), False), ("fp64_emu", 9, (7, 7, 7), True),
                          ("fp64_emu", 9, (10, 10, 10), True), ("fp64_emu", 11, (4, 5, 7), False),
                          ("fp64_emu", 11, (4, 7, 7), False), ("fp64_emu", 11, (9, 9, 9), False),
                          ("fp64_emu", 11, (4, 5, 7), True), ("fp64_emu", 11, (5, 7, 9), True),
                          ("fp64_emu", 11, (10, 10, 10), True), ("fp64", 6, (2, 3, 2), False),
                          ("fp64", 12, (2, 3, 2), False), ("fp64", 13, (5, 7, 9), False), ("fp64", 14, (7, 7, 7), False)])
def test_cg_step_kernel(orc, prec, N, box, general):
    import torch

    import paper_1403_0968_gb300 as sem

    v = W.box_vertices(*box, seed=N)
    E, n3, ng = v.shape[0], (N + 1) ** 3, orc.box_nglobal(*box, N)
    al = np.full((E, n3), 50.0)
    glo, mask = orc.box_numbering(*box, N), orc.box_dirichlet(*box, N)
    kw = {"bc": "box"}
    if general:
        perm, m = W.rng(5).permutation(ng), np.zeros(ng, dtype=np.uint8)
        m[perm] = mask
        glo, mask = perm[glo], m
        kw = {"bc": "mask", "dirichlet": mask, "glo_num": glo, "nglobal": ng}
    feat = sem.SEM_FEAT_EMU if prec == "fp64_emu" else sem.SEM_FEAT_FP64
    P = sem.Problem(N, v, box=box, alpha=al, features=feat | sem.SEM_FEAT_PCG, **kw)
    b = W.uniform(ng, seed=N) * (mask == 0)
    x, info = P.pcg(torch.from_numpy(b).cuda(), rtol=1e-10, mode="fp64", apply_prec=prec)
    G, wJ = orc.factors(N, v)
    r = b - orc.apply(N, glo, G, x.cpu().numpy(), mask=mask, wJalpha=al * wJ)
    # the solver's own FP64-accurate true residual is at most rtol; the oracle's is off it by rounding of A x
    assert np.linalg.norm(r) < 1.1e-10 * np.linalg.norm(b)
