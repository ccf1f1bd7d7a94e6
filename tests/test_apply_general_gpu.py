"""Explicit numbering with a mask, alpha and kappa at every order and stored type (the kernels without a
solve's sum), ragged last blocks among them; and refinement solves on it (the kernels with it)."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
TOL = {"fp64": 1e-12, "fp32": 1e-5, "bf16": 1e-5, "fp32_otf": 1e-5}  # as for every apply of these types


def _problem(orc, N, box, features):
    import paper_1403_0968_gb300 as sem

    v = W.box_vertices(*box, perturb=0.15, seed=N)
    E, n3, ng = v.shape[0], (N + 1) ** 3, orc.box_nglobal(*box, N)
    modes = W.kappa_modes(4, seed=N)
    al = (0.5 + W.uniform(E * n3, seed=33, lo=0, hi=1)).reshape(E, n3)
    perm = W.rng(5).permutation(ng)
    glo, mask = perm[orc.box_numbering(*box, N)], np.zeros(ng, dtype=np.uint8)
    mask[perm] = orc.box_dirichlet(*box, N)
    P = sem.Problem(N, v, box=box, glo_num=glo, nglobal=ng, kappa_modes=modes, alpha=al, bc="mask", dirichlet=mask,
                    features=features)
    G, wJ = orc.factors(N, v, modes=modes)
    return P, glo, mask, G, al * wJ


@pytest.mark.parametrize("N", range(1, 16))
@pytest.mark.parametrize("box", [(1, 1, 1), (3, 3, 1)])
@pytest.mark.parametrize("prec", ["fp64", "fp32", "bf16", "fp32_otf"])
def test_apply_matches_oracle(orc, N, box, prec):
    import torch

    import paper_1403_0968_gb300 as sem
    from oracle import mlp

    feat = {"fp64": sem.SEM_FEAT_FP64, "fp32": sem.SEM_FEAT_FP32, "bf16": sem.SEM_FEAT_FP32 | sem.SEM_FEAT_BF16,
            "fp32_otf": sem.SEM_FEAT_OTF}[prec]
    P, glo, mask, G, wJa = _problem(orc, N, box, feat)
    u = W.uniform(len(mask), seed=N + 40)
    ud = torch.from_numpy(u).cuda()
    if prec != "fp64":
        ud = ud.float()
        u = ud.double().cpu().numpy()
    y = P.apply(ud, prec=prec).double().cpu().numpy()
    ref = orc.apply(N, glo, mlp.bf16(G) if prec == "bf16" else G, u, mask=mask, wJalpha=wJa)
    assert np.max(np.abs(y - ref)) <= TOL[prec] * np.max(np.abs(ref))


@pytest.mark.parametrize("N,box", [(3, (3, 3, 3)), (5, (3, 2, 2)), (7, (3, 2, 1)), (11, (2, 2, 1))])
@pytest.mark.parametrize("inner", ["fp32", "bf16", "fp32_otf"])
def test_refinement_solve(orc, N, box, inner):
    import torch

    import paper_1403_0968_gb300 as sem

    feat = {"fp32": sem.SEM_FEAT_FP32, "bf16": sem.SEM_FEAT_FP32 | sem.SEM_FEAT_BF16, "fp32_otf": sem.SEM_FEAT_OTF}[inner]
    P, glo, mask, G, wJa = _problem(orc, N, box, feat | sem.SEM_FEAT_FP64 | sem.SEM_FEAT_PCG)
    b = W.uniform(len(mask), seed=N) * (mask == 0)
    x, info = P.pcg(torch.from_numpy(b).cuda(), rtol=1e-10, mode="ir", apply_prec="fp64", inner_rtol=1e-3,
                    inner_prec=inner)
    r = b - orc.apply(N, glo, G, x.cpu().numpy(), mask=mask, wJalpha=wJa)
    assert np.linalg.norm(r) < 1.1e-10 * np.linalg.norm(b)
