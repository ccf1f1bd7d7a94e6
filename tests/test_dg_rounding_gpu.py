"""Rounding of the DG volume kernel in FP32: its error against the FP64 oracle is no larger than that of the
plain order of the sums (each node's two products added together, then to the output), restated here."""
import numpy as np
import pytest

import workloads as W
from oracle import dg

pytestmark = pytest.mark.gpu
F = np.float32


def _fma(a, b, c):
    """a b + c of FP32 values, rounded to FP32 (the product is exact in FP64)"""
    return (a.astype(np.float64) * b.astype(np.float64) + c.astype(np.float64)).astype(F)


def _operators(N):
    """The library's operator block of order N and its two matrices in FP32."""
    import torch

    import paper_1403_0968_gb300 as sem

    ops, Np = sem.dg_load_operators(N, torch.float32), (N + 1) * (N + 2) // 2
    Dr, Ds = ops.cpu().numpy().view(F).reshape(2, Np, -1)[:, :, :Np]
    for D, k in ((Dr, "Drw"), (Ds, "Dsw")):  # rows padded: [2][Np][row stride]
        assert np.max(np.abs(D - dg.operators(N)[k])) < 1e-6 * np.max(np.abs(D))
    return ops, Dr, Ds


def _pair_order(Dr, Ds, Q, B, geo, g):
    g = F(g)
    h, hu, hv = Q[:, 0], Q[:, 1], Q[:, 2]
    ih = F(1) / h
    a, b, p = hu * ih, hv * ih, F(0.5) * g * h * h
    Fx, Gx = [hu, _fma(hu, a, p), hu * b], [hv, hv * a, _fma(hv, b, p)]
    rx, ry, sx, sy = (q[:, None] for q in geo)
    out = np.empty_like(Q)
    for f in range(3):
        Xr, Xs = _fma(rx, Fx[f], ry * Gx[f]), _fma(sx, Fx[f], sy * Gx[f])
        acc = np.zeros_like(h)
        for j in range(h.shape[1]):
            acc = acc + _fma(Dr[:, j][None], Xr[:, j:j + 1], Ds[:, j][None] * Xs[:, j:j + 1])
        out[:, f] = acc if f == 0 else _fma(-(g * h), B[:, f - 1], acc)
    return out


# element counts of each form: one thread per node, four, two and one lanes per element.  Both orders round
# the same number of times in their fluxes; the sums of groups of nodes round fewer times at full size, so
# the bound is the plain order's own error.
@pytest.mark.parametrize("N", range(3, 9))
@pytest.mark.parametrize("cells", [20, 80, 110])
def test_error_at_most_that_of_plain_sums(N, cells):
    import torch

    import paper_1403_0968_gb300 as sem

    verts = W.tri_mesh(cells, cells, perturb=0.2, seed=N)
    E, Np = len(verts), (N + 1) * (N + 2) // 2
    Q, B = (a.astype(F) for a in W.swe_fields(E, Np, seed=N + 7))
    geo = [a.astype(F) for a in dg.geometry(verts)[:4]]
    ref = dg.volume(N, Q.astype(float), B.astype(float), [a.astype(float) for a in geo], 9.81)
    ops, Dr, Ds = _operators(N)
    got = sem.dg_volume(N, torch.from_numpy(Q).cuda(), torch.from_numpy(B).cuda(),
                        torch.from_numpy(np.stack(geo, 1)).cuda(), 9.81, ops)
    rms = lambda a: float(np.sqrt(np.mean((a.astype(float) - ref) ** 2)))  # noqa: E731
    assert rms(got.cpu().numpy()) <= rms(_pair_order(Dr, Ds, Q, B, geo, 9.81))
