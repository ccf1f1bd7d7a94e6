"""The DG volume kernel's reciprocal of the depth in FP32: within one unit in the last place of the correctly
rounded quotient (what CUDA's division gives) over random bit patterns, subnormal and huge depths included,
and infinite where the quotient is."""
import numpy as np
import pytest

import workloads as W
from oracle import dg

pytestmark = pytest.mark.gpu
F = np.float32


def _operators(N):
    """The library's operator block of order N and its two matrices in FP32."""
    import torch

    import paper_1403_0968_gb300 as sem

    ops, Np = sem.dg_load_operators(N, torch.float32), (N + 1) * (N + 2) // 2
    Dr, Ds = ops.cpu().numpy().view(F).reshape(2, Np, -1)[:, :, :Np]
    for D, k in ((Dr, "Drw"), (Ds, "Dsw")):  # rows padded: [2][Np][row stride]
        assert np.max(np.abs(D - dg.operators(N)[k])) < 1e-6 * np.max(np.abs(D))
    return ops, Dr, Ds


# rx = sy = 1, ry = sx = 0, g = 0 and hu = 1 at one node only: the second field is Drw[i][j0] / h at that
# node's row i plus zeros, one rounding after the reciprocal's.
@pytest.mark.parametrize("N,E", [(1, 2000), (1, 120000), (4, 2000), (4, 40000)])
def test_reciprocal_of_random_bit_patterns(N, E):
    import torch

    import paper_1403_0968_gb300 as sem

    bits = W.rng(E).integers(0, 2 ** 32, E, dtype=np.uint64).astype(np.uint32)
    bits[: E // 4] &= np.uint32(0x81FFFFFF)  # exponents of 2^-126 and a little above, subnormals
    hv = bits.view(F)
    with np.errstate(all="ignore"):
        ih = F(1) / hv
    hv = np.where(np.isfinite(ih) & np.isfinite(hv), hv, F(1))  # (the infinite ones below)
    ih = F(1) / hv
    ops, D, _ = _operators(N)
    i, j = np.unravel_index(np.argmax(np.abs(D)), D.shape)
    Np = len(D)
    Q = np.zeros((E, 3, Np), F)
    Q[:, 0], Q[:, 0, j], Q[:, 1, j] = 1, hv, 1
    geo = np.tile(np.array([1, 0, 0, 1], F), (E, 1))
    got = sem.dg_volume(N, torch.from_numpy(Q).cuda(), torch.zeros((E, 2, Np), device="cuda"),
                        torch.from_numpy(geo).cuda(), 0.0, ops)
    got = got.cpu().numpy()[:, 1, i].astype(float)
    with np.errstate(over="ignore"):
        want = (D[i, j] * ih).astype(float)  # as FP32
    ulp = np.spacing(np.abs(ih)).astype(float)
    ok = np.isfinite(want)
    # one unit of the reciprocal, and half a unit of the product
    assert np.all(np.abs(got - float(D[i, j]) * ih.astype(float))[ok] <=
                  abs(float(D[i, j])) * ulp[ok] + 0.5 * np.spacing(np.abs(want[ok]).astype(F)).astype(float))
    assert np.array_equal(got[~ok], want[~ok])


@pytest.mark.parametrize("N,E", [(2, 600), (4, 600), (4, 40000), (7, 20000)])
@pytest.mark.parametrize("depth", [1e-39, 0.0, -1e-40, np.inf])
def test_infinite_reciprocal(N, E, depth):
    """A depth whose reciprocal is infinite (or that is infinite) at one node gives the infinities and NaNs
    of the formulas in FP32."""
    import torch

    import paper_1403_0968_gb300 as sem

    g, Np = W.rng(N), (N + 1) * (N + 2) // 2
    ops, Dr, Ds = _operators(N)
    Q = np.empty((E, 3, Np), F)
    Q[:, 0] = g.uniform(1, 2, (E, Np))
    Q[:, 1:] = g.uniform(0.5, 1, (E, 2, Np))
    at = g.integers(0, Np, E)
    Q[np.arange(E), 0, at] = F(depth)
    geo = np.tile(np.array([2, 2, 1, 2], F), (E, 1))  # all positive: no zero times infinity
    got = sem.dg_volume(N, torch.from_numpy(Q).cuda(), torch.zeros((E, 2, Np), device="cuda"),
                        torch.from_numpy(geo).cuda(), 0.0, ops).cpu().numpy()
    with np.errstate(all="ignore"):
        h, hu, hv = Q[:, 0], Q[:, 1], Q[:, 2]
        ih = F(1) / h
        a, b, p = hu * ih, hv * ih, F(0) * h * h
        Fx, Gx = [hu, hu * a + p, hu * b], [hv, hv * a, hv * b + p]
        want = np.empty_like(Q)
        for f in range(3):
            Xr, Xs = F(2) * Fx[f] + F(2) * Gx[f], Fx[f] + F(2) * Gx[f]
            want[:, f] = (Dr[None] * Xr[:, None] + Ds[None] * Xs[:, None]).sum(-1)
    np.testing.assert_array_equal(np.isnan(got), np.isnan(want))
    inf = np.isinf(want)
    np.testing.assert_array_equal(np.isinf(got), inf)
    np.testing.assert_array_equal(np.sign(got[inf]), np.sign(want[inf]))
    if depth == 1e-39:
        assert inf.any()  # the case is not all NaN
