"""The DG volume kernel on both sides of the mesh sizes where its form changes (one thread per node, four, two
or one lanes per element; the limits are triangles per SM, 152 SMs), aligned and 4 or 8 bytes off."""
import numpy as np
import pytest

import workloads as W
from oracle import dg

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-12, "fp32": 1e-5}  # relative max-norm, as for every volume parity test
LIMITS = [("fp32", 1, 260), ("fp32", 2, 85), ("fp32", 3, 50), ("fp32", 4, 50), ("fp32", 5, 26), ("fp32", 6, 40),
          ("fp32", 7, 50), ("fp32", 8, 27), ("fp64", 1, 50), ("fp64", 2, 30), ("fp64", 3, 145), ("fp64", 4, 46),
          ("fp64", 4, 115), ("fp64", 5, 145), ("fp64", 6, 25), ("fp64", 7, 25), ("fp64", 8, 25)]


@pytest.mark.parametrize("prec,N,per_sm", LIMITS)
@pytest.mark.parametrize("side", [-1, 0])
def test_forms(prec, N, per_sm, side):
    import torch

    import paper_1403_0968_gb300 as sem

    dt = torch.float64 if prec == "fp64" else torch.float32
    E, Np, offset = 152 * per_sm + side, (N + 1) * (N + 2) // 2, -side
    verts = W.tri_mesh(200, E // 400 + 1, perturb=0.2, seed=N)[:E]
    Q, B = W.swe_fields(E, Np, seed=N + 7)

    def put(a):  # the array `offset` values into its allocation
        buf = torch.empty(a.size + offset, dtype=dt, device="cuda")
        v = buf[offset:].view(a.shape)
        v.copy_(torch.from_numpy(a))
        return v

    out = put(np.full_like(Q, np.nan))
    sem.dg_volume(N, put(Q), put(B), sem.dg_geometry(verts, dt), 9.81, sem.dg_load_operators(N, dt), out=out)
    ref = dg.volume(N, Q, B, dg.geometry(verts)[:4], 9.81)
    assert np.max(np.abs(out.double().cpu().numpy() - ref)) < TOL[prec] * np.max(np.abs(ref))
