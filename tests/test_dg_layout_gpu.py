"""The DG volume kernel's layouts: element counts around a warp's batch and around the count from
which one or two lanes share an element instead of four, and arrays that start off a 16-byte
boundary (one value at a time instead of 16 bytes)."""
import numpy as np
import pytest

import workloads as W
from oracle import dg

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-12, "fp32": 1e-5}  # relative max-norm, as for every volume parity test


def _volume(N, E, prec, offset):
    import torch

    import paper_1403_0968_gb300 as sem

    dt = torch.float64 if prec == "fp64" else torch.float32
    verts = W.tri_mesh(2, (E + 3) // 4 + 1, perturb=0.2, seed=N)[:E]
    Np = (N + 1) * (N + 2) // 2
    Q, B = W.swe_fields(E, Np, seed=N + 7)

    def put(a):  # the array `offset` values into its allocation
        buf = torch.empty(a.size + offset, dtype=dt, device="cuda")
        v = buf[offset:].view(a.shape)
        v.copy_(torch.from_numpy(a))
        return v

    out = put(np.zeros_like(Q))
    sem.dg_volume(N, put(Q), put(B), sem.dg_geometry(verts, dt), 9.81, sem.dg_load_operators(N, dt), out=out)
    rx, ry, sx, sy, _ = dg.geometry(verts)
    ref = dg.volume(N, Q, B, (rx, ry, sx, sy), 9.81)
    return np.max(np.abs(out.double().cpu().numpy() - ref)) / np.max(np.abs(ref))


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("N,E,offset", [(2, 1, 0), (4, 7, 0), (7, 8, 1), (8, 9, 0), (3, 33, 1),
                                        (1, 19455, 0), (1, 19457, 1), (4, 19460, 0), (5, 19489, 1), (6, 9729, 0),
                                        (8, 9727, 1), (8, 9735, 0)])
def test_layouts(N, E, offset, prec):
    assert _volume(N, E, prec, offset) < TOL[prec]
